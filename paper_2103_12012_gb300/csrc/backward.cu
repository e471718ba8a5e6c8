// K6 backward: dL/dw for L = sum_s sum_v g[s][v] * dist_s(v).
//
// dist_s(v) is the sum of the weights on the tree path from s to v, so
// dL/dw(e) = sum over sources of the upstream gradient summed over the
// subtree hanging below tree edge e.  The subtree sums are formed children
// before parents without any sort or level loop: every vertex counts its
// children; each leaf walks up its tree, adding its accumulated sum to its tree
// edge and to its parent, then decrements the parent's child count; only the
// lane that brings the count to zero continues upward (the parent's sum is then
// complete), all others stop.  Each tree edge is visited exactly once, so the
// work is O(S*V) plus the binary searches that locate edge (pred(v), v) in
// pred(v)'s sorted row; those run for every vertex at once before the walks, so
// a walk's step is a chain of loads and atomics only.  One acquire-release
// decrement orders a child's contributions before the parent's count falls and,
// for the lane that brings it to zero, every sibling's contributions before it
// reads the parent's sum.  Accumulation is float64.
//
// The state has a vertex's sources side by side (item v * S + s).  The trees of
// different sources share most of their edges (far from the sources the
// shortest paths are the same), so neighbouring lanes have one parent: their
// counts and sums are neighbouring words, which an atomic takes a sector at a
// time, their searches read the same row, and their additions to the edge's
// gradient become one.  R-MAT scale 18, 32 sources, against an array per source: counts
// 45 -> 26, searches 117 -> 67, walks 255 -> 107 us (153 with the shared edges summed one after another);
// the transposition costs 8 us more than the copy it replaces.  Bound by the
// atomics' latency and throughput (four leaves of a thread together: 396 us).
#include <algorithm>

#include "common.cuh"
#include "internal.h"

namespace sssp {
namespace {

struct BwWs {
    uint32_t* nchild;  // [S*V]
    double* acc;       // [S*V]
    double* grad;      // [E]
    uint8_t* leaf;     // [S*V] snapshot of "has no children" taken before any walk starts
    uint32_t* eidx;    // [S*V] index of the tree edge (pred(v), v), NONE for a source or unreached vertex
    uint32_t* pred;    // [S*V] the caller's, transposed
    size_t total;
};

BwWs carve_bw(void* ws, uint32_t V, uint32_t E, uint32_t S) {
    BwWs b{};
    char* p = static_cast<char*>(ws);
    size_t off = WS_HEADER_BYTES;
    const size_t n = (size_t)S * V;
    b.nchild = reinterpret_cast<uint32_t*>(p ? p + off : nullptr);
    off += align_up(4 * std::max<size_t>(n, 1), 256);
    b.acc = reinterpret_cast<double*>(p ? p + off : nullptr);
    off += align_up(8 * std::max<size_t>(n, 1), 256);
    b.grad = reinterpret_cast<double*>(p ? p + off : nullptr);
    off += align_up(8 * std::max<size_t>(E, 1), 256);
    b.leaf = reinterpret_cast<uint8_t*>(p ? p + off : nullptr);
    off += align_up(std::max<size_t>(n, 1), 256);
    b.eidx = reinterpret_cast<uint32_t*>(p ? p + off : nullptr);
    off += align_up(4 * std::max<size_t>(n, 1), 256);
    b.pred = reinterpret_cast<uint32_t*>(p ? p + off : nullptr);
    off += align_up(4 * std::max<size_t>(n, 1), 256);
    b.total = off;
    return b;
}

__device__ __forceinline__ int64_t find_edge(const uint32_t* row_ptr, const uint32_t* col, uint32_t a, uint32_t b) {
    uint32_t lo = __ldg(&row_ptr[a]), hi = __ldg(&row_ptr[a + 1]);
    const uint32_t end = hi;
    while (lo < hi) {
        const uint32_t m = lo + ((hi - lo) >> 1);
        if (__ldg(&col[m]) < b)
            lo = m + 1;
        else
            hi = m;
    }
    return (lo < end && __ldg(&col[lo]) == b) ? (int64_t)lo : -1;
}

// Item v * S + s of the state from element s * V + v of the caller's arrays, 32 by 32 through shared memory.
__global__ void __launch_bounds__(256) k_bw_init(uint32_t V, uint32_t S, uint32_t E, const float* __restrict__ g,
                                                 const uint32_t* __restrict__ pred, uint32_t* nchild, double* acc,
                                                 uint32_t* pred_t, double* grad) {
    __shared__ float gs[32][33];
    __shared__ uint32_t ps[32][33];
    const uint32_t lane = threadIdx.x & 31u, wid = threadIdx.x >> 5, tiles = (V + 31u) / 32u;
    for (uint32_t t = blockIdx.x; t < tiles; t += gridDim.x) {
        const uint32_t v0 = t * 32u;
        for (uint32_t s0 = 0; s0 < S; s0 += 32u) {
            const uint32_t ns = min(32u, S - s0), nv = min(32u, V - v0);
            if (lane < nv)
                for (uint32_t s = wid; s < ns; s += 8u) {
                    const size_t at = (size_t)(s0 + s) * V + v0 + lane;
                    gs[s][lane] = __ldg(&g[at]);
                    ps[s][lane] = __ldg(&pred[at]);
                }
            __syncthreads();
            for (uint32_t k = threadIdx.x; k < nv * ns; k += 256u) {
                const uint32_t v = k / ns, s = k - v * ns;
                const size_t i = (size_t)(v0 + v) * S + s0 + s;
                nchild[i] = 0u;
                acc[i] = (double)gs[s][v];
                pred_t[i] = ps[s][v];
            }
            __syncthreads();
        }
    }
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < E; i += (size_t)gridDim.x * blockDim.x) grad[i] = 0.0;
}

// an item's vertex
__device__ __forceinline__ uint32_t vertex_of(size_t i, size_t n, uint32_t S) {
    return n >> 32 ? (uint32_t)(i / S) : (uint32_t)i / S;
}

__global__ void k_bw_count(uint32_t V, uint32_t S, size_t n, const uint32_t* __restrict__ pred, uint32_t* nchild, WsHeader* hdr) {
    const size_t stride = (size_t)gridDim.x * blockDim.x;
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
        const uint32_t p = pred[i];
        if (p == NONE) continue;
        if (p >= V) {
            set_status(hdr, SSSP_EINVAL);
            continue;
        }
        atomicAdd(&nchild[(size_t)p * S + (i - (size_t)vertex_of(i, n, S) * S)], 1u);
    }
}

// leaves, and the tree edge of every vertex (the searches of all walks, in parallel)
__global__ void k_bw_leaves(uint32_t V, uint32_t S, size_t n, const uint32_t* __restrict__ row_ptr,
                            const uint32_t* __restrict__ col, const uint32_t* __restrict__ pred,
                            const uint32_t* __restrict__ nchild, uint8_t* leaf, uint32_t* eidx) {
    const size_t stride = (size_t)gridDim.x * blockDim.x;
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
        const uint32_t p = pred[i];
        leaf[i] = (p != NONE && nchild[i] == 0u) ? 1u : 0u;
        const int64_t e = (p != NONE && p < V) ? find_edge(row_ptr, col, p, vertex_of(i, n, S)) : -1;
        eidx[i] = e < 0 ? NONE : (uint32_t)e;
    }
}

// atomic decrement with acquire-release semantics at GPU scope
__device__ __forceinline__ uint32_t dec_acq_rel(uint32_t* p) {
    uint32_t old;
    asm volatile("atom.acq_rel.gpu.global.add.u32 %0, [%1], %2;" : "=r"(old) : "l"(p), "r"(0xFFFFFFFFu) : "memory");
    return old;
}

// A warp walks its 32 items up together; the lanes on one tree edge add to its gradient once.
__global__ void __launch_bounds__(256) k_bw_walk(uint32_t V, uint32_t S, size_t n, const uint32_t* __restrict__ pred,
                                                 const uint32_t* __restrict__ eidx, const uint8_t* __restrict__ leaf,
                                                 uint32_t* nchild, double* acc, double* grad, WsHeader* hdr) {
    const uint32_t lane = threadIdx.x & 31u;
    const size_t stride = (size_t)gridDim.x * blockDim.x;
    for (size_t i0 = (size_t)blockIdx.x * blockDim.x + (threadIdx.x & ~31u); i0 < n; i0 += stride) {
        size_t at = i0 + lane;  // the item
        const uint32_t s = (uint32_t)(at - (size_t)vertex_of(at, n, S) * S);
        bool on = at < n && leaf[at];  // walks start at leaves only
        // bounded by V steps: a tree path has fewer than V edges
        for (uint32_t step = 0; step < V && __any_sync(0xFFFFFFFFu, on); ++step) {
            uint32_t p = NONE, e = NONE;
            double a = 0.0;
            if (on) {
                p = __ldg(&pred[at]);
                e = __ldg(&eidx[at]);
                a = ld_relaxed(&acc[at]);
                if (p >= V) {  // reached the source
                    on = false;
                } else if (e == NONE) {  // (pred(x), x) is not an edge
                    set_status(hdr, SSSP_EINVAL);
                    on = false;
                }
            }
            // one addition to the edge's gradient for the lanes that share it: pairs, pairs of pairs, ... of
            // all edges at once (a lane of odd rank hands its sum to the one before and drops out)
            const uint32_t same = __match_any_sync(0xFFFFFFFFu, on ? e : NONE);
            uint32_t rank = __popc(same & ((1u << lane) - 1u)), rest = on ? same & (0xFFFFFFFEu << lane) : 0u;
            const bool first = rank == 0u;
            double sum = a;
            for (; __any_sync(0xFFFFFFFFu, rest != 0u); rank >>= 1) {
                const uint32_t next = rest ? __ffs(rest) - 1u : lane;
                const double t = __shfl_sync(0xFFFFFFFFu, sum, next);
                if (rest) sum += t;
                rest &= __ballot_sync(0xFFFFFFFFu, !(rank & 1u));
            }
            if (on) {
                if (first) atomicAdd(&grad[e], sum);
                at = (size_t)p * S + s;
                atomicAdd(&acc[at], a);
                // release: my contributions before my decrement; acquire (last child): every
                // sibling's contributions before the read of acc[p] in the next step
                on = dec_acq_rel(&nchild[at]) == 1u;
            }
        }
    }
}

__global__ void k_bw_out(uint32_t E, const double* __restrict__ grad, float* out) {
    for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < E; i += gridDim.x * blockDim.x)
        out[i] = (float)grad[i];
}

unsigned grid_for(size_t n) {
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    return (unsigned)std::max<size_t>(1, std::min<size_t>((n + 255) / 256, (size_t)sms * 16));
}

}  // namespace

size_t backward_workspace_bytes(uint32_t V, uint32_t E, uint32_t S) { return carve_bw(nullptr, V, E, S).total; }

cudaError_t backward_launch(const sssp_graph* g, uint32_t S, const uint32_t* pred, const float* grad_dist,
                            float* grad_w, void* ws, cudaStream_t st) {
    BwWs b = carve_bw(ws, g->V, g->E, S);
    WsHeader* hdr = static_cast<WsHeader*>(ws);
    const size_t n = (size_t)S * g->V;
    cudaError_t e;
    if ((e = cudaMemsetAsync(hdr, 0, WS_HEADER_BYTES, st)) != cudaSuccess) return e;
    k_bw_init<<<grid_for(std::max<size_t>(n, g->E)), 256, 0, st>>>(g->V, S, g->E, grad_dist, pred, b.nchild, b.acc, b.pred, b.grad);
    k_bw_count<<<grid_for(n), 256, 0, st>>>(g->V, S, n, b.pred, b.nchild, hdr);
    k_bw_leaves<<<grid_for(n), 256, 0, st>>>(g->V, S, n, g->row_ptr, g->col, b.pred, b.nchild, b.leaf, b.eidx);
    k_bw_walk<<<grid_for(n), 256, 0, st>>>(g->V, S, n, b.pred, b.eidx, b.leaf, b.nchild, b.acc, b.grad, hdr);
    k_bw_out<<<grid_for(g->E), 256, 0, st>>>(g->E, b.grad, grad_w);
    return cudaGetLastError();
}

}  // namespace sssp
