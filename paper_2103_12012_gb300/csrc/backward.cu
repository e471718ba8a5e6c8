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
// The state has a vertex's sources side by side, and warps take items v * S + s.  The trees of
// different sources share most of their edges (far from the sources the
// shortest paths are the same), so neighbouring lanes have one parent: their
// counts and sums are neighbouring words, which an atomic takes a sector at a
// time, their searches read the same row, and their additions to the edge's
// gradient become one.  R-MAT scale 18, 32 sources, against an array per source: counts
// 45 -> 26, searches 117 -> 67, walks 255 -> 107 us (153 with the shared edges summed one after another);
// the transposition costs 8 us more than the copy it replaces.  Bound by the
// atomics' latency and throughput (four leaves of a thread together: 396 us).
// Sixteen sources are side by side, so that the sums of a vertex with very many children, which all come to
// a few cache lines, are in several of them (star of 1 M leaves, 32 sources: 11.2 ms with all side by side, 6.0 with
// sixteen, 3.7 with eight; random graph of 1 M vertices, 32 sources: 3.1, 3.5 and 3.9).
#include <algorithm>

#include "common.cuh"
#include "internal.h"

namespace sssp {
namespace {

constexpr uint32_t REFILL = 24;  // lanes of a warp (k_bw_walk)
constexpr uint32_t FEW = 8;      // sources that are transposed without shared memory (1 M vertices, 2: 216 -> 196 us)

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

// an item's vertex
__device__ __forceinline__ uint32_t vertex_of(size_t i, size_t n, uint32_t S) {
    return n >> 32 ? (uint32_t)(i / S) : (uint32_t)i / S;
}

// Where the state has (v, s): the sources of a block of sixteen side by side.
struct Place {
    size_t base;
    uint32_t wide;
    __device__ __forceinline__ Place(uint32_t V, uint32_t S, uint32_t s)
        : base((size_t)(s & ~15u) * V + (s & 15u)), wide(min(16u, S - (s & ~15u))) {}
    __device__ __forceinline__ size_t operator()(uint32_t v) const { return base + (size_t)v * wide; }
};

__device__ __forceinline__ void clear_grad(uint32_t E, double* grad) {
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < E; i += (size_t)gridDim.x * blockDim.x) grad[i] = 0.0;
}

// Item v * S + s of the state from element s * V + v of the caller's arrays: a thread per item (a few sources; pred_t
// NULL: one), or 32 by 32 through shared memory.
__global__ void __launch_bounds__(256) k_bw_init_few(uint32_t V, uint32_t S, uint32_t E, const float* __restrict__ g,
                                                     const uint32_t* __restrict__ pred, uint32_t* nchild, double* acc,
                                                     uint32_t* pred_t, double* grad) {
    const size_t n = (size_t)S * V;
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
        const uint32_t v = vertex_of(i, n, S);
        const size_t at = (i - (size_t)v * S) * V + v;
        nchild[i] = 0u;
        acc[i] = (double)__ldg(&g[at]);
        if (pred_t) pred_t[i] = __ldg(&pred[at]);
    }
    clear_grad(E, grad);
}

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
                const size_t i = Place(V, S, s0 + s)(v0 + v);
                nchild[i] = 0u;
                acc[i] = (double)gs[s][v];
                pred_t[i] = ps[s][v];
            }
            __syncthreads();
        }
    }
    clear_grad(E, grad);
}

__global__ void k_bw_count(uint32_t V, uint32_t S, size_t n, const uint32_t* __restrict__ pred, uint32_t* nchild, WsHeader* hdr) {
    const size_t stride = (size_t)gridDim.x * blockDim.x;
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
        const uint32_t v = vertex_of(i, n, S);
        const Place at(V, S, (uint32_t)(i - (size_t)v * S));
        const uint32_t p = pred[at(v)];
        if (p == NONE) continue;
        if (p >= V) {
            set_status(hdr, SSSP_EINVAL);
            continue;
        }
        atomicAdd(&nchild[at(p)], 1u);
    }
}

// leaves, and the tree edge of every vertex (the searches of all walks, in parallel)
__global__ void k_bw_leaves(uint32_t V, uint32_t S, size_t n, const uint32_t* __restrict__ row_ptr,
                            const uint32_t* __restrict__ col, const uint32_t* __restrict__ pred,
                            const uint32_t* __restrict__ nchild, uint8_t* leaf, uint32_t* eidx) {
    const size_t stride = (size_t)gridDim.x * blockDim.x;
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
        const uint32_t v = vertex_of(i, n, S);
        const size_t at = Place(V, S, (uint32_t)(i - (size_t)v * S))(v);
        const uint32_t p = pred[at];
        leaf[at] = (p != NONE && nchild[at] == 0u) ? 1u : 0u;
        const int64_t e = (p != NONE && p < V) ? find_edge(row_ptr, col, p, v) : -1;
        eidx[at] = e < 0 ? NONE : (uint32_t)e;
    }
}

// atomic decrement with acquire-release semantics at GPU scope
__device__ __forceinline__ uint32_t dec_acq_rel(uint32_t* p) {
    uint32_t old;
    asm volatile("atom.acq_rel.gpu.global.add.u32 %0, [%1], %2;" : "=r"(old) : "l"(p), "r"(0xFFFFFFFFu) : "memory");
    return old;
}

// A warp walks the leaves among its items up.  A lane whose walk has ended takes another item while others go on (once
// REFILL lanes or fewer do): walks are as long as the tree is deep, and a warp that waited for its longest one left
// the other lanes idle.  Grid of 1000 x 1000, 8 sources: 17.2 -> 3.5 ms (7.2 with an array per source and a thread
// per leaf); random graph of 1 M vertices, 32 sources: 2.5 -> 2.9 (3.7), since fewer lanes share an edge; with 4 lanes
// for REFILL 4.0 and 2.8, with 31 3.6 and 2.9.
// SHARED: the lanes on one tree edge add to its gradient once.
template <bool SHARED>
__global__ void __launch_bounds__(256) k_bw_walk(uint32_t V, uint32_t S, size_t n, size_t per, const uint32_t* __restrict__ pred,
                                                 const uint32_t* __restrict__ eidx, const uint8_t* __restrict__ leaf,
                                                 uint32_t* nchild, double* acc, double* grad, WsHeader* hdr) {
    const uint32_t lane = threadIdx.x & 31u;
    size_t next = (((size_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5) * per;  // first item not taken yet
    const size_t end = min(next + per, n);
    size_t at = 0;  // where the lane is
    Place place(V, S, 0);
    uint32_t steps = 0;
    bool on = false;
    for (;;) {
        const uint32_t live = __ballot_sync(0xFFFFFFFFu, on);
        bool fresh = false;  // (walks start at leaves only)
        if (next < end && __popc(live) <= (int)REFILL) {
            if (!on) {
                const size_t i = next + __popc(~live & ((1u << lane) - 1u));
                fresh = i < end;
                steps = 0;
                if (fresh) {
                    const uint32_t v = vertex_of(i, n, S);
                    place = Place(V, S, (uint32_t)(i - (size_t)v * S));
                    at = place(v);
                }
            }
            next += 32u - __popc(live);
        } else if (!live) {
            break;
        }
        uint32_t p = NONE, e = NONE;
        double a = 0.0;
        if (on || fresh) {
            p = __ldg(&pred[at]);
            e = __ldg(&eidx[at]);
            a = ld_relaxed(&acc[at]);
            if (fresh) on = leaf[at];
            if (on && p >= V) {  // reached the source
                on = false;
            } else if (on && e == NONE) {  // (pred(x), x) is not an edge
                set_status(hdr, SSSP_EINVAL);
                on = false;
            }
        }
        const bool act = on;
        uint32_t left = 0;
        if (act) {
            at = place(p);
            atomicAdd(&acc[at], a);
            // release: my contributions before my decrement; acquire (last child): every
            // sibling's contributions before the read of acc[p] in the next step
            left = dec_acq_rel(&nchild[at]);
        }
        // (the edges' gradients, while the decrement is on its way)
        bool first = act;
        double sum = a;
        if constexpr (SHARED) {
            // one addition to the edge's gradient for the lanes that share it: pairs, pairs of pairs, ... of
            // all edges at once (a lane of odd rank hands its sum to the one before and drops out)
            const uint32_t same = __match_any_sync(0xFFFFFFFFu, act ? e : NONE);
            uint32_t rank = __popc(same & ((1u << lane) - 1u)), rest = act ? same & (0xFFFFFFFEu << lane) : 0u;
            first = act && rank == 0u;
            for (; __any_sync(0xFFFFFFFFu, rest != 0u); rank >>= 1) {
                const uint32_t other = rest ? __ffs(rest) - 1u : lane;
                const double t = __shfl_sync(0xFFFFFFFFu, sum, other);
                if (rest) sum += t;
                rest &= __ballot_sync(0xFFFFFFFFu, !(rank & 1u));
            }
        }
        if (first) atomicAdd(&grad[e], sum);
        on = act && left == 1u && ++steps < V;  // (a tree path has fewer than V edges)
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
    const unsigned init = grid_for(std::max<size_t>(n, g->E));
    if (S == 1) b.pred = nullptr;  // (the caller's is in this order)
    if (S <= FEW)
        k_bw_init_few<<<init, 256, 0, st>>>(g->V, S, g->E, grad_dist, pred, b.nchild, b.acc, b.pred, b.grad);
    else
        k_bw_init<<<init, 256, 0, st>>>(g->V, S, g->E, grad_dist, pred, b.nchild, b.acc, b.pred, b.grad);
    if (S > 1) pred = b.pred;
    k_bw_count<<<grid_for(n), 256, 0, st>>>(g->V, S, n, pred, b.nchild, hdr);
    k_bw_leaves<<<grid_for(n), 256, 0, st>>>(g->V, S, n, g->row_ptr, g->col, pred, b.nchild, b.leaf, b.eidx);
    const unsigned walks = grid_for(n);
    const size_t per = ((n + walks * 8ull - 1) / (walks * 8ull) + 31) & ~(size_t)31;
    (S > 1 ? k_bw_walk<true> : k_bw_walk<false>)<<<walks, 256, 0, st>>>(g->V, S, n, per, pred, b.eidx, b.leaf, b.nchild, b.acc,
                                                                        b.grad, hdr);
    k_bw_out<<<grid_for(g->E), 256, 0, st>>>(g->E, b.grad, grad_w);
    return cudaGetLastError();
}

}  // namespace sssp
