// K3 Trishla triangle prune (Sec. III.B, Algorithm 1).
//
// Every edge (u, v_i) whose v_i may be a witness (local mode, the paper's "(v_i, v_j) in E_i": v_i in
// u's partition) is a pair: N(u) and N(v_i) are intersected, the shorter walked and the longer
// searched, and keep[(u, v_j)] is cleared where w(u, v_j) > w(u, v_i) + w(v_i, v_j), the least
// witness recorded.  A block finds the pairs of its edges, collects them, and splits the elements to
// walk evenly over its warps, whatever the lists' lengths.  The launch that finishes a job begun by the
// idle blocks of a solve (sssp_solve_prune) tests the heavy pairs of the chunks they took and every
// pair of the rest.
//
// Bound by the instructions and the latency of the searches (about ten dependent loads an element, most
// from L1): 32 registers, so that an SM holds 64 warps.  Against a warp per chunk of 32 edges, one pair
// after another (whose tail, a few chunks of hub rows, left two thirds of the warps idle, and which
// searched the row pointers for every chunk): R-MAT of 2.1 M vertices and 32 M edges, 148 partitions,
// local mode, 4.21 -> 0.96 ms; 60,013 vertices and 800,001 edges, any witness, float32, 0.85 -> 0.65 ms.
// Two searches of a lane in flight: 1.59 and 0.87 ms (40 registers or spills); units of 128 to 512
// elements handed out one by one instead of even shares: 1.70 and 0.95.
#include <algorithm>

#include "common.cuh"
#include "internal.h"
#include "rowwalk.cuh"
#include "trishla.cuh"

namespace sssp {
namespace {

constexpr uint32_t TRISHLA_CHUNK = 32;  // edges of a chunk that an idle block of a solve takes

// A pair: x: first element walked, less the elements of the pairs before it; y, z: first element and
// length of the list searched; w: its edge (N(u) is searched if it holds the edge).
//
// Elements [t0, t1) of the walks of the n pairs in P (start: elements before each).
template <class W>
__device__ __forceinline__ void test_pairs(const TrishlaJob& J, const uint4* P, const uint32_t* start, uint32_t n,
                                           uint32_t t0, uint32_t t1) {
    const uint32_t lane = threadIdx.x & 31u;
    if (t0 >= t1) return;
    uint32_t lo = 0, len = n;  // the last pair that starts at t0 or before (every pair has elements)
    while (len > 1u) {
        const uint32_t h = len >> 1;
        if (start[lo + h] <= t0) lo += h;
        len -= h;
    }
    uint32_t first = lo, seen = 0;  // pairs [first, first + 32) are at hand, one a lane
    uint32_t p = first + lane < n ? start[first + lane] : 0xFFFFFFFFu;
    seen = __popc(__ballot_sync(0xFFFFFFFFu, p < t0));
    uint32_t end = first + 32u < n ? start[first + 32u] : 0xFFFFFFFFu;
    for (uint32_t t = t0; t < t1; t += 32u) {
        uint32_t c = 0;
        for (;;) {  // (a lane at or past the window's end finds its pair in a later window)
            const uint32_t at = __reduce_or_sync(0xFFFFFFFFu, p - t < 32u ? 1u << (p - t) : 0u);
            const uint32_t q = seen + __popc(at & (0xFFFFFFFFu >> (31u - lane)));
            if (q) c = first + q - 1u;
            seen += __popc(at);
            if (end >= min(t + 32u, t1)) break;
            first += 32u;
            p = first + lane < n ? start[first + lane] : 0xFFFFFFFFu;
            end = first + 32u < n ? start[first + 32u] : 0xFFFFFFFFu;
            seen = 0;
        }
        if (t + lane >= t1) continue;
        const uint4 q = P[c];
        const uint32_t j = q.x + t + lane, x = __ldg(&J.col[j]);
        uint32_t k = q.y, m = q.z;
        while (m > 1u) {  // to the first element that is not below x, if there is one
            const uint32_t h = m >> 1;
            if (__ldg(&J.col[k + h - 1u]) < x) k += h;
            m -= h;
        }
        if (__ldg(&J.col[k]) == x) {
            const bool in_u = q.w - q.y < q.z;
            const uint32_t eu = in_u ? k : j, ev = in_u ? j : k;
            if (tri_dominated<W>(__ldg(&J.w[eu]), __ldg(&J.w[q.w]), __ldg(&J.w[ev]))) {
                J.keep[eu] = 0;
                if (J.witness) atomicMin(&J.witness[eu], __ldg(&J.col[q.w]));
            }
        }
    }
}

// A warp finds the pairs among `per` consecutive edges (a multiple of 32).  With a cursor (the end of
// a job the idle blocks of a solve began: they handed out chunks [0, *cursor) and tested their light
// pairs) the chunks below the cursor get their heavy pairs only, the others every pair.
template <class W, uint32_t TT>
__global__ void __launch_bounds__(TT, 2048 / TT) k_trishla(TrishlaJob J, const unsigned long long* cursor, uint32_t per) {
    constexpr uint32_t TW = TT / 32, PAIRS = TT * 3 / 2;
    __shared__ __align__(16) uint4 pairs[PAIRS];
    __shared__ unsigned long long sums[TW];
    __shared__ uint32_t start[PAIRS], count, rows[TW][32], starts[TW][32];
    const uint32_t tid = threadIdx.x, lane = tid & 31u, wid = tid >> 5;
    const unsigned long long light_done =
        cursor ? min(*cursor, (unsigned long long)J.nchunks) * J.chunk : 0ull;  // edges below: heavy pairs only
    const unsigned long long from = (unsigned long long)(blockIdx.x * TW + wid) * per;
    const uint32_t e0 = (uint32_t)min(from, (unsigned long long)J.E), e1 = (uint32_t)min(from + per, (unsigned long long)J.E);
    RowWalk walk{J.row_ptr, J.V, rows[wid], starts[wid]};
    if (e0 < e1) walk.seek(e0);
    if (tid == 0) count = 0u;
    uint32_t n = 0;     // pairs collected
    uint32_t part = 0;  // first vertex of a partition
    const uint32_t B = (uint32_t)J.B;
    __syncthreads();
    for (uint32_t done = 0; done < per; done += 32u) {
        const uint32_t eb = e0 + done, e = eb + lane;
        bool cand = false;
        uint32_t u = 0, v = NONE;
        if (eb < e1) {
            if (e < e1) v = __ldg(&J.col[e]);
            u = walk.step(eb, e1);
            cand = v < J.V;
            if (J.mode == 0) {
                if (__any_sync(0xFFFFFFFFu, e < e1 && u - part >= B)) part = u - u % B;
                cand = cand && v - part < B;
            }
        }
        uint32_t a0 = 0, da = 0, b0 = 0, db = 0;
        if (cand) {
            a0 = __ldg(&J.row_ptr[u]), da = __ldg(&J.row_ptr[u + 1]) - a0;
            b0 = __ldg(&J.row_ptr[v]), db = __ldg(&J.row_ptr[v + 1]) - b0;
            cand = db != 0u && (e >= light_done || max(da, db) > TRISHLA_LIGHT);
        }
        const uint32_t got = __ballot_sync(0xFFFFFFFFu, cand);
        if (got) {
            uint32_t at = 0;
            if (lane == 0) at = atomicAdd(&count, (uint32_t)__popc(got));
            at = __shfl_sync(0xFFFFFFFFu, at, 0) + __popc(got & ((1u << lane) - 1u));
            if (cand) {
                const bool walks_v = db < da;
                pairs[at] = walks_v ? make_uint4(b0, a0, da, e) : make_uint4(a0, b0, db, e);
                start[at] = walks_v ? db : da;
            }
        }
        n += (uint32_t)__syncthreads_count(cand);
        if (n == 0u || (n <= PAIRS - TT && done + 32u < per)) continue;  // room for another round
        // lengths to starts, two a thread
        const uint32_t x0 = 2u * tid < n ? start[2u * tid] : 0u, x1 = 2u * tid + 1u < n ? start[2u * tid + 1u] : 0u;
        unsigned long long inc = (unsigned long long)x0 + x1;
#pragma unroll
        for (uint32_t o = 1; o < 32u; o <<= 1) {
            const unsigned long long y = __shfl_up_sync(0xFFFFFFFFu, inc, o);
            if (lane >= o) inc += y;
        }
        if (lane == 31u) sums[wid] = inc;
        __syncthreads();
        unsigned long long base = inc - x0 - x1, total = 0;
#pragma unroll
        for (uint32_t i = 0; i < TW; ++i) {
            if (i < wid) base += sums[i];
            total += sums[i];
        }
        if (total < 0xFFFF0000ull) {
            const uint32_t b = (uint32_t)base, t = (uint32_t)total;
            if (2u * tid < n) start[2u * tid] = b, pairs[2u * tid].x -= b;
            if (2u * tid + 1u < n) start[2u * tid + 1u] = b + x0, pairs[2u * tid + 1u].x -= b + x0;
            __syncthreads();
            const uint32_t share = (t / TW + 32u) & ~31u;
            test_pairs<W>(J, pairs, start, n, min(wid * share, t), min((wid + 1u) * share, t));
        } else {  // (some pairs of a graph of billions of edges: one at a time)
            for (uint32_t i = 0; i < n; ++i) {
                const uint32_t t = start[i], share = (t / TW + 32u) & ~31u;
                __syncthreads();
                if (tid == 0) start[i] = 0u;
                __syncthreads();
                test_pairs<W>(J, pairs + i, start + i, 1u, min(wid * share, t), min((wid + 1u) * share, t));
            }
        }
        n = 0;
        if (tid == 0) count = 0u;
        __syncthreads();
    }
}

}  // namespace

TrishlaJob trishla_job(const sssp_graph* g, int mode, uint8_t* keep, uint32_t* witness) {
    TrishlaJob J{};
    J.V = g->V;
    J.E = g->E;
    J.B = ((unsigned long long)g->V + g->partitions - 1) / g->partitions;
    J.mode = mode;
    J.row_ptr = g->row_ptr;
    J.col = g->col;
    J.w = static_cast<const uint32_t*>(g->w);
    J.keep = keep;
    J.witness = witness;
    J.chunk = TRISHLA_CHUNK;
    J.nchunks = (uint32_t)(((uint64_t)g->E + TRISHLA_CHUNK - 1) / TRISHLA_CHUNK);
    return J;
}

cudaError_t trishla_init(const TrishlaJob& J, cudaStream_t st) {
    cudaError_t e;
    if ((e = cudaMemsetAsync(J.keep, 1, J.E, st)) != cudaSuccess) return e;
    if (J.witness && (e = cudaMemsetAsync(J.witness, 0xFF, sizeof(uint32_t) * (size_t)J.E, st)) != cudaSuccess)
        return e;
    return cudaSuccess;
}

cudaError_t trishla_launch(const TrishlaJob& J, int wtype, const unsigned long long* cursor, cudaStream_t st) {
    if (J.nchunks == 0) return cudaSuccess;
    // Local mode with many partitions: few edges are pairs, and a few blocks hold most of the elements
    // (hubs of one partition), so blocks are as large as they get and take several rounds of edges
    // (32 M edges, 148 partitions: 0.96 ms; 2.05 with blocks of 256 threads and one round).  Otherwise
    // every block has plenty, and small ones end more evenly: 4.2 M edges, one partition, 3.43 against
    // 4.01 ms; at 8 partitions both take 0.67.
    const bool few = J.mode == 0 && J.B <= J.V / 8;
    uint64_t per = 32;
    if (few) {
        int dev = 0, sms = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        per *= std::min<uint64_t>(std::max<uint64_t>(J.E / ((uint64_t)std::max(sms, 1) * 8192u), 1u), 8u);
    }
    const uint32_t TT = few ? 1024u : 256u;
    const unsigned grid = (unsigned)((J.E + per * (TT / 32u) - 1) / (per * (TT / 32u)));
    const bool f32 = wtype == SSSP_W_F32;
    auto* const k = few ? (f32 ? k_trishla<WF32, 1024> : k_trishla<WU32, 1024>) : (f32 ? k_trishla<WF32, 256> : k_trishla<WU32, 256>);
    k<<<grid, TT, 0, st>>>(J, cursor, (uint32_t)per);
    return cudaGetLastError();
}

cudaError_t prune_launch(const sssp_graph* g, int mode, uint8_t* keep, uint32_t* witness, cudaStream_t st) {
    const TrishlaJob J = trishla_job(g, mode, keep, witness);
    cudaError_t e;
    if ((e = trishla_init(J, st)) != cudaSuccess) return e;
    return trishla_launch(J, g->wtype, nullptr, st);
}

}  // namespace sssp
