// K5b: the problems of a batch in shared memory: all of them if every graph fits, or the ones that do of a
// large batch (api.cu).  A block takes a unit (one problem, or up to 16 of a
// graph, as copies of it with a source each) from a queue and keeps its distances there, 4 bytes an
// item: reading a head's distance, lowering it and marking it cost tens of cycles instead of the L2 round
// trips of the general kernel (k_batched, relax.cu), which stays for larger graphs.
//
// Buckets of distances in turn: items below the bound are marked near, the others far.  A round takes
// the near marks, 512 items at a time, and its warps relax their rows; a warp holds 32 rows and
// walks their edges together, rows of HUB edges and more are cut into segments that all warps share (api.cu's
// in_smem says which graphs are not for it: very dense ones, and wide grids at a given width).
// When no near mark is left, the bound moves to the end of the bucket of the least far distance, and the
// round takes the far marks below it.  A mark is cleared before its distance is read, and set after
// the distance is lowered, so no fall is lost.  Predecessors come from one walk over the edges at the end:
// pred(v) is the least tail u with dist(u) + w = dist(v), to which the packed words of the general kernel
// converge too.
//
// Bound by instructions (half of the issue slots at 32 warps an SM) and by the rounds' barriers.  Against the
// general kernel, ms (vertices, graphs x sources; uint32 / float32): 1,024-2,048, 512 x 16: 6.17 -> 1.87 / 6.26 -> 1.08;
// 1,024-4,096, 32 x 16: 0.59 -> 0.24 / 0.58 -> 0.17; 1,024-16,384, 200 x 5: 1.28 -> 0.80 / 1.22 -> 0.52; 1,024-46,000,
// 512 x 16: 14.6 -> 9.0 / 13.6 -> 6.3.  Two or four steps of a warp in flight: 1 to 8% slower.  Distances of
// larger graphs in the shared memory of a cluster (2 or 4 blocks, 47,104 to 131,072 vertices) took 27 against 23
// ms, in L2 with the marks in shared memory 40: there the general kernel's 64 warps an SM hide more.
// 512 threads a block while units are small (several blocks an SM: 1,024-2,048, 512 x 2: 0.53 against 0.84 ms with
// 1,024), else 1,024 (1,024-32,768, 100 x 3: 0.60 against 0.88).
#include "common.cuh"
#include "internal.h"
#include "rowwalk.cuh"

namespace sssp {
namespace {

// rows from here on are cut into segments of this size (512: the warp with the longest rows held up the round: 100 R-MAT
// graphs of 4,000 vertices, 16 sources each, 0.80 -> 0.72 ms, 256 0.75, 64 0.65; 30 of 40,000, 16 edges each, 2.62 -> 2.79)
constexpr uint32_t HUB = 128;
constexpr uint32_t HCAP = 512;                   // hub segments of a round
constexpr uint32_t EB = 1;                       // steps of 32 edges in flight
constexpr uint64_t LIMIT_FACTOR = 3;
constexpr uint32_t BATCH_SMALL = 8192;           // units of at most this: 512 threads a block

template <uint32_t BW>
struct Mem {
    BatchUnit unit;
    uint32_t unit_at;
    uint4 row[BW][32];       // a warp's rows: first edge - edges before it, first item of the copy, distance
    uint32_t q[BW][64];      // a warp's items to relax
    uint2 hub[HCAP];         // item, segment
    uint32_t next, hnext[2], nhub[2], low[2], flags[2];  // by round parity
    unsigned long long stats[6];
    uint32_t reach[BATCH_COPIES];  // vertices that a copy's source has reached
};

// The items of a unit: copy * V + vertex.
struct Items {
    uint32_t *dist, *near, *far;
    uint32_t V;

    __device__ __forceinline__ uint32_t vertex(uint32_t i) const { return i < V ? i : i % V; }
    __device__ __forceinline__ uint32_t get(uint32_t i) const { return *reinterpret_cast<volatile uint32_t*>(dist + i); }
    __device__ __forceinline__ void mark(uint32_t i, bool is_near) const {
        atomicOr((is_near ? near : far) + (i >> 5), 1u << (i & 31u));
    }
};

template <class W, uint32_t BT>
struct Round {
    const Items& I;
    Mem<BT / 32>& M;
    const uint32_t *row_ptr, *col, *w;
    uint32_t V, lane, wid, par, thr;
    uint32_t low, bad, any_near;      // least distance marked far, an item marked near
    uint32_t n_at, n_imp, n_vert;     // (a lane's counts)
    unsigned long long n_edges;

    // Relaxes edges [0, total) of the rows held.  Row r's edges start at the p of some lane (ascending;
    // lanes without a row: none), so the rows that start within the 32 edges of a step are a bit mask,
    // and a lane's row is the count of starts up to it.
    __device__ __forceinline__ void run(uint32_t total, uint32_t p) {
        const uint4* const row = M.row[wid];
        uint32_t seen = 0;
        for (uint32_t k0 = 0; k0 < total; k0 += 32u * EB) {
            uint32_t v[EB], x[EB], a[EB], at[EB], d[EB], l = 0;
#pragma unroll
            for (uint32_t j = 0; j < EB; ++j) {
                const uint32_t k = k0 + 32u * j;
                v[j] = NONE;
                if (k >= total) continue;
                const uint32_t starts = __reduce_or_sync(0xFFFFFFFFu, p - k < 32u ? 1u << (p - k) : 0u);
                a[j] = seen + __popc(starts & (0xFFFFFFFFu >> (31u - lane))) - 1u;
                seen += __popc(starts);
                if (k + lane < total) {
                    const uint32_t e = row[a[j]].x + k + lane;
                    v[j] = __ldg(&col[e]);
                    x[j] = __ldg(&w[e]);
                }
            }
#pragma unroll
            for (uint32_t j = 0; j < EB; ++j) {
                d[j] = 0;  // (x becomes the candidate distance)
                if (v[j] == NONE) continue;
                if (!W::weight_ok(x[j]) || v[j] >= V) {
                    bad |= 1u;
                    continue;
                }
                const uint4 r = row[a[j]];
                if (!W::add(r.z, x[j], x[j])) {
                    bad |= 2u;
                    continue;
                }
                at[j] = r.y + v[j];
                d[j] = I.get(at[j]);
            }
#pragma unroll
            for (uint32_t j = 0; j < EB; ++j)
                if (d[j] > x[j]) {
                    ++n_at;
                    if (atomicMin(I.dist + at[j], x[j]) > x[j]) l |= 1u << j;
                }
            if (l) {
                __threadfence_block();  // the distance before its mark
#pragma unroll
                for (uint32_t j = 0; j < EB; ++j)
                    if (l & (1u << j)) {
                        const bool is_near = x[j] < thr;
                        ++n_imp;
                        I.mark(at[j], is_near);
                        if (is_near)
                            any_near = 1u;
                        else
                            low = min(low, x[j]);
                    }
            }
        }
        if (lane == 0) n_edges += total;
    }

    // the first n items of the warp's queue, whose marks are cleared
    __device__ __forceinline__ void relax_items(uint32_t n) {
        __syncwarp();
        __threadfence_block();  // a distance lowered after this read marks its item again
        uint32_t item = 0, v = 0, beg = 0, deg = 0, d = 0;
        if (lane < n) {
            item = M.q[wid][lane];
            v = I.vertex(item);
            beg = __ldg(&row_ptr[v]);
            deg = __ldg(&row_ptr[v + 1]) - beg;
            d = I.get(item);
            ++n_vert;
            if (deg >= HUB) {  // segments for the whole block
                const uint32_t k = (deg - 1u) / HUB + 1u, at = k <= HCAP ? atomicAdd(&M.nhub[par], k) : HCAP;
                const bool fits = k <= HCAP && at + k <= HCAP;
                for (uint32_t i = 0; i < k && at + i < HCAP; ++i) M.hub[at + i] = make_uint2(fits ? item : NONE, i);
                if (fits) deg = 0;
            }
        }
        uint32_t inc = deg;
#pragma unroll
        for (uint32_t o = 1; o < 32u; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, inc, o);
            if (lane >= o) inc += y;
        }
        const uint32_t rows = __ballot_sync(0xFFFFFFFFu, deg != 0u);
        if (deg)
            M.row[wid][__popc(rows & ((1u << lane) - 1u))] = make_uint4(beg - (inc - deg), item - v, d, 0u);
        __syncwarp();
        run(__shfl_sync(0xFFFFFFFFu, inc, 31), deg ? inc - deg : 0xFFFFFFFFu);
        __syncwarp();
    }

    // A round: the items marked near, up to 512 of them at a time (16 marks a lane; fewer of a small unit, so that
    // every warp gets some, and two lots if there are copies: 20 graphs of 1,500 vertices and 300,000 edges, 1 source
    // each, 3.1 -> 1.0 ms; 100 R-MAT graphs of 4,000 vertices, 16 sources each, 1.30 -> 0.80, four lots the same, but
    // random graphs 0.99 and 1.15), in turn by the block's warps, and then the hubs' segments.  A round that advances (a new thr) takes the
    // items marked far that are below thr.
    __device__ __forceinline__ void work(uint32_t n_items, bool advance) {
        const uint32_t words = (n_items + 31u) / 32u, sh = 16u * (lane & 1u);
        const uint32_t turns = n_items > V ? BT / 16u : BT / 32u;
        const uint32_t few = min((words + turns - 1u) / turns, 16u);  // words at a time
        uint32_t nq = 0;
        for (;;) {
            uint32_t c = 0;
            if (lane == 0) c = atomicAdd(&M.next, few);
            c = __shfl_sync(0xFFFFFFFFu, c, 0);
            if (c >= words) break;
            const uint32_t wi = c + lane / 2u, first = wi * 32u + sh;
            uint32_t take = 0;
            if (wi < words && lane < 2u * few) {
                if (advance) {
                    for (uint32_t t = *reinterpret_cast<volatile uint32_t*>(&I.far[wi]) >> sh & 0xFFFFu; t; t &= t - 1u) {
                        const uint32_t j = __ffs(t) - 1;
                        const uint32_t d = I.get(first + j);
                        if (d < thr)
                            take |= 1u << j;
                        else
                            low = min(low, d);
                    }
                    if (take) atomicAnd(&I.far[wi], ~(take << sh));
                } else {
                    take = *reinterpret_cast<volatile uint32_t*>(&I.near[wi]) >> sh & 0xFFFFu;
                    if (take) {
                        atomicAnd(&I.near[wi], ~(take << sh));
                        if (*reinterpret_cast<volatile uint32_t*>(&I.far[wi]) & take << sh) atomicAnd(&I.far[wi], ~(take << sh));
                    }
                }
            }
            for (uint32_t b; (b = __ballot_sync(0xFFFFFFFFu, take != 0u)) != 0u;) {
                if (take) {
                    M.q[wid][nq + __popc(b & ((1u << lane) - 1u))] = first + __ffs(take) - 1u;
                    take &= take - 1u;
                }
                nq += __popc(b);
                if (nq >= 32u) {
                    relax_items(32u);
                    nq -= 32u;
                    const uint32_t x = M.q[wid][32u + lane];
                    __syncwarp();
                    M.q[wid][lane] = x;
                    __syncwarp();
                }
            }
        }
        if (nq) relax_items(nq);
        __syncthreads();
        const uint32_t nh = min(M.nhub[par], HCAP);
        for (uint32_t i = 0; nh;) {
            if (lane == 0) i = atomicAdd(&M.hnext[par], 1u);
            i = __shfl_sync(0xFFFFFFFFu, i, 0);
            if (i >= nh) break;
            const uint2 h = M.hub[i];
            if (h.x == NONE) continue;
            const uint32_t item = h.x, v = I.vertex(item), s = h.y * HUB;
            const uint32_t beg = __ldg(&row_ptr[v]) + s, left = __ldg(&row_ptr[v + 1]) - beg;
            if (lane == 0)
                M.row[wid][0] = make_uint4(beg, item - v, I.get(item), 0u);
            __syncwarp();
            run(min(left, HUB), lane == 0 ? 0u : 0xFFFFFFFFu);
            __syncwarp();
        }
    }
};

// SSSP_EOVERFLOW if a candidate from a final distance does not fit.  (One that was met on the way may be from
// a distance that was lowered later: more of them than in the general kernel, whose buckets are narrower.)
// Inlined: a call's stack costs the launch 13 us.
template <class W>
__device__ __forceinline__ void judge_overflow(const uint32_t* dist, uint32_t V, uint32_t S, const uint32_t* row_ptr,
                                            const uint32_t* col, const uint32_t* w, WsHeader* hdr) {
    const uint32_t lane = threadIdx.x & 31u;
    for (uint32_t u = threadIdx.x >> 5; u < V; u += blockDim.x >> 5) {
        uint32_t most = 0;
        bool reached = false, bad = false;
        for (uint32_t s = 0; s < S; ++s) {
            const uint32_t d = dist[s * V + u];
            if (d < W::inf_out()) reached = true, most = max(most, d);
        }
        if (!reached) continue;
        for (uint32_t e = row_ptr[u] + lane; e < row_ptr[u + 1u]; e += 32u) {
            uint32_t z;
            bad = bad || (col[e] < V && W::weight_ok(w[e]) && !W::add(most, w[e], z));
        }
        if (bad) set_status(hdr, SSSP_EOVERFLOW);
    }
}

// One unit, by the block.
template <class W, uint32_t BT>
__device__ __forceinline__ void solve_unit(const BatchSmem& B, Mem<BT / 32>& M, uint32_t* dsm, uint64_t deadline) {
    const uint32_t tid = threadIdx.x, lane = tid & 31u, wid = tid >> 5;
    const BatchUnit& U = M.unit;
    const uint32_t V = U.V, S = U.S, n_items = S * V, words = (n_items + 31u) / 32u;
    Items I;
    I.dist = dsm;
    I.near = dsm + n_items;
    I.far = I.near + words;
    I.V = V;
    for (uint32_t i = tid; i < n_items; i += BT) I.dist[i] = W::inf_out();
    for (uint32_t i = tid; i < words; i += BT) I.near[i] = I.far[i] = 0u;
    __syncthreads();
    if (tid < S) {
        const uint32_t i = tid * V + U.src[tid];
        I.dist[i] = 0u;
        I.mark(i, true);
    }
    __syncthreads();

    Round<W, BT> R{I, M, B.row_ptr + U.row_off, B.col + U.edge_off, B.w + U.edge_off, V, lane, wid, 0, 0, 0, 0, 0, 0, 0, 0, 0ull};
    uint32_t rounds = 0;
    bool stopped = false, advance = false;
    R.thr = W::bucket_end(0u, B.delta_bits);
    R.low = W::inf_out();
    for (uint32_t par = 0;; par ^= 1u) {
        R.par = par;
        R.any_near = 0u;
        R.work(n_items, advance);
        const uint32_t low = __reduce_min_sync(0xFFFFFFFFu, R.low);
        const bool any_near = __any_sync(0xFFFFFFFFu, R.any_near);
        if (lane == 0) {
            atomicMin(&M.low[par], low);
            if (any_near) atomicOr(&M.flags[par], 1u);
        }
        if (tid == 0) {  // for the next round
            M.next = M.hnext[par ^ 1u] = M.nhub[par ^ 1u] = M.flags[par ^ 1u] = 0u;
            M.low[par ^ 1u] = W::inf_out();
            if (globaltimer_ns() > deadline) atomicOr(&M.flags[par], 2u);
        }
        __syncthreads();
        const uint32_t least = M.low[par], flags = M.flags[par];
        ++rounds;
        stopped = flags & 2u;
        advance = !(flags & 1u);
        if (stopped || (advance && least == W::inf_out())) break;
        if (advance) {
            R.thr = W::bucket_end(least, B.delta_bits);
            R.low = W::inf_out();
        }
    }
    if (stopped && tid == 0) {
        set_status(B.hdr, SSSP_ETIMEOUT);
        atomicExch(&B.hdr->abort_flag, 1u);
    }

    for (uint32_t s = 0; s < S; ++s) {
        uint32_t n = 0;
        for (uint32_t v = tid; v < V; v += BT) {
            const uint32_t d = I.dist[s * V + v];
            n += d < W::inf_out();
            B.dist[U.out[s] + v] = d;
            if (B.pred) B.pred[U.out[s] + v] = NONE;
        }
        n = __reduce_add_sync(0xFFFFFFFFu, n);
        if (lane == 0 && n) atomicAdd(&M.reach[s], n);
    }
    const bool over = __syncthreads_or((int)(R.bad & 2u));
    // The walk over all edges is for the copies that have reached many vertices (an isolated source of 40,000
    // vertices and 1.4 M edges: 229 -> 19 us); the rows of the few that the others have reached are gone through.
    uint32_t many = 0;
    for (uint32_t s = 0; s < S; ++s) many |= M.reach[s] > V / 8u ? 1u << s : 0u;
    if (B.pred && !stopped) {
        for (uint32_t m = ~many & ((1u << S) - 1u); m; m &= m - 1u) {
            const uint32_t s = __ffs(m) - 1u;
            if (M.reach[s] < 2u) continue;
            for (uint32_t v0 = wid * 32u; v0 < V; v0 += BT) {
                const uint32_t mine = v0 + lane < V ? I.get(s * V + v0 + lane) : W::inf_out();
                for (uint32_t b = __ballot_sync(0xFFFFFFFFu, mine < W::inf_out()); b; b &= b - 1u) {
                    const uint32_t l = __ffs(b) - 1u, d = __shfl_sync(0xFFFFFFFFu, mine, l), end = __ldg(&R.row_ptr[v0 + l + 1u]);
                    for (uint32_t e = __ldg(&R.row_ptr[v0 + l]) + lane; e < end; e += 32u) {
                        const uint32_t v = __ldg(&R.col[e]), x = __ldg(&R.w[e]);
                        uint32_t c;
                        if (v < V && W::weight_ok(x) && W::add(d, x, c) && c == I.get(s * V + v))
                            atomicMin(&B.pred[U.out[s] + v], v0 + l);
                    }
                }
            }
        }
    }
    if (B.pred && many && !stopped) {
        uint32_t* const rows = reinterpret_cast<uint32_t*>(M.row[wid]);
        RowWalk walk{R.row_ptr, V, rows, rows + 32};
        const uint32_t first = R.row_ptr[0], E = R.row_ptr[V] - first;
        const uint32_t per = (E / (BT / 32u) + 32u) & ~31u;
        const unsigned long long k = (unsigned long long)wid * per;
        if (k < E) {
            const uint32_t e0 = first + (uint32_t)k, e1 = e0 + min(per, E - (uint32_t)k);
            walk.seek(e0);
            uint32_t v[2], x[2];
            auto fetch = [&](uint32_t eb, int j) {
                v[j] = NONE;
                if (eb + lane < e1) v[j] = __ldg(&R.col[eb + lane]), x[j] = __ldg(&R.w[eb + lane]);
            };
            auto step = [&](uint32_t eb, int j) {
                const uint32_t u = walk.step(eb, e1);
                if (v[j] >= V || !W::weight_ok(x[j])) return;
                for (uint32_t m = many; m; m &= m - 1u) {
                    const uint32_t s = __ffs(m) - 1u;
                    uint32_t c;
                    if (W::add(I.get(s * V + u), x[j], c) && c == I.get(s * V + v[j]))
                        atomicMin(&B.pred[U.out[s] + v[j]], u);
                }
            };
            fetch(e0, 0);
            for (uint32_t eb = e0; eb < e1; eb += 64u) {
                fetch(eb + 32u, 1);
                step(eb, 0);
                __syncwarp();
                fetch(eb + 64u, 0);
                if (eb + 32u < e1) step(eb + 32u, 1);
                __syncwarp();
            }
        }
    }
    if (__any_sync(0xFFFFFFFFu, R.bad & 1u) && lane == 0) set_status(B.hdr, SSSP_EINVAL);
    if (over && !stopped) judge_overflow<W>(I.dist, V, S, R.row_ptr, R.col, R.w, B.hdr);
    // edges_scanned, atomics, improved, activations (but for the sources, an item is relaxed as often as
    // it is marked), rounds, vertices
    R.n_at = __reduce_add_sync(0xFFFFFFFFu, R.n_at);
    R.n_imp = __reduce_add_sync(0xFFFFFFFFu, R.n_imp);
    R.n_vert = __reduce_add_sync(0xFFFFFFFFu, R.n_vert);
    if (lane == 0) {
        atomicAdd(&M.stats[0], R.n_edges);
        atomicAdd(&M.stats[1], (unsigned long long)R.n_at);
        atomicAdd(&M.stats[2], (unsigned long long)R.n_imp);
        atomicAdd(&M.stats[5], (unsigned long long)R.n_vert);
        if (wid == 0) M.stats[4] = rounds;
    }
    __syncthreads();
    if (tid < 6u) {
        unsigned long long n = M.stats[tid == 3u ? 5u : tid];
        if (tid == 3u) n -= min(n, (unsigned long long)S);
        if (n) atomicAdd(&B.hdr->stats[tid], n);
    }
}

template <class W, uint32_t BT>
__global__ void __launch_bounds__(BT, 1024 / BT) k_batch(BatchSmem B) {
    extern __shared__ __align__(16) uint32_t dsm[];
    __shared__ __align__(16) Mem<BT / 32> M;
    const uint32_t tid = threadIdx.x;
    uint64_t deadline = 0;
    if (tid == 0) {  // (all blocks of the call share its first block's start)
        const unsigned long long now = globaltimer_ns(), first = atomicCAS(&B.hdr->begin, 0ull, now);
        deadline = (first ? first : now) + LIMIT_FACTOR * B.timeout_ns;
    }
    for (;;) {
        if (tid == 0) {
            M.unit_at = ld_relaxed(&B.hdr->abort_flag) ? B.n_units : atomicAdd(&B.hdr->unit_next, 1u);
            M.next = M.hnext[0] = M.hnext[1] = M.nhub[0] = M.nhub[1] = M.flags[0] = M.flags[1] = 0u;
            M.low[0] = M.low[1] = W::inf_out();
        }
        if (tid < 6u) M.stats[tid] = 0ull;
        if (tid < BATCH_COPIES) M.reach[tid] = 0u;
        __syncthreads();
        if (M.unit_at >= B.n_units) break;
        if (tid < sizeof(BatchUnit) / 4)
            reinterpret_cast<uint32_t*>(&M.unit)[tid] = reinterpret_cast<const uint32_t*>(&B.units[M.unit_at])[tid];
        __syncthreads();
        solve_unit<W, BT>(B, M, dsm, deadline);
        __syncthreads();
    }
}

size_t smem_bytes(uint32_t items) { return 4 * ((size_t)items + items / 16 + 2); }

uint32_t threads_for(uint32_t items) { return items <= BATCH_SMALL ? 512u : 1024u; }

const void* kernel_for(int wtype, uint32_t items) {
    if (threads_for(items) == 512u)
        return wtype == SSSP_W_F32 ? (const void*)k_batch<WF32, 512> : (const void*)k_batch<WU32, 512>;
    return wtype == SSSP_W_F32 ? (const void*)k_batch<WF32, 1024> : (const void*)k_batch<WU32, 1024>;
}

}  // namespace

cudaError_t batch_smem_setup(int wtype, uint32_t items, int* blocks_per_sm) {
    const void* k = kernel_for(wtype, items);
    const uint32_t most = items <= BATCH_SMALL ? BATCH_SMALL : BATCH_ITEMS;
    const cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_bytes(most));
    if (e != cudaSuccess) return e;
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, k, (int)threads_for(items), smem_bytes(items));
}

void launch_batch_smem(const BatchSmem& B, cudaStream_t st) {
    const size_t smem = smem_bytes(B.items);
    if (threads_for(B.items) == 512u) {
        if (B.wtype == SSSP_W_F32)
            k_batch<WF32, 512><<<B.grid, 512, smem, st>>>(B);
        else
            k_batch<WU32, 512><<<B.grid, 512, smem, st>>>(B);
    } else {
        if (B.wtype == SSSP_W_F32)
            k_batch<WF32, 1024><<<B.grid, 1024, smem, st>>>(B);
        else
            k_batch<WU32, 1024><<<B.grid, 1024, smem, st>>>(B);
    }
}

}  // namespace sssp
