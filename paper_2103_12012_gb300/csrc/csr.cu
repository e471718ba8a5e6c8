// K1 CSR builder, K2 block partitioner, edge compaction.
//
// K1 turns a raw edge list into the canonical adjacency (Sec. III.A's Padj for all partitions at
// once): keys (tail, head) are radix-sorted with their input index (a stable sort, so equal keys
// keep input order; self-loops and bad ids make no pair), runs of equal keys become one edge whose
// weight is the run's minimum (lowest input index on ties: the minimum of weight bits << 32 | index),
// and row_ptr is filled from the run boundaries.  After the sort (sort.cu) the runs are counted per
// tile, the counts scanned, and one kernel gathers the weights, reduces the runs in shared memory and
// writes the edges; the runs that cross tiles (at most one a tile) are finished by a last small one.
// R-MAT scale 22 (67 M edges): 2.6 -> 1.3 ms after the sort, where run minima were 64-bit atomics on
// an array of their own and row numbers came from 64-bit divisions.  k_csr_emit (1.2 ms) is bound by
// the random gather of the weights (8 a thread in flight; 4: the same, 16: 1.5 ms, fewer warps).
#include <algorithm>

#include "common.cuh"
#include "internal.h"
#include "rowwalk.cuh"

namespace sssp {
namespace {

__host__ __device__ inline uint32_t bits_for(unsigned long long x) {
    uint32_t b = 0;
    while (b < 64 && (x >> b) != 0ull) ++b;
    return b;
}

constexpr uint32_t EMIT_THREADS = 256, EMIT_WARPS = EMIT_THREADS / 32, EMIT_STEPS = 8;
constexpr uint32_t EMIT_RUN = 32 * EMIT_STEPS, EMIT_TILE = EMIT_WARPS * EMIT_RUN;  // sorted pairs of a warp, a block
constexpr unsigned long long NO_EDGE = ~0ull;
constexpr uint32_t GAP = 16;  // rows without an edge before one: more are filled in by the warp together

struct CsrWs {
    WsHeader* hdr;
    unsigned long long* keys[2];
    uint32_t* vals[2];
    uint32_t* totals;          // [tiles] runs that start in a tile, then before it
    unsigned long long* lead;  // [tiles] minimum of a tile's pairs before its first run
    void* sort;                // sort temporaries
    void* scan;
    uint64_t tiles;
    size_t total;
};

CsrWs carve_csr(void* ws, uint32_t V, uint64_t n) {
    (void)V;
    CsrWs c{};
    char* p = static_cast<char*>(ws);
    size_t off = 0;
    auto take = [&](size_t bytes) {
        char* r = p ? p + off : nullptr;
        off += align_up(bytes, 256);
        return r;
    };
    c.tiles = (n + EMIT_TILE - 1) / EMIT_TILE;
    c.hdr = reinterpret_cast<WsHeader*>(take(WS_HEADER_BYTES));
    for (int i = 0; i < 2; ++i) c.keys[i] = reinterpret_cast<unsigned long long*>(take(8 * n));
    for (int i = 0; i < 2; ++i) c.vals[i] = reinterpret_cast<uint32_t*>(take(4 * n));
    c.totals = reinterpret_cast<uint32_t*>(take(4 * (c.tiles + 1)));
    c.lead = reinterpret_cast<unsigned long long*>(take(8 * (c.tiles + 1)));
    c.sort = take(sort_temp_bytes(n));
    c.scan = take(scan_temp_bytes(c.tiles + 1));
    c.total = off;
    return c;
}

// runs that start in each tile (totals[tiles] = 0 for the scan's last word)
__global__ void __launch_bounds__(EMIT_THREADS) k_csr_runs(const unsigned long long* __restrict__ count,
                                                           const unsigned long long* __restrict__ keys, uint32_t* totals,
                                                           const uint32_t* run) {
    __shared__ uint32_t sum;
    if (run && !*run) return;
    const unsigned long long n = *count, base = (unsigned long long)blockIdx.x * EMIT_TILE;
    if (threadIdx.x == 0) sum = 0;
    __syncthreads();
    uint32_t mine = 0;
    for (uint32_t i = threadIdx.x; i < EMIT_TILE; i += EMIT_THREADS) {
        const unsigned long long at = base + i;
        if (at < n && (at == 0 || keys[at - 1] != keys[at])) ++mine;
    }
    mine = __reduce_add_sync(0xFFFFFFFFu, mine);
    if ((threadIdx.x & 31u) == 0 && mine) atomicAdd(&sum, mine);
    __syncthreads();
    if (threadIdx.x == 0) totals[blockIdx.x] = sum;
}

// Rows [from, from + rows) start at edge r: by the warp (67 M vertices with 1,000 edges, the whole call: 34.4 ms with a
// thread for the rows before its edge -> 4.9 ms; 1 M vertices, all 16 M edges from one: 5.6 -> 1.4).
__device__ __forceinline__ void fill_rows(uint32_t* row_ptr, uint32_t from, uint32_t rows, uint32_t r) {
    for (uint32_t u = threadIdx.x & 31u; u < rows; u += 32u) row_ptr[from + u] = r;
}

// The edges of a tile's runs.  Each warp marks the run starts of its 256 pairs with ballots; a start
// writes its head and the row_ptr entries up to its tail, and every pair lowers its run's (weight
// bits << 32 | index) in shared memory, from which weights and indices go out in run order.
// (before: runs before each tile, one word past the last tile the number of edges)
__global__ void __launch_bounds__(EMIT_THREADS) k_csr_emit(uint32_t V, uint32_t bits,
                                                           const unsigned long long* __restrict__ count,
                                                           const unsigned long long* __restrict__ keys,
                                                           const uint32_t* __restrict__ vals, const uint32_t* __restrict__ w,
                                                           const uint32_t* __restrict__ before, unsigned long long* lead,
                                                           uint32_t tiles, uint32_t* row_ptr, uint32_t* col,
                                                           uint32_t* w_out, uint32_t* eid, uint32_t* E_out,
                                                           const WsHeader* hdr, const uint32_t* sorted) {
    if (sorted && !*sorted) return;
    __shared__ unsigned long long best[EMIT_TILE + 1];  // [0]: pairs of a run that starts in an earlier tile
    __shared__ uint32_t wsum[EMIT_WARPS];
    const uint32_t tid = threadIdx.x, lane = tid & 31u, wid = tid >> 5;
    const unsigned long long n = *count, tile0 = (unsigned long long)blockIdx.x * EMIT_TILE;
    const bool failed = hdr->status == SSSP_EINTERNAL;  // the sort gave up: its pairs mean nothing
    if (blockIdx.x == 0 && tid == 0) *E_out = failed ? 0u : before[tiles];
    if (tile0 >= n || failed) {
        if (tid == 0) lead[blockIdx.x] = NO_EDGE;
        return;
    }
    const unsigned long long first = tile0 + wid * EMIT_RUN + lane;
    unsigned long long k[EMIT_STEPS];
    uint32_t v[EMIT_STEPS], starts[EMIT_STEPS];  // starts: ballots (uniform)
    unsigned long long last = first - lane < n && first - lane ? keys[first - lane - 1] : NO_EDGE;  // key before the step
    const unsigned long long last0 = last;
    uint32_t mine = 0;
#pragma unroll
    for (uint32_t j = 0; j < EMIT_STEPS; ++j) {
        const unsigned long long at = first + 32u * j;
        k[j] = at < n ? keys[at] : NO_EDGE;
        v[j] = at < n ? vals[at] : 0u;
    }
    uint32_t x32[EMIT_STEPS];  // the weights, gathered together
#pragma unroll
    for (uint32_t j = 0; j < EMIT_STEPS; ++j) x32[j] = __ldg(&w[v[j]]);
#pragma unroll
    for (uint32_t j = 0; j < EMIT_STEPS; ++j) {
        unsigned long long prev = __shfl_up_sync(0xFFFFFFFFu, k[j], 1);
        if (lane == 0) prev = last;
        last = __shfl_sync(0xFFFFFFFFu, k[j], 31);
        starts[j] = __ballot_sync(0xFFFFFFFFu, k[j] != NO_EDGE && k[j] != prev);
        mine += __popc(starts[j]);
    }
    if (lane == 0) wsum[wid] = mine;
    for (uint32_t i = tid; i <= EMIT_TILE; i += EMIT_THREADS) best[i] = NO_EDGE;
    __syncthreads();
    uint32_t run = 0, all = 0;  // runs of the tile before this warp's
    for (uint32_t i = 0; i < EMIT_WARPS; ++i) {
        if (i < wid) run += wsum[i];
        all += wsum[i];
    }
    const uint32_t base = before[blockIdx.x], R = before[tiles];
    const unsigned long long hmask = (1ull << bits) - 1ull;
    last = last0;
#pragma unroll
    for (uint32_t j = 0; j < EMIT_STEPS; ++j) {
        unsigned long long prev = __shfl_up_sync(0xFFFFFFFFu, k[j], 1);
        if (lane == 0) prev = last;
        last = __shfl_sync(0xFFFFFFFFu, k[j], 31);
        const uint32_t at = run + __popc(starts[j] & (0xFFFFFFFFu >> (31u - lane)));  // runs up to this pair
        run += __popc(starts[j]);
        uint32_t from = 0, rows = 0;  // that start at this pair
        if (k[j] != NO_EDGE) {
            const unsigned long long x = (unsigned long long)x32[j] << 32 | v[j];
            const bool alone = (starts[j] >> lane & 1u) && lane < 31u && (starts[j] >> (lane + 1u) & 1u);
            if (alone)
                best[at] = x;
            else
                atomicMin(&best[at], x);
            if (starts[j] >> lane & 1u) {
                const uint32_t r = base + at - 1u, s = (uint32_t)(k[j] >> bits);
                col[r] = (uint32_t)(k[j] & hmask);
                from = prev == NO_EDGE ? 0u : (uint32_t)(prev >> bits) + 1u;
                rows = s + 1u - from;
                if (rows <= GAP)
                    for (uint32_t u = from; u <= s; ++u) row_ptr[u] = r;
            }
        }
        for (uint32_t m = __ballot_sync(0xFFFFFFFFu, rows > GAP); m; m &= m - 1u) {
            const uint32_t l = __ffs(m) - 1u;
            fill_rows(row_ptr, __shfl_sync(0xFFFFFFFFu, from, l), __shfl_sync(0xFFFFFFFFu, rows, l),
                      __shfl_sync(0xFFFFFFFFu, base + at - 1u, l));
        }
        if (first - lane + 32u * j < n && first - lane + 32u * (j + 1u) >= n) {  // the rows after the last
            const uint32_t s = __shfl_sync(0xFFFFFFFFu, (uint32_t)(k[j] >> bits), (uint32_t)(n - 1u) & 31u);
            fill_rows(row_ptr, s + 1u, V - s, R);
        }
    }
    __syncthreads();
    if (tid == 0) lead[blockIdx.x] = best[0];
    for (uint32_t i = tid; i < all; i += EMIT_THREADS) {
        const unsigned long long x = best[i + 1u];
        w_out[base + i] = (uint32_t)(x >> 32);
        if (eid) eid[base + i] = (uint32_t)x;
    }
}

// a run that crosses into tile t and starts before it: the minimum of what the tiles from t on hold of it
__global__ void k_csr_cross(uint32_t tiles, const uint32_t* __restrict__ before,
                            const unsigned long long* __restrict__ lead, uint32_t* w_out, uint32_t* eid, const uint32_t* run) {
    const uint32_t t = blockIdx.x * blockDim.x + threadIdx.x;
    if (run && !*run) return;
    if (t == 0 || t >= tiles || lead[t] == NO_EDGE || before[t] == before[t - 1]) return;
    unsigned long long m = lead[t];
    for (uint32_t x = t; before[x + 1] == before[x] && x + 1 < tiles && lead[x + 1] != NO_EDGE; ++x) m = min(m, lead[x + 1]);
    const uint32_t r = before[t] - 1u;
    if (m < ((unsigned long long)w_out[r] << 32 | (eid ? eid[r] : 0xFFFFFFFFu))) {
        w_out[r] = (uint32_t)(m >> 32);
        if (eid) eid[r] = (uint32_t)m;
    }
}

// Block partition bounds and inter-edge counts.  A partition is a block of vertices, so its edges
// are one contiguous range of the CSR, and an edge leaves it when its head is outside the block: a
// warp takes `range` consecutive edges, finds the partition of the first by a 32-way search over
// the partitions' first edges, and counts partition by partition, four loads a lane in flight, with
// one atomic per partition it meets.  Nothing is looked up per row.  R-MAT scale 22, 148 partitions:
// 0.73 -> 0.06 ms (65 M heads read once, 4.2 TB/s; bound by HBM).
__global__ void __launch_bounds__(256) k_partition(uint32_t V, uint32_t E, uint32_t P, unsigned long long B, uint32_t range,
                                                   const uint32_t* __restrict__ row_ptr,
                                                   const uint32_t* __restrict__ col, uint32_t* bounds,
                                                   unsigned long long* inter) {
    const uint32_t gtid = blockIdx.x * blockDim.x + threadIdx.x, lane = threadIdx.x & 31u;
    for (unsigned long long p = gtid; p <= P; p += (unsigned long long)gridDim.x * blockDim.x)
        bounds[p] = (uint32_t)(p * B < V ? p * B : V);
    const unsigned long long first = (unsigned long long)(gtid >> 5) * range;
    if (!inter || first >= E) return;
    auto start = [&](uint32_t p) {  // first edge of partition p
        const unsigned long long v = p * B;
        return __ldg(&row_ptr[v < V ? v : V]);
    };
    uint32_t e = (uint32_t)first;
    const uint32_t e1 = (uint32_t)min(first + range, (unsigned long long)E);
    uint32_t p = 0, len = P;  // the last partition whose first edge is <= e holds it
    while (len > 1u) {
        const uint32_t step = (len + 31u) / 32u, i = lane * step;
        const bool le = i < len && start(p + i) <= e;
        const uint32_t k = 31u - (uint32_t)__clz(__ballot_sync(0xFFFFFFFFu, le) | 1u);
        p += k * step;
        len = min(step, len - k * step);
    }
    while (e < e1) {
        const uint32_t end = p + 1u < P ? min(start(p + 1u), e1) : e1;
        const unsigned long long lo = p * B;
        uint32_t cnt = 0;
        for (uint32_t i = e + lane; i < end;) {
            const uint32_t n = min((end - i + 31u) / 32u, 4u);
            uint32_t c[4];
#pragma unroll
            for (uint32_t j = 0; j < 4u; ++j) c[j] = j < n ? __ldg(&col[i + 32u * j]) : (uint32_t)lo;
#pragma unroll
            for (uint32_t j = 0; j < 4u; ++j) cnt += (unsigned long long)c[j] - lo >= B;
            if (end - i <= 128u) break;
            i += 128u;
        }
        cnt = __reduce_add_sync(0xFFFFFFFFu, cnt);
        if (lane == 0 && cnt) atomicAdd(&inter[p], (unsigned long long)cnt);
        e = max(e, end);
        ++p;
    }
}

// Compaction, in tiles of KEEP_TILE edges.  First the keep bytes become one bit an edge, with the
// kept edges before each word of 32 within its tile and the tile's total; then, with the totals
// scanned, the kept edges are moved word by word (coalesced loads and stores, loads of dropped edges
// left out) and a row's new start is the rank of its old one: tile offset + word count + bits below.
// The mask and the counts are E / 4 bytes, where a word per edge and its scan moved 16 E.  R-MAT scale
// 22, 4% dropped: 0.77 -> 0.29 ms (k_compact 4.9 TB/s of the 20 bytes an edge it reads and writes).
constexpr uint32_t KEEP_THREADS = 256, KEEP_WORDS = 4 * KEEP_THREADS, KEEP_TILE = 32 * KEEP_WORDS;
constexpr uint32_t KEEP_FLY = 8;  // k_compact 269 us on R-MAT scale 22 (4: 297, 16: 332)

// ALIGNED: keep is 16-byte aligned (a lane loads 32 bytes); else byte by byte
template <bool ALIGNED>
__global__ void __launch_bounds__(KEEP_THREADS) k_keep_bits(uint32_t E, const uint8_t* __restrict__ keep, uint32_t* mask,
                                                            uint32_t* before, uint32_t* totals) {
    __shared__ uint32_t wsum[KEEP_THREADS / 32];
    const uint32_t lane = threadIdx.x & 31u, wid = threadIdx.x >> 5;
    const uint32_t words = E / 32u + 1u;  // (the last word, perhaps empty, holds the rank of E)
    uint32_t run = 0;
    for (uint32_t k = 0; k < KEEP_WORDS; k += KEEP_THREADS) {
        const uint32_t wd = blockIdx.x * KEEP_WORDS + k + threadIdx.x;
        uint32_t bits = 0;
        if (wd < words) {
            const uint32_t e0 = wd * 32u, n = min(32u, E - e0);
            if (ALIGNED && n == 32u) {
                const uint4* p = reinterpret_cast<const uint4*>(keep + e0);
                const uint4 a = __ldg(p), b = __ldg(p + 1);
                const uint32_t x[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
#pragma unroll
                for (uint32_t i = 0; i < 8u; ++i) {
                    const uint32_t nz = __vcmpne4(x[i], 0u) & 0x01010101u;  // a byte's bit 0: it is not 0
                    bits |= (nz * 0x01020408u >> 24 & 15u) << (4u * i);
                }
            } else {
                for (uint32_t i = 0; i < n; ++i) bits |= (keep[e0 + i] != 0u ? 1u : 0u) << i;
            }
        }
        const uint32_t c = __popc(bits);
        uint32_t inc = c;
#pragma unroll
        for (uint32_t o = 1; o < 32u; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, inc, o);
            if (lane >= o) inc += y;
        }
        if (lane == 31u) wsum[wid] = inc;
        __syncthreads();
        uint32_t base = run, all = 0;
        for (uint32_t i = 0; i < KEEP_THREADS / 32u; ++i) {
            if (i < wid) base += wsum[i];
            all += wsum[i];
        }
        if (wd < words) {
            mask[wd] = bits;
            before[wd] = base + inc - c;
        }
        run += all;
        __syncthreads();
    }
    if (threadIdx.x == 0) totals[blockIdx.x] = run;
}

// offsets: exclusive scan of the totals
__global__ void __launch_bounds__(256) k_compact(uint32_t V, uint32_t E, const uint32_t* __restrict__ row_ptr,
                                                 const uint32_t* __restrict__ col, const uint32_t* __restrict__ w,
                                                 const uint32_t* __restrict__ mask, const uint32_t* __restrict__ before,
                                                 const uint32_t* __restrict__ offsets, uint32_t* row_ptr_out,
                                                 uint32_t* col_out, uint32_t* w_out, uint32_t* emap, uint32_t* E_out) {
    const uint32_t gtid = blockIdx.x * blockDim.x + threadIdx.x, lane = threadIdx.x & 31u;
    const uint32_t warps = (gridDim.x * blockDim.x) >> 5, words = E / 32u + 1u;
    for (uint32_t w0 = (gtid >> 5) * 32u; w0 < words; w0 += warps * 32u) {  // 32 words, one a lane
        const uint32_t wd = w0 + lane;
        const uint32_t m = wd < words ? __ldg(&mask[wd]) : 0u;
        const uint32_t at = wd < words ? __ldg(&offsets[wd / KEEP_WORDS]) + __ldg(&before[wd]) : 0u;
        for (uint32_t i0 = 0; i0 < 32u; i0 += KEEP_FLY) {  // the loads of KEEP_FLY words in flight together
            uint32_t c[KEEP_FLY], x[KEEP_FLY];
#pragma unroll
            for (uint32_t i = 0; i < KEEP_FLY; ++i) {
                const uint32_t mi = __shfl_sync(0xFFFFFFFFu, m, i0 + i), e = (w0 + i0 + i) * 32u + lane;
                if (mi >> lane & 1u) c[i] = __ldg(&col[e]), x[i] = __ldg(&w[e]);
            }
#pragma unroll
            for (uint32_t i = 0; i < KEEP_FLY; ++i) {
                const uint32_t mi = __shfl_sync(0xFFFFFFFFu, m, i0 + i), ai = __shfl_sync(0xFFFFFFFFu, at, i0 + i);
                if (mi >> lane & 1u) {
                    const uint32_t j = ai + __popc(mi & ((1u << lane) - 1u));
                    col_out[j] = c[i];
                    w_out[j] = x[i];
                    if (emap) emap[j] = (w0 + i0 + i) * 32u + lane;
                }
            }
        }
    }
    auto rank = [&](uint32_t e) {  // kept edges before e (e <= E)
        const uint32_t wd = e >> 5;
        return __ldg(&offsets[wd / KEEP_WORDS]) + __ldg(&before[wd]) + __popc(__ldg(&mask[wd]) & ((1u << (e & 31u)) - 1u));
    };
    for (uint64_t u = gtid; u <= V; u += gridDim.x * blockDim.x) row_ptr_out[u] = rank(row_ptr[u]);
    if (gtid == 0) *E_out = rank(E);
}

// ---- locality layout: renumber vertices inside each block partition by degree

constexpr uint32_t COO_RANGE = 1024;
constexpr uint32_t LAY_TILE = 1024, LAY_SEG = 2048;     // stored edges of a block; longest segment
constexpr uint32_t LAY_DEEP = 256;                      // edges this far into their segments are counted
constexpr uint32_t LAY_CAP = LAY_TILE + LAY_SEG + 32u;  // stored edges that a block holds

__global__ void k_lay_deg(uint32_t V, const uint32_t* __restrict__ row_ptr, uint32_t* deg) {
    for (uint32_t v = blockIdx.x * blockDim.x + threadIdx.x; v < V; v += gridDim.x * blockDim.x)
        deg[v] = row_ptr[v + 1] - row_ptr[v];
}

// In-degrees; and whether the rows can be sorted segment by segment (k_lay_rows): they are as sssp_build_csr
// makes them, no segment is longer than LAY_SEG, and (k_lay_keys) few edges are LAY_DEEP or more into theirs.
__global__ void __launch_bounds__(256) k_lay_check(uint32_t V, uint32_t E, uint32_t B, const uint32_t* __restrict__ row_ptr,
                                                   const uint32_t* __restrict__ col, const uint32_t* __restrict__ w, int wtype,
                                                   uint32_t* deg, WsHeader* hdr) {
    __shared__ uint32_t rows[8][32], starts[8][32];
    const uint32_t lane = threadIdx.x & 31u, wid = threadIdx.x >> 5;
    const unsigned long long first = ((unsigned long long)blockIdx.x * 8u + wid) * COO_RANGE;
    if (first >= E) return;
    const uint32_t e0 = (uint32_t)first, e1 = (uint32_t)min(first + COO_RANGE, (unsigned long long)E);
    RowWalk walk{row_ptr, V, rows[wid], starts[wid]};
    walk.seek(e0);
    uint32_t before = e0 ? __ldg(&col[e0 - 1u]) : 0u;  // head of the edge before the step
    bool odd = false;
    uint32_t deep = 0;
    uint32_t v = e0 + lane < e1 ? __ldg(&col[e0 + lane]) : 0u;
    for (uint32_t eb = e0; eb < e1 && eb >= e0; eb += 32u) {
        const uint32_t e = eb + lane, u = walk.step(eb, e1), x = v;
        if (e1 - eb > 32u + lane) v = __ldg(&col[e + 32u]);  // the next step's
        uint32_t y = __shfl_up_sync(0xFFFFFFFFu, x, 1);
        if (lane == 0) y = before;
        before = __shfl_sync(0xFFFFFFFFu, x, 31);
        if (e < e1) {
            const uint32_t at = e - __ldg(&row_ptr[u]), wt = __ldg(&w[e]);
            odd = odd || x >= V || x == u || (at && y >= x) || !(wtype == SSSP_W_F32 ? WF32::weight_ok(wt) : WU32::weight_ok(wt));
            if (at >= LAY_DEEP && __ldg(&col[e - LAY_DEEP]) / B == x / B) {
                ++deep;
                if (at >= LAY_SEG && __ldg(&col[e - LAY_SEG]) / B == x / B) odd = true;
            }
            if (x < V) atomicAdd(&deg[x], 1u);
        }
    }
    if (first == 0 && (row_ptr[0] != 0u || row_ptr[V] != E)) odd = true;
    if (__any_sync(0xFFFFFFFFu, odd) && lane == 0) hdr->lay_general = 1u;
    deep = __reduce_add_sync(0xFFFFFFFFu, deep);
    if (deep && lane == 0) atomicAdd(&hdr->lay_deep, deep);
}

// Degrees of the stored vertices (and a last word for the scan).
__global__ void k_lay_degrees(uint32_t V, const uint32_t* __restrict__ row_ptr, const uint32_t* __restrict__ ids, uint32_t* deg) {
    for (uint32_t n = blockIdx.x * blockDim.x + threadIdx.x; n <= V; n += gridDim.x * blockDim.x) {
        const uint32_t v = n < V ? ids[n] : 0u;
        deg[n] = n < V && v < V ? row_ptr[v + 1] - row_ptr[v] : 0u;
    }
}

// The stored rows' starts, and how far each row's edges have come from.
__global__ void k_lay_starts(uint32_t V, const uint32_t* __restrict__ row_ptr, const uint32_t* __restrict__ ids,
                             const uint32_t* __restrict__ start, uint32_t* from, uint32_t* row_ptr_out, const WsHeader* hdr) {
    if (hdr->lay_general || hdr->status == SSSP_EINTERNAL) return;  // (EINTERNAL: the vertex sort gave up)
    for (uint32_t n = blockIdx.x * blockDim.x + threadIdx.x; n <= V; n += gridDim.x * blockDim.x) {
        row_ptr_out[n] = start[n];
        if (n < V && ids[n] < V) from[n] = row_ptr[ids[n]] - start[n];
    }
}

// The renumbered rows.  Renumbering keeps every head in its partition, and rows are sorted, so a row's edges
// to one partition (a segment) stay where they are in the row and only change places among themselves.  A
// block takes the segments that start in a tile of LAY_TILE stored edges, holds their new heads in shared
// memory, and every edge counts the smaller heads of its segment: most segments are of a few edges (148
// partitions), so this costs less than two passes of a sort.  Bound by instructions (350 a step of 32 edges,
// 55% of the issue slots).  R-MAT, 4.2 M vertices, 63 M edges, 148 partitions: 1.0 ms where the renumbered
// edge list and its sort took 4.1; the whole layout 10.7 -> 4.87 -> 2.06 ms.  Tiles of 512, 1,024, 2,048 and 4,096
// edges: 2.11, 2.08, 2.12, 2.19; two, four and eight steps of a warp in flight: 2.12, 2.19, 2.37.
// A row with a longer segment (hubs, few partitions) sends the whole graph to the builder, whose launches
// otherwise find an empty list (0.11 ms): 1 M vertices, one partition 3.68 -> 3.74 ms.  So does a share of
// 1/8 of the edges that are LAY_DEEP or more into their segments, where the counts cost more than the builder's
// passes: random graphs of 8,192 vertices, one partition, segments of 1,370 2.78 -> 0.92 ms, four, 342 1.06 -> 0.92;
// of 65,536, one, 299 1.48 and 1.50; of 8,192, eight, 171 (here) 0.78 against 0.92.
__global__ void __launch_bounds__(256) k_lay_rows(uint32_t V, uint32_t E, uint32_t B, const uint32_t* __restrict__ start,
                                                  const uint32_t* __restrict__ from, const uint32_t* __restrict__ col,
                                                  const uint32_t* __restrict__ w, const uint32_t* __restrict__ slots,
                                                  const WsHeader* hdr, uint32_t* col_out, uint32_t* w_out, uint32_t* emap) {
    __shared__ uint32_t head[LAY_CAP], old[LAY_CAP], flags[LAY_CAP / 32], rows[8][32], starts[8][32], total;
    if (hdr->lay_general || hdr->status == SSSP_EINTERNAL) return;  // (EINTERNAL: the vertex sort gave up)
    const uint32_t tid = threadIdx.x, lane = tid & 31u, wid = tid >> 5;
    const uint32_t k0 = blockIdx.x * LAY_TILE, most = min(LAY_CAP, E - k0);
    const uint32_t a = wid * (LAY_TILE / 8u), z = wid == 7u ? most : min(a + LAY_TILE / 8u, most);
    if (tid == 0) total = min(LAY_TILE, most);
    __syncthreads();
    if (a < most) {
        RowWalk walk{start, V, rows[wid], starts[wid]};
        walk.seek(k0 + a);
        uint32_t row = 0, part = 0;  // of the edge before the step
        for (uint32_t at = a; at < z; at += 32u) {
            const uint32_t k = k0 + at + lane, u = walk.step(k0 + at, E);
            const bool on = k < E;
            const uint32_t e = on ? k + __ldg(&from[u]) : 0u, v = on ? __ldg(&col[e]) : 0u, p = v / B;
            uint32_t r = __shfl_up_sync(0xFFFFFFFFu, u, 1), q = __shfl_up_sync(0xFFFFFFFFu, p, 1);
            if (lane == 0) {
                if (at == a) {
                    const bool opens = __ldg(&start[u]) == k;
                    row = opens ? NONE : u;
                    part = opens ? 0u : __ldg(&col[e - 1u]) / B;
                }
                r = row;
                q = part;
            }
            row = __shfl_sync(0xFFFFFFFFu, u, 31);
            part = __shfl_sync(0xFFFFFFFFu, p, 31);
            const uint32_t f = __ballot_sync(0xFFFFFFFFu, on && (r != u || q != p));
            head[at + lane] = on ? __ldg(&slots[v]) : 0u;
            old[at + lane] = e;
            if (lane == 0) flags[at >> 5] = f;
            if (at >= LAY_TILE) {  // the last warp, to the end of the tile's last segment
                if (lane == 0) total = min(at + 32u, most);
                if (f) break;
            }
        }
    }
    __syncthreads();
    const uint32_t n = total;
    for (uint32_t i = tid; i < n; i += 256u) {
        uint32_t wd = i >> 5, m = flags[wd] & (0xFFFFFFFFu >> (31u - (i & 31u)));
        while (!m && wd) m = flags[--wd];
        const uint32_t s = wd * 32u + 31u - (uint32_t)__clz(m);
        if (!m || s >= LAY_TILE) continue;  // another tile's
        wd = i >> 5;
        m = (i & 31u) == 31u ? 0u : flags[wd] & (0xFFFFFFFEu << (i & 31u));
        while (!m && (wd + 1u) * 32u < n) m = flags[++wd];
        const uint32_t end = m ? wd * 32u + (uint32_t)__ffs(m) - 1u : n;
        const uint32_t h = head[i], e = old[i];
        uint32_t c = 0;
        for (uint32_t j = s; j < end; ++j) c += head[j] < h;
        const uint32_t o = k0 + s + c;
        col_out[o] = h;
        w_out[o] = __ldg(&w[e]);
        if (emap) emap[o] = e;
    }
}

__global__ void k_lay_keys(uint32_t V, uint32_t E, unsigned long long B, const uint32_t* __restrict__ deg,
                           uint32_t bits, unsigned long long* keys, uint32_t* vals, WsHeader* hdr) {
    if (blockIdx.x == 0 && threadIdx.x == 0 && hdr->lay_deep > E / 8u) hdr->lay_general = 1u;
    for (uint32_t v = blockIdx.x * blockDim.x + threadIdx.x; v < V; v += gridDim.x * blockDim.x) {
        keys[v] = ((unsigned long long)(v / B) << bits) | ((0xFFFFFFFFu >> (32u - bits)) - deg[v]);
        vals[v] = v;
    }
}

__global__ void k_lay_slots(uint32_t V, const uint32_t* __restrict__ order, uint32_t* ids, uint32_t* slots) {
    for (uint32_t n = blockIdx.x * blockDim.x + threadIdx.x; n < V; n += gridDim.x * blockDim.x) {
        const uint32_t v = order[n];
        ids[n] = v;
        if (v < V) slots[v] = n;  // (always, unless the sort gave up)
    }
}

// The edge list in the new numbering, in the old edge order: a warp walks a range of edges.  (R-MAT
// scale 22: 2.4 ms with a warp per row, half of whose lanes had no edge, -> 0.31 ms, bound by the random
// reads of slots.)

__global__ void __launch_bounds__(256) k_lay_coo(uint32_t V, uint32_t E, const uint32_t* __restrict__ row_ptr,
                                                 const uint32_t* __restrict__ col, const uint32_t* __restrict__ slots,
                                                 const uint32_t* run, uint32_t* src, uint32_t* dst) {
    __shared__ uint32_t rows[8][32], starts[8][32];
    const uint32_t lane = threadIdx.x & 31u, wid = threadIdx.x >> 5;
    const unsigned long long first = ((unsigned long long)blockIdx.x * 8u + wid) * COO_RANGE;
    if (first >= E || (run && !*run)) return;
    const uint32_t e0 = (uint32_t)first, e1 = (uint32_t)min(first + COO_RANGE, (unsigned long long)E);
    RowWalk walk{row_ptr, V, rows[wid], starts[wid]};
    walk.seek(e0);
    uint32_t v = e0 + lane < e1 ? __ldg(&col[e0 + lane]) : 0u;
    for (uint32_t eb = e0; eb < e1 && eb >= e0; eb += 32u) {
        const uint32_t e = eb + lane, u = walk.step(eb, e1), x = v;
        if (e1 - eb > 32u + lane) v = __ldg(&col[e + 32u]);  // the next step's
        if (e < e1) {
            src[e] = __ldg(&slots[u]);
            dst[e] = x < V ? __ldg(&slots[x]) : 0xFFFFFFFFu;  // a bad head stays bad: the CSR builder reports it
        }
    }
}

unsigned grid_for(uint64_t n, unsigned threads = 256) {
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const uint64_t want = (n + threads - 1) / threads;
    return (unsigned)std::max<uint64_t>(1, std::min<uint64_t>(want, (uint64_t)sms * 16));
}

}  // namespace

size_t csr_workspace_bytes(uint32_t V, uint64_t E_raw) { return carve_csr(nullptr, V, E_raw).total; }

#define CK(x)                                        \
    do {                                             \
        if ((x) != cudaSuccess) return SSSP_ECUDA;   \
    } while (0)

sssp_status csr_build(uint32_t V, uint64_t n, const uint32_t* src, const uint32_t* dst, const uint32_t* w, int wtype,
                      uint32_t* row_ptr, uint32_t* col, uint32_t* w_out, uint32_t* eid, uint32_t* E_out, void* ws,
                      size_t ws_bytes, cudaStream_t st, bool clear, const uint32_t* run) {
    CsrWs c = carve_csr(ws, V, n);
    if (ws_bytes < c.total) return SSSP_ENOMEM;
    const uint32_t bits = bits_for(V - 1u);
    if (clear) CK(cudaMemsetAsync(c.hdr, 0, WS_HEADER_BYTES, st));
    CK(cudaMemsetAsync(row_ptr, 0, sizeof(uint32_t) * ((size_t)V + 1), st));
    if (n == 0) {
        CK(cudaMemsetAsync(E_out, 0, sizeof(uint32_t), st));
        return SSSP_OK;
    }
    bool second = false;
    CK(sort_edges(c.sort, V, bits, src, dst, w, wtype, n, c.keys[0], c.keys[1], c.vals[0], c.vals[1], run, c.hdr, st, &second));
    const unsigned long long* keys = c.keys[second];
    const uint32_t* vals = c.vals[second];
    const unsigned long long* count = sort_count(c.sort);
    const unsigned tiles = (unsigned)c.tiles;
    k_csr_runs<<<tiles + 1, EMIT_THREADS, 0, st>>>(count, keys, c.totals, run);  // (the last block counts nothing)
    CK(cudaGetLastError());
    CK(exclusive_scan_u32(c.scan, c.totals, c.totals, c.tiles + 1, st));
    k_csr_emit<<<tiles, EMIT_THREADS, 0, st>>>(V, bits, count, keys, vals, w, c.totals, c.lead, tiles, row_ptr, col, w_out,
                                               eid, E_out, c.hdr, run);
    CK(cudaGetLastError());
    k_csr_cross<<<(tiles + 255) / 256, 256, 0, st>>>(tiles, c.totals, c.lead, w_out, eid, run);
    CK(cudaGetLastError());
    return SSSP_OK;
}

cudaError_t partition_launch(const sssp_graph* g, uint32_t* bounds, uint64_t* inter, cudaStream_t st) {
    const unsigned long long B = ((unsigned long long)g->V + g->partitions - 1) / g->partitions;
    cudaError_t e;
    if (inter && (e = cudaMemsetAsync(inter, 0, sizeof(uint64_t) * g->partitions, st)) != cudaSuccess) return e;
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    // a range per warp: long enough to pay for its search, short enough to give every warp one
    const uint32_t range =
        (uint32_t)std::min<uint64_t>(std::max<uint64_t>((g->E / ((uint64_t)sms * 32) + 127) & ~127ull, 256), 4096);
    const uint64_t warps = inter ? ((uint64_t)g->E + range - 1) / range : 0;
    const unsigned blocks = (unsigned)std::max<uint64_t>(1, (warps * 32 + 255) / 256);
    k_partition<<<blocks, 256, 0, st>>>(g->V, g->E, g->partitions, B, range, g->row_ptr, g->col, bounds,
                                        reinterpret_cast<unsigned long long*>(inter));
    return cudaGetLastError();
}

namespace {
struct LayoutWs {
    size_t off_deg, off_kin, off_kout, off_vin, off_vout, off_tmp, off_src, off_dst, off_eout, total;
    size_t csr_bytes, tmp_bytes;
};

LayoutWs layout_ws(uint32_t V, uint32_t E) {
    LayoutWs w{};
    w.csr_bytes = csr_workspace_bytes(V, E);
    w.tmp_bytes = sort_temp_bytes(V);
    size_t off = align_up(w.csr_bytes, 256);  // the CSR builder's workspace first: its header is the status word
    auto take = [&](size_t bytes) {
        const size_t r = off;
        off += align_up(std::max<size_t>(bytes, 4), 256);
        return r;
    };
    w.off_deg = take(4ull * V);
    w.off_kin = take(8ull * V);
    w.off_kout = take(8ull * V);
    w.off_vin = take(4ull * V);
    w.off_vout = take(4ull * V);
    w.off_tmp = take(w.tmp_bytes);
    w.off_src = take(4ull * E);
    w.off_dst = take(4ull * E);
    w.off_eout = take(4);
    w.total = off;
    return w;
}
}  // namespace

size_t layout_workspace_bytes(uint32_t V, uint32_t E) { return layout_ws(V, E).total; }

sssp_status layout_build(const sssp_graph* g, uint32_t* row_ptr_out, uint32_t* col_out, uint32_t* w_out,
                         uint32_t* emap_out, uint32_t* ids_out, uint32_t* slots_out, void* ws, size_t ws_bytes,
                         cudaStream_t st) {
    const LayoutWs L = layout_ws(g->V, g->E);
    if (ws_bytes < L.total) return SSSP_ENOMEM;
    char* p = static_cast<char*>(ws);
    uint32_t* deg = reinterpret_cast<uint32_t*>(p + L.off_deg);
    unsigned long long* kin = reinterpret_cast<unsigned long long*>(p + L.off_kin);
    unsigned long long* kout = reinterpret_cast<unsigned long long*>(p + L.off_kout);
    uint32_t* vin = reinterpret_cast<uint32_t*>(p + L.off_vin);
    uint32_t* vout = reinterpret_cast<uint32_t*>(p + L.off_vout);
    uint32_t* src = reinterpret_cast<uint32_t*>(p + L.off_src);
    uint32_t* dst = reinterpret_cast<uint32_t*>(p + L.off_dst);
    uint32_t* eout = reinterpret_cast<uint32_t*>(p + L.off_eout);
    const unsigned long long B = ((unsigned long long)g->V + g->partitions - 1) / g->partitions;
    const unsigned gv = grid_for(g->V), gr = (unsigned)((g->E + 8ull * COO_RANGE - 1) / (8ull * COO_RANGE));
    const uint32_t* const w = static_cast<const uint32_t*>(g->w);
    WsHeader* const hdr = reinterpret_cast<WsHeader*>(p);
    const bool segments = g->E != 0u && g->E < 0xF0000000u;
    CK(cudaMemsetAsync(p, 0, WS_HEADER_BYTES, st));
    k_lay_deg<<<gv, 256, 0, st>>>(g->V, g->row_ptr, deg);
    CK(cudaGetLastError());
    if (g->E) {
        k_lay_check<<<gr, 256, 0, st>>>(g->V, g->E, (uint32_t)B, g->row_ptr, g->col, w, g->wtype, deg, hdr);
        CK(cudaGetLastError());
    }
    const uint32_t bits = std::min(std::max(bits_for(g->E) + 1u, 1u), 32u);  // of a degree (in + out: at most 2 E)
    k_lay_keys<<<gv, 256, 0, st>>>(g->V, g->E, B, deg, bits, kin, vin, hdr);
    CK(cudaGetLastError());
    bool second = false;
    CK(sort_pairs_u64(p + L.off_tmp, kin, kout, vin, vout, g->V, (int)(bits + bits_for(g->partitions - 1u)), hdr, st, &second));
    k_lay_slots<<<gv, 256, 0, st>>>(g->V, second ? vout : vin, ids_out, slots_out);
    CK(cudaGetLastError());
    const uint32_t* const run = segments ? &hdr->lay_general : nullptr;
    if (g->E) {
        k_lay_coo<<<gr, 256, 0, st>>>(g->V, g->E, g->row_ptr, g->col, slots_out, run, src, dst);
        CK(cudaGetLastError());
    }
    // the renumbered edge list through the CSR builder: rows sorted by new head id, and
    // its input-index output maps each stored edge back to its index in g
    const sssp_status built = csr_build(g->V, g->E, src, dst, w, g->wtype, row_ptr_out, col_out, w_out, emap_out, eout, ws,
                                        L.csr_bytes, st, false, run);  // (the status of the vertex sort stays)
    if (built != SSSP_OK || !segments) return built;
    uint32_t* const start = reinterpret_cast<uint32_t*>(kin);
    uint32_t* const from = reinterpret_cast<uint32_t*>(kout);
    k_lay_degrees<<<gv, 256, 0, st>>>(g->V, g->row_ptr, ids_out, start);
    CK(cudaGetLastError());
    CK(exclusive_scan_u32(deg, start, start, (uint64_t)g->V + 1, st));
    k_lay_starts<<<gv, 256, 0, st>>>(g->V, g->row_ptr, ids_out, start, from, row_ptr_out, hdr);
    CK(cudaGetLastError());
    k_lay_rows<<<(g->E + LAY_TILE - 1u) / LAY_TILE, 256, 0, st>>>(g->V, g->E, (uint32_t)B, start, from, g->col, w, slots_out, hdr,
                                                                  col_out, w_out, emap_out);
    CK(cudaGetLastError());
    return SSSP_OK;
}

namespace {
struct CompactWs {
    size_t off_mask, off_before, off_totals, off_tmp, total;
    uint64_t words, tiles;
};

CompactWs compact_ws(uint32_t E) {
    CompactWs c{};
    c.words = E / 32u + 1u;
    c.tiles = (c.words + KEEP_WORDS - 1) / KEEP_WORDS;
    c.off_mask = WS_HEADER_BYTES;
    c.off_before = c.off_mask + align_up(4 * c.words, 256);
    c.off_totals = c.off_before + align_up(4 * c.words, 256);
    c.off_tmp = c.off_totals + align_up(4 * c.tiles, 256);
    c.total = c.off_tmp + align_up(scan_temp_bytes(c.tiles), 256);
    return c;
}
}  // namespace

size_t compact_workspace_bytes(uint32_t V, uint32_t E) {
    (void)V;
    return compact_ws(E).total;
}

sssp_status compact_launch(const sssp_graph* g, const uint8_t* keep, uint32_t* row_ptr_out, uint32_t* col_out,
                           uint32_t* w_out, uint32_t* emap_out, uint32_t* E_out, void* ws, size_t ws_bytes,
                           cudaStream_t st) {
    const CompactWs c = compact_ws(g->E);
    if (ws_bytes < c.total) return SSSP_ENOMEM;
    char* p = static_cast<char*>(ws);
    uint32_t* mask = reinterpret_cast<uint32_t*>(p + c.off_mask);
    uint32_t* before = reinterpret_cast<uint32_t*>(p + c.off_before);
    uint32_t* totals = reinterpret_cast<uint32_t*>(p + c.off_totals);
    CK(cudaMemsetAsync(p, 0, WS_HEADER_BYTES, st));
    if ((reinterpret_cast<uintptr_t>(keep) & 15u) == 0)
        k_keep_bits<true><<<(unsigned)c.tiles, KEEP_THREADS, 0, st>>>(g->E, keep, mask, before, totals);
    else
        k_keep_bits<false><<<(unsigned)c.tiles, KEEP_THREADS, 0, st>>>(g->E, keep, mask, before, totals);
    CK(cudaGetLastError());
    CK(exclusive_scan_u32(p + c.off_tmp, totals, totals, c.tiles, st));
    // a warp per 32 words of the mask (1,024 edges)
    const unsigned gr = grid_for(std::max<uint64_t>(c.words, (uint64_t)g->V + 1));
    k_compact<<<gr, 256, 0, st>>>(g->V, g->E, g->row_ptr, g->col, static_cast<const uint32_t*>(g->w), mask, before, totals,
                                  row_ptr_out, col_out, w_out, emap_out, E_out);
    CK(cudaGetLastError());
    return SSSP_OK;
}

}  // namespace sssp
