// Device-wide primitives of the one-time graph steps (CSR build, locality layout, compaction):
// a stable radix sort of (64-bit key, 32-bit value) pairs and a prefix sum of 32-bit counts.
//
// Sort: least-significant digit first, digits of up to 9 bits, one pass over the pairs per digit (the
// single-pass scheme of Adinets and Merrill's "Onesweep", with the decoupled look-back of Merrill and
// Garland).  The histograms of all digits are taken first, in one read of the keys (or of the edge
// list the keys are made from).  A pass then cuts the pairs into tiles of TILE, taken in ticket order:
//   1. a warp holds a run of 512 pairs in registers and ranks equal digits within 32 lanes (a ballot
//      per bit) over a running count per digit, so pairs keep their order (stable, which LSD needs);
//      the warps' counts make the tile's, which it publishes;
//   2. the tile is ordered by digit in shared memory;
//   3. each thread looks back over the published counts of the tiles before it for its two digits
//      until it meets a running total, which gives the tile's output positions with no pass over
//      counts.  A wait is bounded: after SPIN_MAX looks the tile gives up, reports SSSP_EINTERNAL and
//      writes nothing;
//   4. the tile goes out run by run, consecutive threads storing consecutive pairs of one digit.
// 9 bits against 8 saves a pass on the 44-bit keys of 4 M vertices (5 instead of 6) at runs of 8
// pairs a tile.  R-MAT scale 22 (67 M pairs): 6.2 ms as count, scan and place kernels of 8 bits ->
// 3.3 ms, 0.6 ms a pass (24 bytes a pair read and written, 2.7 TB/s).  A pass is bound by the latency
// of its phases at 24 warps per SM: of 40,000 cycles a tile, 9,000 load, 8,000 rank, 5,000 order,
// 9,000 look back, 4,000 store.  Measured and slower: __match_any_sync (0.61 ms), 512 threads of 8
// pairs (0.65 to 0.73), 12 or 20 pairs a thread (0.67, 0.68), counts published before the ranks
// (0.65), the look-back before the ranks (0.68), 8 descriptors at a time (0.67).
// Scan: tiles of SCAN_TILE values staged in shared memory; a first kernel sums each tile, the
// tile sums are scanned (recursively while there are more than one tile of them), and a second
// kernel scans each tile from its offset.
#include <algorithm>
#include <type_traits>

#include "common.cuh"
#include "internal.h"

namespace sssp {
namespace {

constexpr uint32_t THREADS = 256, WARPS = THREADS / 32;
constexpr uint32_t ITEMS = 16;                  // pairs a thread holds
constexpr uint32_t WARP_RUN = 32 * ITEMS;       // consecutive pairs a warp takes
constexpr uint32_t TILE = THREADS * ITEMS;      // pairs a block takes
constexpr uint32_t RADIX = 512;                 // largest count of digit values: one a thread
constexpr uint32_t DPT = RADIX / THREADS;       // digits a thread looks after: tid, tid + THREADS, ...
constexpr uint32_t PASSES = 8;                  // most passes (64-bit keys)
constexpr uint32_t LOOK = 4;                    // descriptors looked at together
constexpr uint32_t SPIN_MAX = 1u << 22;         // looks at one descriptor (seconds)

constexpr uint32_t SCAN_THREADS = 256;
constexpr uint32_t SCAN_ITEMS = 16;
constexpr uint32_t SCAN_TILE = SCAN_THREADS * SCAN_ITEMS;

struct Digits {  // pass p sorts by bits [shift[p], shift[p] + bits[p])
    uint32_t passes;
    uint8_t shift[PASSES], bits[PASSES];
};

Digits digits_for(uint32_t end_bit) {
    Digits d{};
    d.passes = (end_bit + 8u) / 9u;
    for (uint32_t p = 0, at = 0; p < d.passes; ++p) {
        d.shift[p] = (uint8_t)at;
        d.bits[p] = (uint8_t)((end_bit - at + d.passes - p - 1u) / (d.passes - p));
        at += d.bits[p];
    }
    return d;
}

// Temporaries of a sort: cleared before it up to the descriptors of the passes it makes.
struct SortTmp {
    unsigned long long count;               // pairs
    uint32_t ticket[PASSES];                // next tile of each pass
    uint32_t hist[PASSES][RADIX];           // digit counts, then first output positions
};
// descriptor of (tile, digit): a state in the top two bits, pairs below (32 bits while there are fewer
// than 2^30 pairs); 1: the tile's own count, 2: with all tiles before it
template <class D>
constexpr D DESC_OWN = D(1) << (8 * sizeof(D) - 2);
template <class D>
constexpr D DESC_ALL = D(2) << (8 * sizeof(D) - 2);
template <class D>
constexpr D DESC_VALUE = DESC_OWN<D> - 1;

__device__ __forceinline__ void st_desc(uint32_t* p, uint32_t v) { st_relaxed(p, v); }
__device__ __forceinline__ void st_desc(unsigned long long* p, unsigned long long v) {
    asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}

// Where the pairs come from: an array of keys and values, or an edge list, whose keys are
// (tail << bits) | head and whose values are the edges' indices; loops and bad edges make no pair.
struct Source {
    const unsigned long long* keys;
    const uint32_t* vals;
    const uint32_t* src;
    const uint32_t* dst;
    uint32_t V, bits;
    const uint32_t* run;  // edges: not NULL and zero: there are none
};

__device__ __forceinline__ bool edge_key(const Source& s, uint32_t a, uint32_t b, unsigned long long& k) {
    k = (unsigned long long)a << s.bits | b;
    return a < s.V && b < s.V && a != b;
}

// block-wide exclusive scan of one value per thread; returns the block total in *total
__device__ __forceinline__ uint32_t block_excl(uint32_t x, uint32_t* wsum, uint32_t* total) {
    const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    uint32_t inc = x;
#pragma unroll
    for (uint32_t o = 1; o < 32u; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, inc, o);
        if (lane >= o) inc += y;
    }
    if (lane == 31u) wsum[warp] = inc;
    __syncthreads();
    if (warp == 0) {
        uint32_t t = lane < nw ? wsum[lane] : 0u;
#pragma unroll
        for (uint32_t o = 1; o < 32u; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, t, o);
            if (lane >= o) t += y;
        }
        if (lane < nw) wsum[lane] = t;
    }
    __syncthreads();
    const uint32_t r = (warp ? wsum[warp - 1] : 0u) + inc - x;
    *total = wsum[nw - 1];
    __syncthreads();
    return r;
}

// Digit counts of every pass and the count of pairs.  W: the edges' weights are checked on the way
// (void: no edges).  A block keeps the counts in shared memory over all it reads.
template <class W>
__global__ void __launch_bounds__(512) k_sort_hist(Source s, unsigned long long n, const uint32_t* __restrict__ w, Digits dg,
                                                   SortTmp* tmp, WsHeader* hdr) {
    constexpr bool EDGES = !std::is_void<W>::value;
    __shared__ uint32_t h[PASSES][RADIX];
    __shared__ uint32_t cnt;
    if (EDGES && s.run && !*s.run) return;
    for (uint32_t i = threadIdx.x; i < dg.passes * RADIX; i += blockDim.x) (&h[0][0])[i] = 0u;
    if (threadIdx.x == 0) cnt = 0u;
    __syncthreads();
    bool bad = false;
    uint32_t mine = 0;
    constexpr uint32_t FLY = 4;  // pairs a thread loads together
    const unsigned long long step = (unsigned long long)gridDim.x * blockDim.x * FLY;
    for (unsigned long long i0 = (unsigned long long)blockIdx.x * blockDim.x * FLY + threadIdx.x; i0 < n; i0 += step) {
        unsigned long long k[FLY];
        uint32_t a[FLY], b[FLY], x[FLY];
#pragma unroll
        for (uint32_t f = 0; f < FLY; ++f) {
            const unsigned long long i = i0 + f * blockDim.x;
            if (i >= n) continue;
            if constexpr (EDGES)
                a[f] = __ldg(&s.src[i]), b[f] = __ldg(&s.dst[i]), x[f] = __ldg(&w[i]);
            else
                k[f] = s.keys[i];
        }
#pragma unroll
        for (uint32_t f = 0; f < FLY; ++f) {
            if (i0 + f * blockDim.x >= n) continue;
            if constexpr (EDGES) {
                bad |= a[f] >= s.V || b[f] >= s.V || !W::weight_ok(x[f]);
                if (!edge_key(s, a[f], b[f], k[f])) continue;
            }
            ++mine;
#pragma unroll
            for (uint32_t p = 0; p < PASSES; ++p)
                if (p < dg.passes)
                    atomicAdd(&h[p][(uint32_t)(k[f] >> dg.shift[p]) & ((1u << dg.bits[p]) - 1u)], 1u);
        }
    }
    if (bad) set_status(hdr, SSSP_EINVAL);
    mine = __reduce_add_sync(0xFFFFFFFFu, mine);
    if ((threadIdx.x & 31u) == 0 && mine) atomicAdd(&cnt, mine);
    __syncthreads();
    for (uint32_t i = threadIdx.x; i < dg.passes * RADIX; i += blockDim.x)
        if ((&h[0][0])[i]) atomicAdd(&(&tmp->hist[0][0])[i], (&h[0][0])[i]);
    if (threadIdx.x == 0 && cnt) atomicAdd(&tmp->count, (unsigned long long)cnt);
}

// counts -> first output position of each digit (a block per pass)
__global__ void __launch_bounds__(RADIX) k_sort_bases(SortTmp* tmp) {
    __shared__ uint32_t wsum[32];
    uint32_t total;
    const uint32_t x = tmp->hist[blockIdx.x][threadIdx.x];
    tmp->hist[blockIdx.x][threadIdx.x] = block_excl(x, wsum, &total);
}

// Shared memory of a pass (dynamic: more than 48 KB).
struct PassMem {
    unsigned long long key[TILE];
    uint32_t val[TILE];
    uint16_t count[WARPS][RADIX];  // per warp: digit counts, then those of the warps before it
    uint32_t out[RADIX];           // output position of the tile's pairs of a digit, less their place in the tile
    uint32_t wsum[32];
    uint32_t tile;
    int fail;
};

template <bool EDGES, class D>
__global__ void __launch_bounds__(THREADS, 3) k_sort_pass(Source s, unsigned long long n_in, uint32_t shift, uint32_t bits,
                                                          uint32_t pass, SortTmp* tmp,
                                                          D* desc, unsigned long long* __restrict__ kout,
                                                          uint32_t* __restrict__ vout, WsHeader* hdr) {
    extern __shared__ __align__(16) unsigned char raw[];
    PassMem& m = *reinterpret_cast<PassMem*>(raw);
    const uint32_t tid = threadIdx.x, lane = tid & 31u, warp = tid >> 5, nd = 1u << bits;
    const unsigned long long count = tmp->count, n = EDGES ? (s.run && !*s.run ? 0ull : n_in) : count;
    if (n == 0) return;
    if (tid == 0) {
        m.tile = atomicAdd(&tmp->ticket[pass], 1u);
        m.fail = 0;
    }
    for (uint32_t i = tid; i < WARPS * RADIX / 2; i += THREADS) reinterpret_cast<uint32_t*>(&m.count[0][0])[i] = 0u;
    __syncthreads();
    const uint32_t tile = m.tile;
    const unsigned long long base = (unsigned long long)tile * TILE + warp * WARP_RUN + lane;
    if ((unsigned long long)tile * TILE >= n) return;
    unsigned long long k[ITEMS];
    uint32_t v[ITEMS], r[ITEMS];
#pragma unroll
    for (uint32_t j = 0; j < ITEMS; ++j) {
        const unsigned long long i = base + 32u * j;
        if (i >= n) continue;
        if constexpr (EDGES)
            v[j] = __ldg(&s.src[i]), r[j] = __ldg(&s.dst[i]);
        else
            k[j] = s.keys[i], v[j] = s.vals[i];
    }
#pragma unroll
    for (uint32_t j = 0; j < ITEMS; ++j) {
        bool ok = base + 32u * j < n;
        if constexpr (EDGES) {
            ok = ok && edge_key(s, v[j], r[j], k[j]);
            v[j] = (uint32_t)(base + 32u * j);
        }
        r[j] = ok ? (uint32_t)(k[j] >> shift) & (nd - 1u) : RADIX;  // RADIX: no pair
    }
    D* const mine = desc + (size_t)tile * RADIX + tid;
    uint32_t tot[DPT], start[DPT], all = 0;
    D before[DPT] = {};
    // what the tiles before it hold: look back, LOOK tiles at a time
    auto look_back = [&]() {
#pragma unroll
        for (uint32_t x = 0; x < DPT; ++x) {
            bool done = tile == 0u;
            uint32_t t = tile, spin = 0;  // tiles still to look at
            while (!done) {
                D a[LOOK];
#pragma unroll
                for (uint32_t l = 0; l < LOOK; ++l)
                    a[l] = l < t ? ld_relaxed(&desc[(size_t)(t - 1u - l) * RADIX + tid + x * THREADS]) : D(0);
                const uint32_t t0 = t;
#pragma unroll
                for (uint32_t l = 0; l < LOOK; ++l) {
                    if (done || t != t0 - l || !(a[l] >> (8 * sizeof(D) - 2))) continue;
                    before[x] += a[l] & DESC_VALUE<D>;
                    done = (a[l] & DESC_ALL<D>) != 0;
                    --t;
                }
                if (t == t0 && ++spin >= SPIN_MAX) {
                    m.fail = 1;
                    break;
                }
            }
            if (tile) st_desc(mine + x * THREADS, DESC_ALL<D> | (before[x] + tot[x]));
        }
    };
    // 1. ranks: r = digit | rank in the warp's run << 16
#pragma unroll
    for (uint32_t j = 0; j < ITEMS; ++j) {
        const uint32_t d = r[j];
        uint32_t peers = __ballot_sync(0xFFFFFFFFu, d != RADIX);
        if (d == RADIX) peers = 0u;
#pragma unroll
        for (uint32_t b = 0; b < 9u; ++b) {
            const bool one = d >> b & 1u;
            const uint32_t v1 = __ballot_sync(0xFFFFFFFFu, one);
            peers &= one ? v1 : ~v1;
        }
        if (d != RADIX) r[j] = d | (m.count[warp][d] + __popc(peers & ((1u << lane) - 1u))) << 16;
        __syncwarp();
        if (peers && lane == 31u - (uint32_t)__clz(peers)) m.count[warp][d] = (uint16_t)((r[j] >> 16) + 1u);
        __syncwarp();
    }
    __syncthreads();
    // the tile's count of each digit, published (the tiles after it look for it), and its place in the tile
#pragma unroll
    for (uint32_t x = 0; x < DPT; ++x) {
        uint32_t sum = 0;
#pragma unroll
        for (uint32_t i = 0; i < WARPS; ++i) sum += m.count[i][tid + x * THREADS];
        tot[x] = sum;
        st_desc(mine + x * THREADS, (tile ? DESC_OWN<D> : DESC_ALL<D>) | tot[x]);
    }
#pragma unroll
    for (uint32_t x = 0; x < DPT; ++x) {
        uint32_t t;
        start[x] = all + block_excl(tot[x], m.wsum, &t);
        all += t;
        uint32_t sum = start[x];  // (places in the tile fit 16 bits)
#pragma unroll
        for (uint32_t i = 0; i < WARPS; ++i) {
            const uint32_t c = m.count[i][tid + x * THREADS];
            m.count[i][tid + x * THREADS] = (uint16_t)sum;
            sum += c;
        }
    }
    __syncthreads();
    // 2. the tile in digit order
#pragma unroll
    for (uint32_t j = 0; j < ITEMS; ++j) {
        if (r[j] == RADIX) continue;
        const uint32_t at = m.count[warp][r[j] & (RADIX - 1u)] + (r[j] >> 16);
        m.key[at] = k[j];
        m.val[at] = v[j];
    }
    look_back();
#pragma unroll
    for (uint32_t x = 0; x < DPT; ++x) m.out[tid + x * THREADS] = tmp->hist[pass][tid + x * THREADS] + (uint32_t)before[x] - start[x];
    __syncthreads();
    if (m.fail) {
        if (tid == 0) set_status(hdr, SSSP_EINTERNAL);
        return;
    }
    for (uint32_t i = tid; i < all; i += THREADS) {
        const unsigned long long key = m.key[i];
        const unsigned long long pos = m.out[(uint32_t)(key >> shift) & (nd - 1u)] + i;
        if (pos < count) {  // (always, unless an earlier pass gave up)
            kout[(uint32_t)pos] = key;
            vout[(uint32_t)pos] = m.val[i];
        }
    }
}

// --- scan

// sum of each tile
__global__ void __launch_bounds__(SCAN_THREADS) k_scan_sums(const uint32_t* __restrict__ in, unsigned long long n,
                                                            uint32_t* sums) {
    __shared__ uint32_t wsum[32];
    const unsigned long long base = (unsigned long long)blockIdx.x * SCAN_TILE;
    uint32_t s = 0;
    for (uint32_t i = threadIdx.x; i < SCAN_TILE; i += SCAN_THREADS) {
        const unsigned long long at = base + i;
        if (at < n) s += in[at];
    }
    uint32_t total;
    block_excl(s, wsum, &total);
    if (threadIdx.x == 0) sums[blockIdx.x] = total;
}

// exclusive scan of each tile from its offset (offsets NULL: 0)
__global__ void __launch_bounds__(SCAN_THREADS) k_scan_tiles(const uint32_t* __restrict__ in, unsigned long long n,
                                                             const uint32_t* __restrict__ offsets, uint32_t* out) {
    __shared__ uint32_t tilev[SCAN_TILE];
    __shared__ uint32_t wsum[32];
    const unsigned long long base = (unsigned long long)blockIdx.x * SCAN_TILE;
    for (uint32_t i = threadIdx.x; i < SCAN_TILE; i += SCAN_THREADS) {
        const unsigned long long at = base + i;
        tilev[i] = at < n ? in[at] : 0u;
    }
    __syncthreads();
    uint32_t vals[SCAN_ITEMS], s = 0;
#pragma unroll
    for (uint32_t j = 0; j < SCAN_ITEMS; ++j) {
        vals[j] = tilev[threadIdx.x * SCAN_ITEMS + j];
        s += vals[j];
    }
    uint32_t total;
    uint32_t run = block_excl(s, wsum, &total) + (offsets ? offsets[blockIdx.x] : 0u);
#pragma unroll
    for (uint32_t j = 0; j < SCAN_ITEMS; ++j) {
        tilev[threadIdx.x * SCAN_ITEMS + j] = run;
        run += vals[j];
    }
    __syncthreads();
    for (uint32_t i = threadIdx.x; i < SCAN_TILE; i += SCAN_THREADS) {
        const unsigned long long at = base + i;
        if (at < n) out[at] = tilev[i];
    }
}

uint64_t tiles_of(uint64_t n, uint64_t tile) { return (n + tile - 1) / tile; }

// temp words the scan of n values needs: the tile sums of every level
size_t scan_temp_words(uint64_t n) {
    size_t w = 0;
    for (uint64_t m = tiles_of(n, SCAN_TILE); m > 1; m = tiles_of(m, SCAN_TILE)) w += align_up(m, 64);
    return w + 64;
}

cudaError_t scan_u32(uint32_t* tmp, const uint32_t* in, uint32_t* out, uint64_t n, cudaStream_t st) {
    if (n == 0) return cudaSuccess;
    const uint64_t nt = tiles_of(n, SCAN_TILE);
    if (nt == 1) {
        k_scan_tiles<<<1, SCAN_THREADS, 0, st>>>(in, n, nullptr, out);
        return cudaGetLastError();
    }
    uint32_t* sums = tmp;
    uint32_t* rest = tmp + align_up(nt, 64);
    k_scan_sums<<<(unsigned)nt, SCAN_THREADS, 0, st>>>(in, n, sums);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    if ((e = scan_u32(rest, sums, sums, nt, st)) != cudaSuccess) return e;  // tile offsets, in place
    k_scan_tiles<<<(unsigned)nt, SCAN_THREADS, 0, st>>>(in, n, sums, out);
    return cudaGetLastError();
}

uint64_t sort_tiles(uint64_t n) { return std::max<uint64_t>(tiles_of(n, TILE), 1); }

template <bool EDGES, class D>
cudaError_t run_passes(const Source& first, uint64_t n, const Digits& dg, SortTmp* tmp, unsigned long long* k0,
                       unsigned long long* k1, uint32_t* v0, uint32_t* v1, WsHeader* hdr, cudaStream_t st) {
    cudaError_t e;
    const uint64_t tiles = sort_tiles(n);
    D* const desc = reinterpret_cast<D*>(reinterpret_cast<char*>(tmp) + align_up(sizeof(SortTmp), 256));
    for (const void* k : {(const void*)k_sort_pass<EDGES, D>, (const void*)k_sort_pass<false, D>})
        if ((e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(PassMem))) != cudaSuccess)
            return e;
    k_sort_bases<<<dg.passes, RADIX, 0, st>>>(tmp);
    Source s = first;
    for (uint32_t p = 0; p < dg.passes; ++p) {
        (p ? k_sort_pass<false, D> : k_sort_pass<EDGES, D>)<<<(unsigned)tiles, THREADS, sizeof(PassMem), st>>>(
            s, n, dg.shift[p], dg.bits[p], p, tmp, desc + (size_t)p * tiles * RADIX, k0, v0, hdr);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
        s = Source{k0, v0, nullptr, nullptr, 0u, 0u, nullptr};
        std::swap(k0, k1);
        std::swap(v0, v1);
    }
    return cudaSuccess;
}

bool narrow(uint64_t n) { return n < (1ull << 30); }

cudaError_t clear_sort(void* tmp, const Digits& dg, uint64_t n, cudaStream_t st) {
    return cudaMemsetAsync(tmp, 0, align_up(sizeof(SortTmp), 256) + (narrow(n) ? 4ull : 8ull) * dg.passes * sort_tiles(n) * RADIX,
                           st);
}

unsigned hist_grid(uint64_t n) {
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    return (unsigned)std::max<uint64_t>(1, std::min<uint64_t>((n + 2047) / 2048, (uint64_t)sms * 4));
}

}  // namespace

size_t sort_temp_bytes(uint64_t n) { return align_up(sizeof(SortTmp), 256) + 8ull * PASSES * sort_tiles(n) * RADIX; }

size_t scan_temp_bytes(uint64_t n) { return 4 * scan_temp_words(n); }

cudaError_t exclusive_scan_u32(void* tmp, const uint32_t* in, uint32_t* out, uint64_t n, cudaStream_t st) {
    return scan_u32(static_cast<uint32_t*>(tmp), in, out, n, st);
}

const unsigned long long* sort_count(const void* tmp) { return &static_cast<const SortTmp*>(tmp)->count; }

cudaError_t sort_pairs_u64(void* tmp, unsigned long long* k0, unsigned long long* k1, uint32_t* v0, uint32_t* v1,
                           uint64_t n, int end_bit, WsHeader* hdr, cudaStream_t st, bool* in_second) {
    *in_second = false;
    if (n <= 1 || end_bit <= 0) return cudaSuccess;
    const Digits dg = digits_for((uint32_t)end_bit);
    cudaError_t e;
    if ((e = clear_sort(tmp, dg, n, st)) != cudaSuccess) return e;
    SortTmp* t = static_cast<SortTmp*>(tmp);
    const Source s{k0, v0, nullptr, nullptr, 0u, 0u, nullptr};
    k_sort_hist<void><<<hist_grid(n), 512, 0, st>>>(s, n, nullptr, dg, t, hdr);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    *in_second = dg.passes & 1u;
    return narrow(n) ? run_passes<false, uint32_t>(s, n, dg, t, k1, k0, v1, v0, hdr, st)
                     : run_passes<false, unsigned long long>(s, n, dg, t, k1, k0, v1, v0, hdr, st);
}

cudaError_t sort_edges(void* tmp, uint32_t V, uint32_t bits, const uint32_t* src, const uint32_t* dst, const uint32_t* w,
                       int wtype, uint64_t n, unsigned long long* k0, unsigned long long* k1, uint32_t* v0, uint32_t* v1,
                       const uint32_t* run, WsHeader* hdr, cudaStream_t st, bool* in_second) {
    const Digits dg = digits_for(std::max<uint32_t>(2u * bits, 1u));
    cudaError_t e;
    if ((e = clear_sort(tmp, dg, n, st)) != cudaSuccess) return e;
    SortTmp* t = static_cast<SortTmp*>(tmp);
    const Source s{nullptr, nullptr, src, dst, V, bits, run};
    if (wtype == SSSP_W_F32)
        k_sort_hist<WF32><<<hist_grid(n), 512, 0, st>>>(s, n, w, dg, t, hdr);
    else
        k_sort_hist<WU32><<<hist_grid(n), 512, 0, st>>>(s, n, w, dg, t, hdr);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    *in_second = !(dg.passes & 1u);  // the first pass writes k0
    return narrow(n) ? run_passes<true, uint32_t>(s, n, dg, t, k0, k1, v0, v1, hdr, st)
                     : run_passes<true, unsigned long long>(s, n, dg, t, k0, k1, v0, v1, hdr, st);
}

}  // namespace sssp
