// K4s sweep: all sources of a solve relax the graph together, Bellman-Ford from a frontier.
//
// On graphs of small diameter and several edges per vertex (random and power-law graphs) the
// persistent solve of relax.cu is bound by its chains of dependent rounds when the graph is small,
// and by random 32-byte sectors, one per edge and source, when it is large.  Here the distances of
// up to eight sources of a vertex share one sector (dist[item][G], item = group * V + vertex), so a
// visit of an edge reads its (col, w) once and one sector for all sources of the group.  The
// visits can be shared because the sources' wavefronts cross such a graph in the same few hops: a
// vertex whose distance fell for some sources is relaxed for all of its group at once (the lanes of
// the others cost nothing more).
//
// One cooperative launch, bulk synchronous: an iteration takes every marked item, relaxes its row
// and marks the items whose distances fall, which are the next iteration's; about 20 iterations in
// all.  There is no bucket order: thresholds above the least queued distance of each source cut the
// relaxations of random graphs to a third, but took more iterations and a second look at every item,
// and on power-law graphs cut nothing (in an earlier form of this kernel, R-MAT scale 22, 8 sources: 4.7 against 4.2
// ms; random graph of 16,384 vertices: 0.36 against 0.24 ms).
//   list A : rows of up to 31 edges; a warp takes 32 of them (fewer when the list is short) and
//            walks their edges together
//   list M : rows of 32 to 511 edges, up to 8 a warp in the same way
//   hubs   : rows of SWEEP_HUB edges or more, cut into segments that all warps share
//   lowered items go to a buffer of the warp and are marked 128 at a time: the chain of a fence, a
//            mark and a degree would otherwise be paid by every step
// Predecessors come from one pass over the edges at the end (k_sweep_out): pred(v) is the least
// label of a tail u with dist(u) + w = dist(v), to which the packed words of the persistent solve
// converge too.  The loop then needs 4 bytes per vertex and source instead of 8.
// Measured against the persistent solve (launches; a call has about 0.1 ms besides): R-MAT scale 22, edge factor
// 16, 8 sources, locality layout 3.3 against 7.1 ms (tuned; whole calls on another graph and sources of this
// recipe 4.1 against 7.4); DRAM traffic 6.2 against 13.1 GB; R-MAT scale 18, 32 float32 sources 0.58 against 1.0 ms
// (tuned); random graph, 16,384 vertices, 4 partitions, 1 source 0.23 against 1.6 ms (default width).
// k_sweep (2.4 ms of the 3.3) is bound by the latency of its L2 accesses, issue slots and barriers (scale 20, ncu: 47%
// of the slots busy at the 32 warps per SM that 64 registers allow, stalls 5.8 cycles an instruction on loads and 4.4
// at barriers; with 48 warps at 40 registers it spills and is not faster), k_sweep_out (0.81 ms) by random 32-byte
// sectors, 80 G a second.
// A warm start (sssp_update) with many tails goes the same way, from the tails' rows: there the rows are of
// packed words (up to four), so that predecessors come along and no pass over all edges is needed, and
// the lists and marks take the caller's dist.  R-MAT, 1 M vertices, 15 M edges, 4 sources, 15,000 tails: 0.39 ->
// 0.27 ms; k_sweep has 0.19 of it, most in the first iteration (the tails' rows are a third of the edges).
// A graph of many hops is left to k_solve after a few iterations (api.cu says when), and so is a long tail: marks become
// inbox bits, distances packed words, and k_solve goes on from them.
// Waits: the grid barrier is bounded by the idle limit, the kernel by LIMIT_FACTOR times it.
#include <algorithm>
#include <type_traits>

#include "common.cuh"
#include "internal.h"
#include "rowwalk.cuh"

namespace sssp {
namespace {

constexpr uint32_t WT = 512, NW = WT / 32;  // threads and warps per block
constexpr uint32_t SMALL_ROW = 32;          // rows below it: list A
constexpr uint32_t SEG = 128;               // edges of a hub segment
constexpr uint32_t BUF = 64;                // a warp's buffer of newly marked items, per list
constexpr uint32_t MQ = 4, MARKS = MQ * 32;  // items a lane, a warp marks at a time
constexpr uint32_t OUT_EDGES = 1024;        // most edges a warp of k_sweep_out takes
constexpr uint64_t LIMIT_FACTOR = 3;
constexpr uint32_t WARM_ITERS = 32;  // a warm start is handed over
// When a sweep stops.  At HOPS_ITERS: a graph of many hops (SweepLaunch::few), unless it is kept.  Every HAND_EVERY
// iterations: a kept one at a pace that predicts more than HAND_ITERS iterations at the first look (a band of
// 30,000 vertices, 7 a hop: 840 to 1,670; a lattice of 64^3: 170 to 290; a ring with short cuts: 320), later four times as
// many; else a tail, fewer than HAND_EDGES relaxations an iteration.
constexpr uint32_t HOPS_ITERS = 5, HAND_EVERY = 32, HAND_EDGES = 256, HAND_ITERS = 512;

template <class W>
struct Dist;
template <>
struct Dist<WU32> {
    static constexpr uint32_t INF = INF32;
    __device__ __forceinline__ static uint32_t add(uint32_t d, uint32_t w) { return min(d, ~w) + w; }  // saturates
};
template <>
struct Dist<WF32> {
    static constexpr uint32_t INF = F32_INF_BITS;
    __device__ __forceinline__ static uint32_t add(uint32_t d, uint32_t w) {
        return __float_as_uint(__fadd_rn(__uint_as_float(d), __uint_as_float(w)));  // +inf stays
    }
};

struct WarpMem {                              // shared memory of a warp, besides the distances it holds
    uint4 row[32];                            // rows held: first edge - edges before it, group base, largest distance
    uint32_t bufA[BUF], bufM[BUF];
    uint32_t low[MARKS];                      // items whose distances were lowered, to be marked
    unsigned long long edges;                 // statistics of the launch
    uint32_t act, vert;
};

struct BlockMem {
    uint32_t c[8];
    uint32_t wA[NW], wM[NW];
    unsigned long long work, at, imp;
    uint32_t next;  // the block's next unit of work
    int ok;
    // the iterations made, their relaxations, those at the last look, many hops and kept all the same; what is next
    uint32_t iters, slow, then;
    unsigned long long total, looked;
};
constexpr uint32_t GO_ON = ~0u, ASK = ~1u;  // BlockMem::then, or how the sweep ends (SWEPT_*)

__device__ __forceinline__ uint32_t ld_acquire(const uint32_t* p) {
    uint32_t v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

__device__ __forceinline__ void fence_gpu() { asm volatile("fence.acq_rel.gpu;" ::: "memory"); }

__device__ __forceinline__ void and_acquire(uint32_t* p, uint32_t v) {
    uint32_t old;
    asm volatile("atom.acquire.gpu.global.and.b32 %0, [%1], %2;" : "=r"(old) : "l"(p), "r"(v) : "memory");
}

// The G distances of an item from L2 (rows are aligned to their size, 32 bytes at most): one
// 256-bit load for eight (two 128-bit ones made twice the L1 and L2 requests).  Not ordered with
// other accesses by the compiler: what an older value lets through is settled by the atomic.
template <int G>
__device__ __forceinline__ void load_row(const uint32_t* p, uint32_t (&r)[G]) {
    if constexpr (G == 8) {
        asm volatile("ld.relaxed.gpu.global.v8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                     : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
                     : "l"(p));
    } else if constexpr (G == 4) {
        asm volatile("ld.relaxed.gpu.global.v4.b32 {%0, %1, %2, %3}, [%4];"
                     : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                     : "l"(p));
    } else if constexpr (G == 2) {
        asm volatile("ld.relaxed.gpu.global.v2.b32 {%0, %1}, [%2];" : "=r"(r[0]), "=r"(r[1]) : "l"(p));
    } else {
        asm volatile("ld.relaxed.gpu.global.b32 %0, [%1];" : "=r"(r[0]) : "l"(p));
    }
}

// the same from data that no longer changes (through L1: lanes share rows)
template <int G>
__device__ __forceinline__ void load_final(const uint32_t* p, uint32_t (&r)[G]) {
    if constexpr (G == 8) {
        asm("ld.global.nc.v8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
            : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
            : "l"(p));
    } else if constexpr (G == 4) {
        const uint4 a = __ldg(reinterpret_cast<const uint4*>(p));
        r[0] = a.x, r[1] = a.y, r[2] = a.z, r[3] = a.w;
    } else if constexpr (G == 2) {
        const uint2 a = __ldg(reinterpret_cast<const uint2*>(p));
        r[0] = a.x, r[1] = a.y;
    } else {
        r[0] = __ldg(p);
    }
}

// G packed words of an item: predecessors, distances.  Loaded as 64-bit elements, each of which is whole (the
// halves of a word read apart could be a new distance with an old, lower label: a candidate of that
// distance and a label between the two would be dropped).
template <int G>
__device__ __forceinline__ void load_keys(const uint32_t* dist, uint32_t item, uint32_t (&lo)[G], uint32_t (&hi)[G]) {
    const uint32_t* const p = dist + (size_t)item * (2 * G);
    unsigned long long x[G];
    if constexpr (G == 4)
        asm volatile("ld.relaxed.gpu.global.v4.b64 {%0, %1, %2, %3}, [%4];" : "=l"(x[0]), "=l"(x[1]), "=l"(x[2]), "=l"(x[3]) : "l"(p));
    else if constexpr (G == 2)
        asm volatile("ld.relaxed.gpu.global.v2.b64 {%0, %1}, [%2];" : "=l"(x[0]), "=l"(x[1]) : "l"(p));
    else
        asm volatile("ld.relaxed.gpu.global.b64 %0, [%1];" : "=l"(x[0]) : "l"(p));
#pragma unroll
    for (int s = 0; s < G; ++s) lo[s] = (uint32_t)x[s], hi[s] = (uint32_t)(x[s] >> 32);
}

template <int G>
__device__ __forceinline__ void shared_row(const uint32_t* p, uint32_t (&r)[G]) {
    if constexpr (G >= 4) {
#pragma unroll
        for (int i = 0; i < G; i += 4) {
            const uint4 a = *reinterpret_cast<const uint4*>(p + i);
            r[i] = a.x, r[i + 1] = a.y, r[i + 2] = a.z, r[i + 3] = a.w;
        }
    } else {
#pragma unroll
        for (int s = 0; s < G; ++s) r[s] = p[s];
    }
}

// All blocks arrive and wait; false once a limit has run out or another block gave up.
__device__ bool grid_barrier(const SweepLaunch& L, BlockMem& bm, uint32_t& n, uint64_t t_begin) {
    ++n;
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        atomicAdd(&L.ctl->bar, 1u);
        const uint32_t target = n * gridDim.x;
        const uint64_t t0 = globaltimer_ns();
        bool late = t0 - t_begin > LIMIT_FACTOR * L.timeout_ns, stop = false;
        while (!late && !stop && (int32_t)(ld_acquire(&L.ctl->bar) - target) < 0) {
            stop = ld_relaxed(&L.hdr->abort_flag) != 0u;
            late = globaltimer_ns() - t0 > L.timeout_ns;
        }
        if (late) {
            set_status(L.hdr, SSSP_ETIMEOUT);
            atomicExch(&L.hdr->abort_flag, 1u);
        }
        __threadfence();
        bm.ok = !late && !stop;
    }
    __syncthreads();
    return bm.ok != 0;
}

template <class W, int G, class Launch>
struct Worker {
    static constexpr bool WARM = std::is_same<Launch, WarmLaunch>::value;
    const Launch& L;
    WarpMem& wm;
    uint32_t* du;  // [32][G] distances of the rows held
    BlockMem& bm;
    uint32_t lane;
    uint32_t* list;              // list being filled (A from the front, M from the back)
    SweepIter* it;               // its counters
    unsigned long long* ex_out;  // hub entries being filled
    uint32_t nA, nM, nC;         // buffered items: new in the lists, to be marked (warp-uniform)
    uint32_t bad, s_at, s_imp;

    __device__ __forceinline__ uint32_t vertex(uint32_t item) const { return L.groups == 1u ? item : item % L.V; }

    __device__ __forceinline__ void put(uint32_t at, uint32_t item, bool back) {
        if constexpr (WARM) {
            if (at < (back ? L.capM : L.capA))
                list[back ? L.capA + L.capM - 1u - at : at] = item;
            else
                it->stop = 1u;  // (its mark stays)
        } else {
            list[back ? L.items - 1u - at : at] = item;
        }
    }

    __device__ __forceinline__ void flush_full(uint32_t* buf, uint32_t& n, uint32_t* cnt, bool back) {
        uint32_t base = 0;
        if (lane == 0) base = atomicAdd(cnt, 32u);
        base = __shfl_sync(0xFFFFFFFFu, base, 0);
        put(base + lane, buf[lane], back);
        n -= 32u;
        const uint32_t x = buf[32u + lane];
        __syncwarp();
        buf[lane] = x;
        __syncwarp();
    }

    // newly marked items of the lanes with `has` (and an edge): hubs get their entry, the others go
    // to the warp's buffers
    __device__ __forceinline__ void push(bool has, uint32_t item, uint32_t deg) {
        has = has && deg != 0u;
        if (has && deg >= SWEEP_HUB) {
            const unsigned long long at = atomicAdd(&it->ex, (1ull << 32) | ((deg + SEG - 1u) / SEG));
            ex_out[at >> 32] = ((unsigned long long)(uint32_t)at << 32) | item;
            has = false;
        }
        const uint32_t ba = __ballot_sync(0xFFFFFFFFu, has && deg < SMALL_ROW);
        const uint32_t bmm = __ballot_sync(0xFFFFFFFFu, has && deg >= SMALL_ROW);
        const uint32_t lt = (1u << lane) - 1u;
        if (has) {
            if (deg < SMALL_ROW)
                wm.bufA[nA + __popc(ba & lt)] = item;
            else
                wm.bufM[nM + __popc(bmm & lt)] = item;
        }
        nA += __popc(ba);
        nM += __popc(bmm);
        __syncwarp();
        if (nA >= 32u) flush_full(wm.bufA, nA, &it->nA, false);
        if (nM >= 32u) flush_full(wm.bufM, nM, &it->nM, true);
    }

    // the leftovers of all warps of the block, with one atomic per list (called by every thread)
    __device__ __forceinline__ void flush_block() {
        if (!__syncthreads_or((int)(nA | nM))) return;
        const uint32_t wid = threadIdx.x >> 5;
        if (lane == 0) bm.wA[wid] = nA, bm.wM[wid] = nM;
        __syncthreads();
        if (threadIdx.x < 32u) {
            // lanes 0..15: list A, lanes 16..31: list M
            const bool m = lane >= NW;
            uint32_t* const c = m ? bm.wM : bm.wA;
            const uint32_t x = c[lane % NW];
            uint32_t inc = x;
#pragma unroll
            for (uint32_t o = 1; o < NW; o <<= 1) {
                const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, inc, o, NW);
                if (lane % NW >= o) inc += y;
            }
            uint32_t base = 0;
            if (lane % NW == NW - 1u && inc) base = atomicAdd(m ? &it->nM : &it->nA, inc);
            base = __shfl_sync(0xFFFFFFFFu, base, NW - 1, NW);
            c[lane % NW] = base + inc - x;
        }
        __syncthreads();
        for (uint32_t i = lane; i < nA; i += 32u) put(bm.wA[wid] + i, wm.bufA[i], false);
        for (uint32_t i = lane; i < nM; i += 32u) put(bm.wM[wid] + i, wm.bufM[i], true);
        nA = nM = 0;
    }

    __device__ __forceinline__ void load_dist(uint32_t item, uint32_t (&r)[G]) const {
        if constexpr (WARM) {
            uint32_t lo[G];
            load_keys<G>(L.dist, item, lo, r);
#pragma unroll
            for (int s = 0; s < G; ++s) r[s] = min(r[s], Dist<W>::INF);
        } else {
            load_row<G>(L.dist + (size_t)item * G, r);
        }
    }

    // Takes the item of each lane with `ok`: its mark is cleared before its distances are read, so a
    // distance lowered after the read marks it again (mark_all).  An atomic with acquire semantics: a
    // reduction, which has no result, reads nothing that could order the loads after it.
    __device__ __forceinline__ void take(bool ok, uint32_t item, uint32_t (&r)[G]) {
#pragma unroll
        for (int s = 0; s < G; ++s) r[s] = Dist<W>::INF;
        if (ok) {
            and_acquire(&L.mark[item >> 5], ~(1u << (item & 31u)));
            load_dist(item, r);
        }
    }

    // a row into slot `at` (off: its first edge less the edges of the rows before it); returns its
    // count of finite distances
    __device__ __forceinline__ uint32_t hold(uint32_t at, const uint32_t (&r)[G], uint32_t item, uint32_t off) {
        uint32_t fin = 0, mx = 0;
#pragma unroll
        for (int s = 0; s < G; ++s)
            if (r[s] < Dist<W>::INF) ++fin, mx = max(mx, r[s]);
        if constexpr (G >= 4) {
#pragma unroll
            for (int s = 0; s < G; s += 4)
                *reinterpret_cast<uint4*>(du + at * G + s) = make_uint4(r[s], r[s + 1], r[s + 2], r[s + 3]);
        } else {
#pragma unroll
            for (int s = 0; s < G; ++s) du[at * G + s] = r[s];
        }
        uint32_t lab = 0;
        if constexpr (WARM) lab = L.ids ? __ldg(&L.ids[vertex(item)]) : vertex(item);
        wm.row[at] = make_uint4(off, L.groups == 1u ? 0u : item - item % L.V, mx, lab);
        return fin;
    }

    // Marks the nC buffered items, whose distances this warp has lowered, MQ a lane; newly marked ones go to
    // the list being filled.  A mark is always set by a read-modify-write, also where the item has one: it
    // comes either before the clearing in take, which then sees the lowered distance (the fence here, the
    // mark, the acquire there), or after it, and lists the item again.  A plain look that left marked items out
    // would not be ordered so (each side would write one word and read the other's) without a sequentially
    // consistent fence on both sides, and with them it is no faster: R-MAT scale 22, 8 sources 4.04 ms with
    // the look, 3.98 without; random graphs of 16,384 vertices, 1 source 333 and 309 us, of 1 M, 8 sources
    // 2.29 and 2.22 ms.
    __device__ __forceinline__ void mark_all() {
        __syncwarp();
        fence_gpu();  // the lowered distances before the marks
        uint32_t nact = 0;
#pragma unroll
        for (uint32_t i = 0; i < MQ; ++i) {
            const uint32_t x = i * 32u + lane;
            bool f = x < nC;
            if (!__any_sync(0xFFFFFFFFu, f)) continue;
            uint32_t item = 0, deg = 0;
            if (f) {
                item = wm.low[x];
                const uint32_t v = vertex(item), bit = 1u << (item & 31u);
                const uint32_t r0 = __ldg(&L.row_ptr[v]), r1 = __ldg(&L.row_ptr[v + 1]);  // in flight with the atomic
                f = !(atomicOr(&L.mark[item >> 5], bit) & bit);
                deg = r1 - r0;
            }
            nact += __popc(__ballot_sync(0xFFFFFFFFu, f));
            push(f, item, deg);
        }
        if (lane == 0) wm.act += nact;
        nC = 0;
        __syncwarp();
    }

    // Relaxes edges [0, total) of the rows held.  Row r's edges start at the value p of lane r
    // (ascending, every row has an edge; lanes without a row: none), so the rows that start within
    // the 32 edges of a step are a bit mask, and a lane's row is the count of starts up to it.
    // A pipeline of three: the (col, w) of the steps after next, the distances of the next ones and
    // the atomics of these are in flight together (EB steps each; four of them for one or two sources, or three, spill
    // registers: R-MAT scale 18, 1 source 0.65 and 0.63 against 0.59 ms, scale 20, 2 sources 1.11 and 0.98
    // against 0.93 ms).
    __device__ __forceinline__ void relax(uint32_t total, uint32_t p) {
        constexpr int EB = G >= 8 || (WARM && G >= 4) ? 1 : 2;
        uint32_t v[EB], w[EB], a[EB];              // steps after next: head, weight, row
        uint32_t x[EB], y[EB], b[EB], d[EB][G];    // next steps: item, weight, row, its distances
        uint32_t pr[EB][WARM ? G : 1];             // (warm) and predecessors
        uint32_t seen = 0;                         // rows that start before the step
        auto fetch = [&](uint32_t k0) {            // k0: first edge of the steps
#pragma unroll
            for (int j = 0; j < EB; ++j) {
                const uint32_t at = k0 + 32u * j;
                v[j] = NONE;
                if (at >= total) continue;
                const uint32_t starts = __reduce_or_sync(0xFFFFFFFFu, p - at < 32u ? 1u << (p - at) : 0u);
                a[j] = seen + __popc(starts & (0xFFFFFFFFu >> (31u - lane))) - 1u;
                seen += __popc(starts);
                if (at + lane < total) {
                    const uint32_t e = wm.row[a[j]].x + at + lane;
                    v[j] = __ldg(&L.col[e]);
                    w[j] = __ldg(&L.w[e]);
                }
            }
        };
        auto heads = [&]() {
#pragma unroll
            for (int j = 0; j < EB; ++j) {
                x[j] = v[j];
                y[j] = w[j];
                b[j] = a[j];
                if (x[j] == NONE) continue;
                if (!W::weight_ok(y[j]) || x[j] >= L.V) {
                    bad |= 1u;
                    x[j] = NONE;
                } else {
                    const uint4 rw = wm.row[b[j]];
                    uint32_t z;
                    if (!W::add(rw.z, y[j], z)) {  // (judged at the end: k_sweep_requeue)
                        bad |= 2u;
                        if constexpr (WARM) {
                            const uint32_t tail = rw.y + (L.slots ? __ldg(&L.slots[rw.w]) : rw.w);
                            atomicOr(&L.over[tail >> 5], 1u << (tail & 31u));
                        }
                    }
                    x[j] += rw.y;
                    if constexpr (WARM)
                        load_keys<G>(L.dist, x[j], pr[j], d[j]);
                    else
                        load_row<G>(L.dist + (size_t)x[j] * G, d[j]);
                }
            }
        };
        fetch(0);
        heads();
        fetch(32u * EB);
        for (uint32_t k0 = 0; k0 < total; k0 += 32u * EB) {
            // these steps: candidates c where they beat the distances read, else INF
            uint32_t c[EB][G], it_[EB], imp[EB], lab[EB], any = 0;
#pragma unroll
            for (int j = 0; j < EB; ++j) {
                it_[j] = x[j];
                imp[j] = 0;
                if (x[j] != NONE) {
                    uint32_t dj[G];
                    shared_row<G>(du + b[j] * G, dj);
                    if constexpr (WARM) lab[j] = wm.row[b[j]].w;
#pragma unroll
                    for (int s = 0; s < G; ++s) {
                        c[j][s] = Dist<W>::add(dj[s], y[j]);
                        if constexpr (WARM) {
                            if (c[j][s] < Dist<W>::INF &&
                                (c[j][s] < d[j][s] || (c[j][s] == d[j][s] && lab[j] < pr[j][s])))
                                imp[j] |= 1u << s;
                        } else if (c[j][s] < d[j][s]) {
                            imp[j] |= 1u << s;
                        }
                    }
                }
                any |= imp[j];
            }
            heads();
            fetch(k0 + 64u * EB);
            if (!__any_sync(0xFFFFFFFFu, any != 0u)) continue;
            uint32_t low[EB];
#pragma unroll
            for (int j = 0; j < EB; ++j) {
                low[j] = 0;
                uint32_t* const row = L.dist + (size_t)it_[j] * (WARM ? 2 * G : G);
                uint32_t old[G];
#pragma unroll
                for (int s = 0; s < G; ++s) {
                    old[s] = 0;
                    if constexpr (WARM) {
                        if (imp[j] & (1u << s))
                            old[s] = (uint32_t)(atomicMin(reinterpret_cast<unsigned long long*>(row) + s,
                                                          (unsigned long long)c[j][s] << 32 | lab[j]) >> 32);
                    } else {
                        if (imp[j] & (1u << s)) old[s] = atomicMin(row + s, c[j][s]);
                    }
                }
#pragma unroll
                for (int s = 0; s < G; ++s)
                    if (old[s] > c[j][s]) low[j] |= imp[j] & (1u << s);
            }
            uint32_t na = 0, nl = 0;
#pragma unroll
            for (int j = 0; j < EB; ++j) {
                na += __popc(imp[j]);
                nl += __popc(low[j]);
                const uint32_t bl = __ballot_sync(0xFFFFFFFFu, low[j] != 0u);
                if (!bl) continue;
                if (low[j]) wm.low[nC + __popc(bl & ((1u << lane) - 1u))] = it_[j];
                nC += __popc(bl);
                if (nC > MARKS - 32u) mark_all();
            }
            s_at += na;
            s_imp += nl;
        }
    }

    // An iteration's work: hub segments, then the rows of M, then those of A, in units that the
    // block's warps take in turn (unit i of block b is unit b + i * blocks of the iteration).
    __device__ __forceinline__ void work(const uint32_t* in, const unsigned long long* ex, uint32_t cA, uint32_t cM,
                                         uint32_t cX, uint32_t segs) {
        const uint32_t TW = gridDim.x * NW;
        uint32_t last = L.items - 1u;  // of a list
        if constexpr (WARM) last = L.capA + L.capM - 1u;
        // segments and rows of a unit: fewer when there are few, so that all warps get some
        const uint32_t rX = min(max(segs / (2u * TW), 1u), 8u), rM = min(max(cM / TW, 1u), 8u);
        const uint32_t rA = cA >= TW * 32u ? 32u : cA >= TW * 16u ? 16u : 8u;
        const uint32_t uX = (segs + rX - 1u) / rX, uM = (cM + rM - 1u) / rM, uA = (cA + rA - 1u) / rA;
        uint32_t t = 0, t1 = 0, k = 0;  // hub segments of the unit, entry of the first
        for (;;) {
            uint32_t total = 0, p = 0xFFFFFFFFu;
            if (t >= t1) {
                uint32_t u = 0;
                if (lane == 0) u = atomicAdd(&bm.next, 1u);
                u = blockIdx.x + __shfl_sync(0xFFFFFFFFu, u, 0) * gridDim.x;
                if (u < uX) {
                    t = u * rX;
                    t1 = min(t + rX, segs);
                    k = 0;  // last entry whose start is <= t: 32-way search of start << 32 | item
                    uint32_t len = cX;
                    while (len > 1u) {
                        const uint32_t step = (len + 31u) / 32u, i = lane * step;
                        const bool le = i < len && (uint32_t)(__ldcg(&ex[k + i]) >> 32) <= t;
                        const uint32_t f = 31u - (uint32_t)__clz(__ballot_sync(0xFFFFFFFFu, le));
                        k += f * step;
                        len = min(step, len - f * step);
                    }
                } else if (u < uX + uM + uA) {
                    const bool m = u < uX + uM;
                    const uint32_t c = m ? (u - uX) * rM : (u - uX - uM) * rA;
                    const bool ok = lane < (m ? rM : rA) && c + lane < (m ? cM : cA);
                    uint32_t item = 0, beg = 0, deg = 0, r[G];
                    if (ok) {
                        item = __ldcg(&in[m ? last - (c + lane) : c + lane]);
                        const uint32_t x = vertex(item);
                        beg = __ldg(&L.row_ptr[x]);
                        deg = __ldg(&L.row_ptr[x + 1]) - beg;
                    }
                    take(ok, item, r);
                    uint32_t inc = deg;
#pragma unroll
                    for (uint32_t o = 1; o < 32u; o <<= 1) {
                        const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, inc, o);
                        if (lane >= o) inc += y;
                    }
                    const uint32_t fin = hold(lane, r, item, beg - (inc - deg));
                    if (ok) p = inc - deg;
                    total = __shfl_sync(0xFFFFFFFFu, inc, 31);
                    const uint32_t se = __reduce_add_sync(0xFFFFFFFFu, fin * deg), sv = __reduce_add_sync(0xFFFFFFFFu, fin);
                    if (lane == 0) wm.edges += se, wm.vert += sv;
                } else {
                    break;
                }
            }
            if (t < t1) {  // the unit's segments of one hub (its mark was cleared before the iteration)
                const unsigned long long x = __ldcg(&ex[k]);
                const uint32_t item = (uint32_t)x, u = vertex(item), s0 = t - (uint32_t)(x >> 32);
                const uint32_t beg = __ldg(&L.row_ptr[u]) + s0 * SEG, left = __ldg(&L.row_ptr[u + 1]) - beg;
                const uint32_t n = min((left + SEG - 1u) / SEG, t1 - t);
                total = min(left, n * SEG);
                if (lane == 0) {
                    uint32_t r[G];
                    load_dist(item, r);
                    const uint32_t fin = hold(0, r, item, beg);
                    wm.edges += (unsigned long long)fin * total;
                    if (s0 == 0) wm.vert += fin;
                    p = 0;
                }
                t += n;
                ++k;
            }
            __syncwarp();
            relax(total, p);
            __syncwarp();
        }
        if (nC) mark_all();
    }
};

// Every distance to INF, marks and counters to zero, predecessors to NONE.
__global__ void k_sweep_init(SweepLaunch L, uint32_t inf) {
    const size_t stride = (size_t)gridDim.x * blockDim.x, i0 = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    const size_t nd = (size_t)L.items * L.G;
    uint4* d4 = reinterpret_cast<uint4*>(L.dist);
    for (size_t i = i0; i < nd / 4; i += stride) d4[i] = make_uint4(inf, inf, inf, inf);
    if (i0 < (nd & 3u)) L.dist[(nd & ~(size_t)3) + i0] = inf;
    for (size_t i = i0; i < ((size_t)L.items + 31) / 32; i += stride) L.mark[i] = 0u;
    for (size_t i = i0; i < sizeof(SweepCtl) / 4; i += stride) reinterpret_cast<uint32_t*>(L.ctl)[i] = 0u;
    for (size_t i = i0; i < L.n_dirty; i += stride) L.dirty[i] = 0u, L.nfsplit[i] = 0u;
    if (L.pred)
        for (size_t i = i0; i < (size_t)L.S * L.V; i += stride) L.pred[i] = NONE;
}

// What is next, from the counters of the iteration to come (one thread; the same answer in every block).
template <class Launch>
__device__ __forceinline__ uint32_t decide(const Launch& L, BlockMem& bm) {
    constexpr bool WARM = std::is_same<Launch, WarmLaunch>::value;
    if (!(bm.c[0] | bm.c[1] | bm.c[3])) return SWEPT_DONE;
    if (WARM) return bm.c[6] || bm.iters == WARM_ITERS ? SWEPT_HANDED : GO_ON;
    if (bm.iters == HOPS_ITERS && bm.total < L.few) return ASK;
    if (bm.iters == 0u || bm.iters % HAND_EVERY != 0u) return GO_ON;
    if (bm.slow) {
        const float done = (float)bm.total / ((float)L.E * (float)L.S);
        const uint32_t most = bm.iters == HAND_EVERY ? HAND_ITERS : 4u * HAND_ITERS;  // (those begun are finished)
        return done * (float)most >= (float)bm.iters ? GO_ON : done < 1.0f ? SWEPT_AGAIN : SWEPT_HANDED;
    }
    if (bm.total - bm.looked < HAND_EVERY * HAND_EDGES) return SWEPT_HANDED;
    bm.looked = bm.total;
    return GO_ON;
}

template <class W, int G, class Launch>
__global__ void __launch_bounds__(WT, 2) k_sweep(Launch L) {
    constexpr bool WARM = std::is_same<Launch, WarmLaunch>::value;
    extern __shared__ __align__(16) uint32_t dsm[];  // [NW][32][G] rows
    __shared__ BlockMem bm;
    __shared__ WarpMem wmem[NW];
    const uint32_t tid = threadIdx.x, lane = tid & 31u, wid = tid >> 5;
    WarpMem& wm = wmem[wid];
    const uint64_t t_begin = globaltimer_ns();
    uint32_t nbar = 0;
    if (tid == 0) {
        bm.work = bm.at = bm.imp = bm.total = bm.looked = 0ull;
        bm.iters = bm.slow = 0u;
        bm.then = SWEPT_HANDED;  // (a limit has run out)
    }
    if (lane == 0) {
        wm.edges = 0ull;
        wm.act = wm.vert = 0u;
    }
    if constexpr (WARM) {  // the tails that a source has reached
        __syncthreads();
        Worker<W, G, Launch> wk{L, wm, dsm + wid * 32u * G, bm, lane, L.list[0], &L.ctl->it[0], L.ex[0], 0, 0, 0, 0, 0, 0};
        for (unsigned long long i0 = (unsigned long long)blockIdx.x * WT + wid * 32u; i0 < L.n_tails;
             i0 += (unsigned long long)gridDim.x * WT) {
            uint32_t t = i0 + lane < L.n_tails ? __ldg(&L.tails[i0 + lane]) : NONE;
            if (i0 + lane < L.n_tails && t >= L.V) set_status(L.hdr, SSSP_EINVAL);
            const bool ok = i0 + lane < L.n_tails && t < L.V;
            if (ok && L.slots) t = __ldg(&L.slots[t]);
            const uint32_t deg = ok ? __ldg(&L.row_ptr[t + 1]) - __ldg(&L.row_ptr[t]) : 0u;
            for (uint32_t g = 0; g < L.groups; ++g) {
                const uint32_t item = g * L.V + t, bit = 1u << (item & 31u);
                bool has = false;
                if (ok) {
                    uint32_t r[G];
                    wk.load_dist(item, r);
#pragma unroll
                    for (int s = 0; s < G; ++s) has = has || r[s] < Dist<W>::INF;
                }
                if (has) has = !(atomicOr(&L.mark[item >> 5], bit) & bit);  // (a tail may be listed twice)
                wk.push(has, item, deg);
            }
        }
        wk.flush_block();
    } else if (blockIdx.x == 0) {  // seeds
        for (uint32_t s = tid; s < L.S; s += WT) {
            uint32_t src = L.sources[s];
            if (src >= L.V) {
                set_status(L.hdr, SSSP_EINVAL);
                continue;
            }
            if (L.slots) src = L.slots[src];
            const uint32_t item = s / G * L.V + src, bit = 1u << (item & 31u);
            L.dist[(size_t)item * G + s % G] = 0u;
            if (atomicOr(&L.mark[item >> 5], bit) & bit) continue;
            const uint32_t deg = __ldg(&L.row_ptr[src + 1]) - __ldg(&L.row_ptr[src]);
            if (deg >= SWEEP_HUB) {
                const unsigned long long at = atomicAdd(&L.ctl->it[0].ex, (1ull << 32) | ((deg + SEG - 1u) / SEG));
                L.ex[0][at >> 32] = ((unsigned long long)(uint32_t)at << 32) | item;
            } else if (deg >= SMALL_ROW) {
                L.list[0][L.items - 1u - atomicAdd(&L.ctl->it[0].nM, 1u)] = item;
            } else if (deg) {
                L.list[0][atomicAdd(&L.ctl->it[0].nA, 1u)] = item;
            }
        }
    }
    uint32_t slot = 0, par = 0;
    while (grid_barrier(L, bm, nbar, t_begin)) {
        if (tid == 0) {  // the counters of this iteration (nobody adds to them any more)
            const uint4* const it = reinterpret_cast<const uint4*>(&L.ctl->it[slot]);
            const uint4 x = __ldcg(it), y = __ldcg(it + 1);
            bm.next = 0u;
            bm.c[0] = x.x, bm.c[1] = x.y, bm.c[2] = x.z, bm.c[3] = x.w, bm.c[6] = y.z;
            bm.total += ((unsigned long long)y.y << 32) | y.x;
            bm.then = decide(L, bm);
            bm.iters += bm.then >= ASK;
        }
        __syncthreads();
        const uint32_t cA = bm.c[0], cM = bm.c[1], segs = bm.c[2], cX = bm.c[3];
        if (!WARM && bm.then == ASK) {  // (the same weights in every block)
            const uint32_t e = (uint32_t)((unsigned long long)tid * L.E / WT);
            const bool keep = __syncthreads_count(__ldg(&L.w[e]) > L.narrow) > (int)WT / 2;
            if (tid == 0) bm.slow = keep, bm.then = keep ? GO_ON : SWEPT_AGAIN;
            __syncthreads();
        }
        if (bm.then != GO_ON) break;
        const uint32_t next = slot == 2u ? 0u : slot + 1u, after = next == 2u ? 0u : next + 1u;
        if (blockIdx.x == 0 && tid == 0) {  // its counters were last read before this barrier
            SweepIter& z = L.ctl->it[after];
            z.nA = z.nM = 0u;
            if (WARM) z.stop = 0u;
            z.ex = z.work = 0ull;
        }
        if (cX) {
            // hubs are taken before the iteration, since several warps relax one: a distance that
            // falls from here on marks it again
            for (uint32_t i = blockIdx.x * WT + tid; i < cX; i += gridDim.x * WT) {
                const uint32_t item = (uint32_t)__ldcg(&L.ex[par][i]);
                atomicAnd(&L.mark[item >> 5], ~(1u << (item & 31u)));
            }
            if (!grid_barrier(L, bm, nbar, t_begin)) break;
        }
        Worker<W, G, Launch> wk{L, wm, dsm + wid * 32u * G, bm, lane, L.list[par ^ 1u], &L.ctl->it[next], L.ex[par ^ 1u], 0, 0, 0, 0, 0, 0};
        const unsigned long long before = wm.edges;
        wk.work(L.list[par], L.ex[par], cA, cM, cX, segs);
        wk.bad = __reduce_or_sync(0xFFFFFFFFu, wk.bad);
        wk.s_at = __reduce_add_sync(0xFFFFFFFFu, wk.s_at);
        wk.s_imp = __reduce_add_sync(0xFFFFFFFFu, wk.s_imp);
        if (lane == 0) {
            if (wk.s_at) atomicAdd(&bm.at, (unsigned long long)wk.s_at);
            if (wk.s_imp) atomicAdd(&bm.imp, (unsigned long long)wk.s_imp);
            if (wm.edges != before) atomicAdd(&bm.work, wm.edges - before);
            if (wk.bad & 1u) set_status(L.hdr, SSSP_EINVAL);
            if (wk.bad & 2u) st_relaxed(&L.hdr->over, 1u);
        }
        wk.flush_block();
        if (tid == 0 && bm.work) {
            atomicAdd(&L.ctl->it[next].work, bm.work);
            bm.work = 0ull;
        }
        slot = next;
        par ^= 1u;
    }
    __syncthreads();
    if (lane == 0) {  // edges_scanned, atomics, improved, activations, vertices
        if (wm.edges) atomicAdd(&L.hdr->stats[0], wm.edges);
        if (wm.act) atomicAdd(&L.hdr->stats[3], (unsigned long long)wm.act);
        if (wm.vert) atomicAdd(&L.hdr->stats[5], (unsigned long long)wm.vert);
    }
    if (tid == 0) {
        if (bm.at) atomicAdd(&L.hdr->stats[1], bm.at);
        if (bm.imp) atomicAdd(&L.hdr->stats[2], bm.imp);
    }
    if (blockIdx.x == 0 && tid == 0) {
        atomicAdd(&L.hdr->stats[4], (unsigned long long)bm.iters);
        L.hdr->swept = bm.then == GO_ON ? SWEPT_HANDED : bm.then;
    }
}

// The results: distances in the caller's order, and predecessors by one pass over the edges.  A
// warp walks a range of edges (rowwalk.cuh).  The (col, w) of the step after next and the heads' distances of the next one are in
// flight while a step is compared; the tails' distances come through L1.
template <class W, int G>
__global__ void __launch_bounds__(256) k_sweep_out(SweepLaunch L, uint32_t per) {
    __shared__ uint32_t rows[8][32], starts[8][32];
    using D = Dist<W>;
    if (L.hdr->swept == SWEPT_AGAIN) return;
    const uint32_t lane = threadIdx.x & 31u, wid = threadIdx.x >> 5;
    for (uint32_t g = 0; g < L.groups; ++g) {
        for (uint32_t c = blockIdx.x * blockDim.x + threadIdx.x; c < L.V; c += gridDim.x * blockDim.x) {
            const uint32_t at = L.slots ? __ldg(&L.slots[c]) : c;
            uint32_t r[G];
            load_final<G>(L.dist + ((size_t)g * L.V + at) * G, r);
#pragma unroll
            for (int s = 0; s < G; ++s)
                if (g * G + s < L.S) L.out[(size_t)(g * G + s) * L.V + c] = r[s];
        }
    }
    if (!L.pred) return;
    const unsigned long long first = (unsigned long long)((blockIdx.x * blockDim.x + threadIdx.x) >> 5) * per;
    if (first >= L.E) return;
    const uint32_t e0 = (uint32_t)first, e1 = (uint32_t)min(first + per, (unsigned long long)L.E);
    RowWalk walk{L.row_ptr, L.V, rows[wid], starts[wid]};
    walk.seek(e0);
    uint32_t v = 0, w = 0;  // the step after next
    auto fetch = [&](uint32_t e) {
        v = NONE;
        if (e < e1) v = __ldg(&L.col[e]), w = __ldg(&L.w[e]);
        if (v != NONE && (v >= L.V || !W::weight_ok(w))) v = NONE;  // (reported by the sweep)
    };
    uint32_t x, y, h[G];  // the next step: head, weight, and (one group) the head's distances
    auto heads = [&]() {
        x = v;
        y = w;
        if (L.groups == 1u && x != NONE) load_final<G>(L.dist + (size_t)x * G, h);
    };
    fetch(e0 + lane);
    heads();
    fetch(e0 + 32u + lane);
    for (uint32_t eb = e0; eb < e1; eb += 32u) {
        const uint32_t u = walk.step(eb, e1);
        uint32_t hv[G];
        const uint32_t head = x, wt = y;
#pragma unroll
        for (int s = 0; s < G; ++s) hv[s] = h[s];
        heads();
        fetch(eb + 64u + lane);
        if (head == NONE) continue;
        for (uint32_t g = 0; g < L.groups; ++g) {
            uint32_t a[G];
            load_final<G>(L.dist + ((size_t)g * L.V + u) * G, a);
            if (L.groups != 1u) load_final<G>(L.dist + ((size_t)g * L.V + head) * G, hv);
            uint32_t tight = 0;
#pragma unroll
            for (int s = 0; s < G; ++s)
                if (D::add(a[s], wt) == hv[s]) tight |= 1u << s;
            if (tight) {
                const uint32_t lab = L.ids ? __ldg(&L.ids[u]) : u, to = L.ids ? __ldg(&L.ids[head]) : head;
#pragma unroll
                for (int s = 0; s < G; ++s)
                    if ((tight & (1u << s)) && hv[s] < D::INF) atomicMin(&L.pred[(size_t)(g * G + s) * L.V + to], lab);
            }
        }
    }
}

// Warm start: the rows from the previous result.
template <int G>
__global__ void k_warm_rows(WarmLaunch L) {
    const size_t stride = (size_t)gridDim.x * blockDim.x, i0 = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    for (size_t i = i0; i < L.n_dirty; i += stride) L.dirty[i] = 0u, L.nfsplit[i] = 0u;
    for (size_t i = i0; i < sizeof(SweepCtl) / 4; i += stride) reinterpret_cast<uint32_t*>(L.ctl)[i] = 0u;
    for (size_t c = i0; c < L.V; c += stride) {
        const uint32_t at = L.slots ? __ldg(&L.slots[c]) : (uint32_t)c;
        for (uint32_t g = 0; g < L.groups; ++g) {
            uint32_t* const row = L.dist + ((size_t)g * L.V + at) * (2 * G);
            uint32_t x[2 * G];
#pragma unroll
            for (int s = 0; s < G; ++s) {
                const size_t i = (size_t)(g * G + s) * L.V + c;
                const uint32_t d = g * G + s < L.S ? __ldg(&L.out[i]) : L.inf;
                x[2 * s] = d != L.inf ? __ldg(&L.pred[i]) : NONE;
                x[2 * s + 1] = d != L.inf ? d : 0xFFFFFFFFu;
            }
            if constexpr (G >= 2) {
#pragma unroll
                for (int s = 0; s < 2 * G; s += 4)
                    *reinterpret_cast<uint4*>(row + s) = make_uint4(x[s], x[s + 1], x[s + 2], x[s + 3]);
            } else {
                *reinterpret_cast<uint2*>(row) = make_uint2(x[0], x[1]);
            }
        }
    }
}

// Warm start: the result from the rows (also that of a sweep that gave up, to be packed again).
template <int G>
__global__ void k_warm_out(WarmLaunch L) {
    const size_t stride = (size_t)gridDim.x * blockDim.x;
    for (size_t c = (size_t)blockIdx.x * blockDim.x + threadIdx.x; c < L.V; c += stride) {
        const uint32_t at = L.slots ? __ldg(&L.slots[c]) : (uint32_t)c;
        for (uint32_t g = 0; g < L.groups; ++g) {
            uint32_t x[2 * G];
            load_final<2 * G>(L.dist + ((size_t)g * L.V + at) * (2 * G), x);
#pragma unroll
            for (int s = 0; s < G; ++s) {
                if (g * G + s >= L.S) continue;
                const size_t i = (size_t)(g * G + s) * L.V + c;
                L.out[i] = min(x[2 * s + 1], L.inf);
                L.pred[i] = x[2 * s];
            }
        }
    }
}

// SSSP_EOVERFLOW if a candidate from an item's final distances does not fit: of all items, or (warm start) of
// those the sweep noted one of.  One warp per item.
template <class W, int G, class Launch>
__device__ __noinline__ void judge_overflow(const Launch& L) {
    constexpr bool WARM = std::is_same<Launch, WarmLaunch>::value;
    const uint32_t lane = threadIdx.x & 31u;
    for (size_t i = ((size_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; i < L.items; i += (size_t)gridDim.x * blockDim.x >> 5) {
        if constexpr (WARM)
            if (!(L.over[i >> 5] >> (i & 31u) & 1u)) continue;
        uint32_t most = 0;
        bool reached = false;
#pragma unroll
        for (int s = 0; s < G; ++s) {
            const uint32_t d = L.dist[WARM ? 2 * (i * G + s) + 1 : i * G + s];
            if (d < L.inf) reached = true, most = max(most, d);
        }
        if (!reached) continue;
        const uint32_t v = (uint32_t)(i % L.V), end = L.row_ptr[v + 1];
        bool bad = false;
        for (uint32_t e = L.row_ptr[v] + lane; e < end; e += 32u) {
            uint32_t z;
            bad = bad || (L.col[e] < L.V && W::weight_ok(L.w[e]) && !W::add(most, L.w[e], z));
        }
        if (bad) set_status(L.hdr, SSSP_EOVERFLOW);
    }
}

// Handed over: the marked vertices become inbox bits of the sources that have reached them, their
// units' doorbells are rung and they are counted.  One thread per inbox word (G = 1: the marks are
// the inbox words already).
// The sweep relaxes vertices at distances far above their final ones, as a solve in bucket order hardly does, so
// a candidate of its that does not fit says nothing yet.  If it has met one and has finished, the final distances
// are judged here; if it is handed over, the persistent solve starts again from the sources, as if
// there had been no sweep (a warm start cannot: it queues the items in question once more).
template <int G, class Launch>
__global__ void k_sweep_requeue(Launch L, uint32_t* bitmap, uint32_t words, uint32_t B, uint32_t Bq, uint32_t split,
                                uint32_t Q) {
    constexpr bool WARM = std::is_same<Launch, WarmLaunch>::value;
    const bool over = L.hdr->over, again = !WARM && (over || L.hdr->swept == SWEPT_AGAIN);
    if (L.hdr->swept == SWEPT_DONE) {
        if (over && L.wtype == SSSP_W_F32)
            judge_overflow<WF32, G>(L);
        else if (over)
            judge_overflow<WU32, G>(L);
        return;
    }
    const size_t n = (size_t)L.S * words, stride = (size_t)gridDim.x * blockDim.x;
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
        const uint32_t s = (uint32_t)(i / words), wd = (uint32_t)(i - (size_t)s * words);
        uint32_t bits = 0;
        for (uint32_t j = 0; j < 32u && wd * 32u + j < L.V; ++j) {
            const uint32_t item = s / G * L.V + wd * 32u + j;
            size_t d = (size_t)item * G + s % G;
            uint32_t m = L.mark[item >> 5];
            if constexpr (WARM) {
                d = 2 * d + 1;
                m |= L.over[item >> 5];
            }
            if (again ? L.dist[d] == 0u : (m >> (item & 31u) & 1u) && L.dist[d] < L.inf) bits |= 1u << j;
        }
        bitmap[i] = bits;
        if (!bits) continue;
        atomicAdd(&L.hdr->pending, (unsigned long long)__popc(bits));
        while (bits) {
            const uint32_t v = wd * 32u + (uint32_t)__ffs(bits) - 1u;
            bits &= bits - 1u;
            const uint32_t p = v / B;
            L.dirty[(size_t)s * Q + p * split + (v - p * B) / Bq] = 1u;
        }
    }
}

template <class W, class Launch>
const void* sweep_kernel(uint32_t G) {
    switch (G) {
        case 1: return (const void*)k_sweep<W, 1, Launch>;
        case 2: return (const void*)k_sweep<W, 2, Launch>;
        case 4: return (const void*)k_sweep<W, 4, Launch>;
        default: return std::is_same<Launch, WarmLaunch>::value ? nullptr : (const void*)k_sweep<W, 8, SweepLaunch>;
    }
}

template <class W>
void out_kernel(const SweepLaunch& L, uint32_t per, unsigned grid, cudaStream_t st) {
    switch (L.G) {
        case 1: k_sweep_out<W, 1><<<grid, 256, 0, st>>>(L, per); break;
        case 2: k_sweep_out<W, 2><<<grid, 256, 0, st>>>(L, per); break;
        case 4: k_sweep_out<W, 4><<<grid, 256, 0, st>>>(L, per); break;
        default: k_sweep_out<W, 8><<<grid, 256, 0, st>>>(L, per); break;
    }
}

size_t sweep_smem(uint32_t G) { return 4 * (size_t)NW * 32 * G; }

}  // namespace

cudaError_t sweep_max_blocks_per_sm(int wtype, uint32_t G, bool warm, int* out) {
    const bool f32 = wtype == SSSP_W_F32;
    const void* k = warm ? (f32 ? sweep_kernel<WF32, WarmLaunch>(G) : sweep_kernel<WU32, WarmLaunch>(G))
                         : (f32 ? sweep_kernel<WF32, SweepLaunch>(G) : sweep_kernel<WU32, SweepLaunch>(G));
    cudaError_t e;
    if ((e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sweep_smem(G))) != cudaSuccess)
        return e;
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(out, k, (int)WT, sweep_smem(G));
}

cudaError_t launch_sweep(const SweepLaunch& L, int sms, cudaStream_t st) {
    cudaError_t e;
    const size_t n = std::max((size_t)L.items * L.G / 4, L.pred ? (size_t)L.S * L.V : (size_t)1);
    const unsigned blocks = (unsigned)std::min<size_t>(std::max<size_t>((n + 255) / 256, 1), (size_t)sms * 8);
    k_sweep_init<<<blocks, 256, 0, st>>>(L, L.inf);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    const void* k = L.wtype == SSSP_W_F32 ? sweep_kernel<WF32, SweepLaunch>(L.G) : sweep_kernel<WU32, SweepLaunch>(L.G);
    void* args[] = {const_cast<SweepLaunch*>(&L)};
    return cudaLaunchCooperativeKernel(k, dim3(L.grid), dim3(WT), args, sweep_smem(L.G), st);
}

cudaError_t launch_warm_sweep(const WarmLaunch& L, int sms, cudaStream_t st) {
    cudaError_t e;
    const unsigned blocks = (unsigned)std::min<size_t>(((size_t)L.V + 255) / 256, (size_t)sms * 8);
    switch (L.G) {
        case 1: k_warm_rows<1><<<blocks, 256, 0, st>>>(L); break;
        case 2: k_warm_rows<2><<<blocks, 256, 0, st>>>(L); break;
        default: k_warm_rows<4><<<blocks, 256, 0, st>>>(L); break;
    }
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    // (the previous result has been read: its place holds the marks and the lists)
    if ((e = cudaMemsetAsync(L.mark, 0, 8 * (((size_t)L.items + 31) / 32), st)) != cudaSuccess) return e;  // (and over)
    const void* k = L.wtype == SSSP_W_F32 ? sweep_kernel<WF32, WarmLaunch>(L.G) : sweep_kernel<WU32, WarmLaunch>(L.G);
    void* args[] = {const_cast<WarmLaunch*>(&L)};
    return cudaLaunchCooperativeKernel(k, dim3(L.grid), dim3(WT), args, sweep_smem(L.G), st);
}

cudaError_t launch_warm_out(const WarmLaunch& L, int sms, cudaStream_t st) {
    const unsigned blocks = (unsigned)std::min<size_t>(((size_t)L.V + 255) / 256, (size_t)sms * 8);
    switch (L.G) {
        case 1: k_warm_out<1><<<blocks, 256, 0, st>>>(L); break;
        case 2: k_warm_out<2><<<blocks, 256, 0, st>>>(L); break;
        default: k_warm_out<4><<<blocks, 256, 0, st>>>(L); break;
    }
    return cudaGetLastError();
}

cudaError_t launch_sweep_out(const SweepLaunch& L, int sms, cudaStream_t st) {
    // a range per warp: long enough to pay for its search, short enough to give every warp one
    const uint32_t per = (uint32_t)std::min<uint64_t>(std::max<uint64_t>((L.E / ((uint64_t)sms * 64) + 31) & ~31ull, 64),
                                                      OUT_EDGES);
    const uint64_t edges = ((uint64_t)L.E + 8 * per - 1) / (8 * per);
    const unsigned grid = (unsigned)std::max<uint64_t>(edges, std::min<uint64_t>((L.V + 255) / 256, (uint64_t)sms * 8));
    if (L.wtype == SSSP_W_F32)
        out_kernel<WF32>(L, per, grid, st);
    else
        out_kernel<WU32>(L, per, grid, st);
    return cudaGetLastError();
}

cudaError_t launch_sweep_requeue(const SweepLaunch& L, uint32_t* bitmap, uint32_t words, uint32_t B, uint32_t Bq,
                                 uint32_t split, uint32_t Q, int sms, cudaStream_t st) {
    const unsigned grid = (unsigned)std::min<uint64_t>(((uint64_t)L.S * words + 255) / 256, (uint64_t)sms * 8);
    switch (L.G) {
        case 1: k_sweep_requeue<1><<<grid, 256, 0, st>>>(L, bitmap, words, B, Bq, split, Q); break;
        case 2: k_sweep_requeue<2><<<grid, 256, 0, st>>>(L, bitmap, words, B, Bq, split, Q); break;
        case 4: k_sweep_requeue<4><<<grid, 256, 0, st>>>(L, bitmap, words, B, Bq, split, Q); break;
        default: k_sweep_requeue<8><<<grid, 256, 0, st>>>(L, bitmap, words, B, Bq, split, Q); break;
    }
    return cudaGetLastError();
}

cudaError_t launch_warm_requeue(const WarmLaunch& L, uint32_t* bitmap, uint32_t words, uint32_t B, uint32_t Bq,
                                uint32_t split, uint32_t Q, int sms, cudaStream_t st) {
    const unsigned grid = (unsigned)std::min<uint64_t>(((uint64_t)L.S * words + 255) / 256, (uint64_t)sms * 8);
    switch (L.G) {
        case 1: k_sweep_requeue<1><<<grid, 256, 0, st>>>(L, bitmap, words, B, Bq, split, Q); break;
        case 2: k_sweep_requeue<2><<<grid, 256, 0, st>>>(L, bitmap, words, B, Bq, split, Q); break;
        default: k_sweep_requeue<4><<<grid, 256, 0, st>>>(L, bitmap, words, B, Bq, split, Q); break;
    }
    return cudaGetLastError();
}

}  // namespace sssp
