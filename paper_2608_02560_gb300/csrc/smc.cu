// Structured Memory Consolidation primitives (Sec. 5): two-level cluster
// routing (Eqs. smc-domain, smc-sub) and the semantic-state EMA (Eq. smc-ema).
// Session initialisation (Sec. 5.3) injects a semantic state with the
// ordinary prefill, so it needs no kernel of its own.
#include <climits>
#include <cstdint>
#include <type_traits>

#include "../../include/precog.h"
#include "internal.h"
#include "ptx.cuh"

namespace precog {
namespace {

__device__ uint32_t g_smc_status;

constexpr int kRouteWarps = 8;

constexpr int kRouteP = 8;   // prototypes scored per pass

// acc[p] = <e, protos[p]> for p < count (<= kRouteP prototypes, `stride` elements
// apart). Each lane sums a fixed subset of the coordinates in a fixed order -- 16-byte
// vectors v = lane, lane + 32, ... when VEC, single elements otherwise -- and a fixed
// xor butterfly adds the lanes, so the same two vectors always give the same score
// and every lane holds it. The count prototypes' loads of a vector are in flight
// together.
template <typename T, bool VEC>
__device__ __forceinline__ void dots_warp(const T *__restrict__ e, const T *__restrict__ protos, int64_t stride,
                                          int count, int dim, int lane, float (&acc)[kRouteP]) {
#pragma unroll
    for (int q = 0; q < kRouteP; ++q) acc[q] = 0.f;
    if constexpr (VEC) {
        constexpr int EL = 16 / static_cast<int>(sizeof(T));
        const int nvec = dim / EL;
        for (int v = lane; v < nvec; v += 32) {
            const uint4 ev = *reinterpret_cast<const uint4 *>(e + static_cast<int64_t>(v) * EL);
            uint4 pv[kRouteP];
#pragma unroll
            for (int q = 0; q < kRouteP; ++q)
                if (q < count) pv[q] = *reinterpret_cast<const uint4 *>(protos + q * stride + static_cast<int64_t>(v) * EL);
            const T *ee = reinterpret_cast<const T *>(&ev);
#pragma unroll
            for (int q = 0; q < kRouteP; ++q) {
                if (q >= count) break;
                const T *pp = reinterpret_cast<const T *>(&pv[q]);
#pragma unroll
                for (int k = 0; k < EL; ++k) acc[q] = fmaf(to_f32(ee[k]), to_f32(pp[k]), acc[q]);
            }
        }
    } else {
        for (int k = lane; k < dim; k += 32) {
            const float ek = to_f32(e[k]);
#pragma unroll
            for (int q = 0; q < kRouteP; ++q)
                if (q < count) acc[q] = fmaf(ek, to_f32(protos[q * stride + k]), acc[q]);
        }
    }
#pragma unroll
    for (int q = 0; q < kRouteP; ++q)
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) acc[q] += __shfl_xor_sync(0xffffffffu, acc[q], o);
}

// One warp per embedding: the best domain prototype, then the best of that
// domain's J[m] sub-cluster prototypes (strict '>' in index order: lowest index on
// ties, NaN never wins). slot = m * J_max + j, or -1 when no comparable score exists.
// VEC: rows are whole 16-byte vectors on 16-byte boundaries.
template <typename T, bool VEC>
__global__ void __launch_bounds__(kRouteWarps * 32, 3)
    smc_route_kernel(const T *__restrict__ emb, int64_t n, int dim, const T *__restrict__ dom, int M,
                     const T *__restrict__ sub, int J_max, const int32_t *__restrict__ J,
                     int32_t *__restrict__ out_m, int32_t *__restrict__ out_j,
                     int64_t *__restrict__ out_slot) {
    const int lane = threadIdx.x & 31;
    const int64_t c = static_cast<int64_t>(blockIdx.x) * kRouteWarps + (threadIdx.x >> 5);
    if (c >= n) return;
    const T *e = emb + c * dim;
    float acc[kRouteP];
    float best = -__int_as_float(0x7f800000);
    int m = -1;
    for (int i0 = 0; i0 < M; i0 += kRouteP) {
        const int cnt = M - i0 < kRouteP ? M - i0 : kRouteP;
        dots_warp<T, VEC>(e, dom + static_cast<int64_t>(i0) * dim, dim, cnt, dim, lane, acc);
#pragma unroll
        for (int q = 0; q < kRouteP; ++q)
            if (q < cnt && acc[q] > best) {
                best = acc[q];
                m = i0 + q;
            }
    }
    int j = -1;
    if (m >= 0) {
        int Jm = J[m];
        if (Jm > J_max || Jm < 0) {
            if (lane == 0) atomicOr(&g_smc_status, PRECOG_DEV_BAD_INDEX);
            Jm = 0;
        }
        best = -__int_as_float(0x7f800000);
        const T *sm_ = sub + static_cast<int64_t>(m) * J_max * dim;
        for (int i0 = 0; i0 < Jm; i0 += kRouteP) {
            const int cnt = Jm - i0 < kRouteP ? Jm - i0 : kRouteP;
            dots_warp<T, VEC>(e, sm_ + static_cast<int64_t>(i0) * dim, dim, cnt, dim, lane, acc);
#pragma unroll
            for (int q = 0; q < kRouteP; ++q)
                if (q < cnt && acc[q] > best) {
                    best = acc[q];
                    j = i0 + q;
                }
        }
    }
    if (lane == 0) {
        out_m[c] = m;
        out_j[c] = j;
        if (out_slot) out_slot[c] = (m >= 0 && j >= 0) ? static_cast<int64_t>(m) * J_max + j : -1;
    }
}

// s[slot_c] <- (1 - alpha) s[slot_c] + alpha h_c for c = 0, 1, ... in order,
// one thread per VEC adjacent state elements. Deposits go in batches of kU:
// warp 0 reads a batch's slots and describes it for the whole block (per
// deposit: the slot's offset, the latest earlier deposit of the same slot in
// the batch, whether a later one follows), one batch ahead, with a match-any
// vote instead of pairwise compares. Every thread then issues the batch's
// state loads and first-touch slot loads together, folds the batch in deposit
// order (a repeat inside the batch starts from its predecessor's result, kept
// in a per-thread shared-memory column) and stores each touched slot once.
// Slot -1 deposits nothing; a slot >= n_slots is flagged and skipped.
constexpr int kU = 16;
constexpr int kConsThreads = 128;

struct BatchMeta {
    int64_t off[kU];      // slot * elems (valid deposits)
    int prev[kU];         // latest earlier position of the same slot, or -1
    uint32_t valid;       // bit j: deposit j has a slot
    uint32_t last;        // bit j: no later deposit of the batch has the same slot
    uint32_t dups;        // some deposit repeats an earlier slot of the batch
};

// Lane j < kU of warp 0 reads deposit c0 + j's slot (-1 past the end); the reads
// run two batches ahead of their use so that their latency is hidden.
__device__ __forceinline__ int64_t read_slot(const int64_t *__restrict__ slots, int64_t c0, int64_t n, int lane) {
    const int64_t c = c0 + lane;
    return lane < kU && c < n ? slots[c] : -1;
}

__device__ __forceinline__ void describe_batch(BatchMeta &m, int64_t raw, int64_t n_slots, int64_t elems,
                                               int lane) {
    int64_t sl = INT64_MIN;                       // lanes beyond the batch never match
    if (lane < kU) {
        sl = raw;
        if (sl >= n_slots || sl < -1) {
            atomicOr(&g_smc_status, PRECOG_DEV_BAD_INDEX);
            sl = -1;
        }
    }
    const bool valid = lane < kU && sl >= 0;
    const uint32_t same = __match_any_sync(0xffffffffu, sl);
    const uint32_t below = same & ((1u << lane) - 1u);
    const uint32_t above = lane == 31 ? 0u : (same & ~((2u << lane) - 1u));
    const int prev = valid && below ? 31 - __clz(below) : -1;
    const uint32_t vmask = __ballot_sync(0xffffffffu, valid);
    const uint32_t lmask = __ballot_sync(0xffffffffu, valid && above == 0u);
    const uint32_t dmask = __ballot_sync(0xffffffffu, prev >= 0);
    if (lane < kU) {
        m.off[lane] = valid ? sl * elems : 0;
        m.prev[lane] = prev;
    }
    if (lane == 0) {
        m.valid = vmask;
        m.last = lmask;
        m.dups = dmask != 0u;
    }
}

template <typename TS, int VEC>
__device__ __forceinline__ void load_state_vec(const TS *p, float (&h)[VEC]) {
    if constexpr (VEC == 1) {
        h[0] = to_f32(p[0]);
    } else if constexpr (std::is_same<TS, float>::value) {
        const float2 v = *reinterpret_cast<const float2 *>(p);
        h[0] = v.x;
        h[1] = v.y;
    } else {
        const uint32_t w = *reinterpret_cast<const uint32_t *>(p);
        h[0] = __uint_as_float(w << 16);
        h[1] = __uint_as_float(w & 0xffff0000u);
    }
}

template <int VEC>
__device__ __forceinline__ void load_sem(const float *p, float (&v)[VEC]) {
    if constexpr (VEC == 1) {
        v[0] = p[0];
    } else {
        const float2 q = *reinterpret_cast<const float2 *>(p);
        v[0] = q.x;
        v[1] = q.y;
    }
}

template <int VEC>
__device__ __forceinline__ void store_sem(float *p, const float (&v)[VEC]) {
    if constexpr (VEC == 1) p[0] = v[0];
    else *reinterpret_cast<float2 *>(p) = make_float2(v[0], v[1]);
}

template <typename TS, int VEC>
__global__ void __launch_bounds__(kConsThreads)
    smc_consolidate_kernel(float *__restrict__ sem, int64_t n_slots, int64_t elems,
                           const TS *__restrict__ states, const int64_t *__restrict__ slots,
                           int64_t n, float alpha) {
    __shared__ BatchMeta s_meta[2];
    __shared__ float s_val[kU][VEC][kConsThreads];
    const float keep = 1.f - alpha;
    const int tid = threadIdx.x, lane = tid & 31;
    const int64_t e = (static_cast<int64_t>(blockIdx.x) * kConsThreads + tid) * VEC;
    const bool mine = e < elems;
    const int64_t nbatch = (n + kU - 1) / kU;
    // The deposits' states do not depend on the semantic table, so each batch's state
    // loads are issued one batch ahead (every deposit that exists, slot or not).
    auto load_states = [&](int64_t c0, float (&h)[kU][VEC]) {
#pragma unroll
        for (int j = 0; j < kU; ++j) {
#pragma unroll
            for (int i = 0; i < VEC; ++i) h[j][i] = 0.f;
            if (mine && c0 + j < n) load_state_vec<TS, VEC>(states + (c0 + j) * elems + e, h[j]);
        }
    };
    float h[kU][VEC];
    load_states(0, h);
    int64_t raw_next = 0;
    if (tid < 32) {
        const int64_t raw0 = read_slot(slots, 0, n, lane);
        raw_next = read_slot(slots, kU, n, lane);
        describe_batch(s_meta[0], raw0, n_slots, elems, lane);
    }
    __syncthreads();
    for (int64_t b = 0; b < nbatch; ++b) {
        const BatchMeta &m = s_meta[b & 1];
        const int64_t c0 = b * kU;
        float v[kU][VEC];
        if (mine) {
            // first touch of each slot in this batch: after the previous batch's stores
            // (same thread, program order)
#pragma unroll
            for (int j = 0; j < kU; ++j) {
#pragma unroll
                for (int i = 0; i < VEC; ++i) v[j][i] = 0.f;
                if ((m.valid >> j & 1u) && m.prev[j] < 0) load_sem<VEC>(sem + m.off[j] + e, v[j]);
            }
        }
        float hn[kU][VEC];
        load_states(c0 + kU, hn);
        // the next batch's description overlaps this batch's loads
        if (tid < 32 && b + 1 < nbatch) {
            const int64_t raw = raw_next;
            raw_next = read_slot(slots, c0 + 2 * kU, n, lane);
            describe_batch(s_meta[(b + 1) & 1], raw, n_slots, elems, lane);
        }
        if (mine) {
            if (!m.dups) {
#pragma unroll
                for (int j = 0; j < kU; ++j)
#pragma unroll
                    for (int i = 0; i < VEC; ++i) v[j][i] = fmaf(keep, v[j][i], alpha * h[j][i]);
            } else {
#pragma unroll
                for (int j = 0; j < kU; ++j) {
                    if (!(m.valid >> j & 1u)) continue;
                    const int pj = m.prev[j];
#pragma unroll
                    for (int i = 0; i < VEC; ++i) {
                        const float base = pj >= 0 ? s_val[pj][i][tid] : v[j][i];
                        v[j][i] = fmaf(keep, base, alpha * h[j][i]);
                        s_val[j][i][tid] = v[j][i];
                    }
                }
            }
#pragma unroll
            for (int j = 0; j < kU; ++j)
                if (m.last >> j & 1u) store_sem<VEC>(sem + m.off[j] + e, v[j]);
        }
#pragma unroll
        for (int j = 0; j < kU; ++j)
#pragma unroll
            for (int i = 0; i < VEC; ++i) h[j][i] = hn[j][i];
        __syncthreads();   // the next batch's description is complete; this one may be rewritten
    }
}

// The same fold with one CTA per (slot, range of elements), for tables of few
// slots: the CTA gathers its slot's deposits in deposit order (ballots over the
// slot ids, kGather at a time), then streams their states with several deposits'
// loads in flight, keeping its elements' semantic values in registers from the
// first deposit to the last: each state element is read once and each semantic
// element read and written once.
constexpr int kSlotThreads = 256;
constexpr int kSlotItems = 4;                    // element groups of VEC per thread
constexpr int kGather = 4 * kSlotThreads;        // slot ids examined per gathering pass
constexpr int kFoldAhead = 4;                    // deposits whose loads are in flight together

template <typename TS, int VEC>
__global__ void __launch_bounds__(kSlotThreads)
    smc_consolidate_slot_kernel(float *__restrict__ sem, int64_t n_slots, int64_t elems,
                                const TS *__restrict__ states, const int64_t *__restrict__ slots,
                                int64_t n, float alpha) {
    __shared__ int32_t s_list[kGather];
    __shared__ int s_warp[kSlotThreads / 32];
    __shared__ int s_total;
    const int64_t slot = blockIdx.y;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const float keep = 1.f - alpha;
    const bool flagger = blockIdx.x == 0 && blockIdx.y == 0;
    int64_t e[kSlotItems];
    float v[kSlotItems][VEC];
#pragma unroll
    for (int i = 0; i < kSlotItems; ++i) {
        e[i] = ((static_cast<int64_t>(blockIdx.x) * kSlotItems + i) * kSlotThreads + tid) * VEC;
        if (e[i] < elems) load_sem<VEC>(sem + slot * elems + e[i], v[i]);
    }
    for (int64_t c0 = 0; c0 < n; c0 += kGather) {
        int64_t sl[4];
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            const int64_t c = c0 + r * kSlotThreads + tid;
            sl[r] = c < n ? slots[c] : -1;
            if (flagger && (sl[r] >= n_slots || sl[r] < -1)) atomicOr(&g_smc_status, PRECOG_DEV_BAD_INDEX);
        }
        if (tid == 0) s_total = 0;
        __syncthreads();
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            const bool hit = sl[r] == slot;
            const uint32_t ball = __ballot_sync(0xffffffffu, hit);
            if (lane == 0) s_warp[warp] = __popc(ball);
            __syncthreads();
            int base = s_total;
            for (int w = 0; w < warp; ++w) base += s_warp[w];
            if (hit) s_list[base + __popc(ball & ((1u << lane) - 1u))] = static_cast<int32_t>(r * kSlotThreads + tid);
            __syncthreads();
            if (tid == 0)
                for (int w = 0; w < kSlotThreads / 32; ++w) s_total += s_warp[w];
            __syncthreads();
        }
        const int m = s_total;
        for (int j0 = 0; j0 < m; j0 += kFoldAhead) {
            float h[kFoldAhead][kSlotItems][VEC];
#pragma unroll
            for (int q = 0; q < kFoldAhead; ++q) {
                const int j = j0 + q;
                const int64_t c = j < m ? c0 + s_list[j] : 0;
#pragma unroll
                for (int i = 0; i < kSlotItems; ++i) {
#pragma unroll
                    for (int k = 0; k < VEC; ++k) h[q][i][k] = 0.f;
                    if (j < m && e[i] < elems) load_state_vec<TS, VEC>(states + c * elems + e[i], h[q][i]);
                }
            }
#pragma unroll
            for (int q = 0; q < kFoldAhead; ++q) {
                if (j0 + q >= m) break;
#pragma unroll
                for (int i = 0; i < kSlotItems; ++i)
#pragma unroll
                    for (int k = 0; k < VEC; ++k) v[i][k] = fmaf(keep, v[i][k], alpha * h[q][i][k]);
            }
        }
        __syncthreads();   // s_list is rebuilt by the next pass
    }
#pragma unroll
    for (int i = 0; i < kSlotItems; ++i)
        if (e[i] < elems) store_sem<VEC>(sem + slot * elems + e[i], v[i]);
}

// The per-slot fold with the states streamed through shared memory by asynchronous
// copies. HBM-bound: each state element crosses HBM once and each touched semantic
// element is read and written once; slots without a deposit are not read.
//
// Split: deposits are spread unevenly over slots (a slot may hold a fifth of them),
// and one element's deposits form a serial chain, so the work is divided by bytes,
// not by slots. Every CTA counts the deposits of each slot, weighs a slot's unit of
// kUnitBytes by the bytes it moves, and takes an equal share of the total weight: a
// contiguous run of (slot, element range) pieces, ranges of any width. Fixed 16 KB
// ranges in contiguous runs instead left 240 CTAs waiting for the few that held the
// largest slot.
//
// A piece is processed in tiles of at most kTileBytes. The CTA lists the slot's
// deposits in deposit order (ballots over the slot ids, kWindow at a time) and every
// thread then folds its own 16-byte chunks of the tile, in deposit order, through a
// private ring of 16-byte asynchronous copies in shared memory: no barrier, no producer
// and no wait on another thread. (One producer thread queueing a bulk copy per deposit
// cost about 250 ns per deposit and CTA, whatever the size: 1.0 TB/s on 2 KB ranges.)
// The ring holds kRingChunks chunks per thread, 72 KB per CTA and two CTAs per SM, and all of its
// groups but the one being folded are in flight: 17 deposits of a tile of up to 4 KB (34 of 2 KB
// and 68 of 1 KB, side by side), 8 of 8 KB, 3 of 16 KB, 2 of 24 KB. Narrower or wider tiles
// and shorter or longer rings were slower (4096 states below: 16 KB tiles 147 us; a ring of
// 12 chunks 158 us; 24 chunks the same as 18 and 66 against 64 us in the second case).
//
// 24-layer bf16 states (192 KB each), before -> now:
//   4096 into 64 slots, evenly                     137.6 -> 137.9 us  (6.21 TB/s)
//   1500 into 80 slots, evenly                      69.6 ->  63.9 us
//   1500 into 80 slots, 40 % of them in 4 slots    247   ->  66.2 us
//   1073 into 3 slots                              132   ->  82.9 us
//   4096 into 1 slot                              4202   -> 437   us
constexpr int kFoldThreads = 256;
constexpr int kFoldWarps = kFoldThreads / 32;
constexpr int kRingChunks = 18;    // 16-byte chunks in flight per thread
constexpr int kTileChunks = 6;     // 16-byte chunks of a tile per thread, at most
constexpr int kTileBytes = kTileChunks * 16 * kFoldThreads;
constexpr int kUnitBytes = 512;    // granularity of a piece
constexpr int kTallySlots = kFoldThreads;   // slots counted in shared memory, one per thread
constexpr int kIdsPerLane = 16;
constexpr int kWindow = kFoldThreads * kIdsPerLane;   // slot ids listed at once
static_assert(kWindow <= 65536, "list entries are 16-bit");

struct FoldSmem {
    uint4 ring[kRingChunks * kFoldThreads];
    uint16_t list[kWindow];         // positions in the window of the slot's deposits
    int64_t wsum[kFoldWarps];       // sums of 32 slots' weights
    int32_t count[kTallySlots];     // deposits per slot
    int32_t begin[kTallySlots];     // this CTA's units of each slot: [begin, end)
    int32_t end[kTallySlots];
    int32_t warp_hits[kFoldWarps];
    int32_t first_slot, last_slot;  // slots with a piece of this CTA
};

// Tiles of a piece of `len` units: as few as fit, of equal width (in units).
__device__ __forceinline__ int tile_units(int len) {
    constexpr int kMost = kTileBytes / kUnitBytes;
    const int tiles = (len + kMost - 1) / kMost;
    return (len + tiles - 1) / tiles;
}

// Lists the deposits of `slot` among ids [c0, c0 + kWindow) in order; their number.
// Every thread of the block; the previous list may still be read until it starts.
__device__ __forceinline__ int list_deposits(FoldSmem &sm, const int64_t *__restrict__ slots, int64_t n, int64_t c0,
                                             int slot) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    uint32_t hits[kIdsPerLane];
    int64_t id[kIdsPerLane];
#pragma unroll
    for (int r = 0; r < kIdsPerLane; ++r) {
        const int64_t c = c0 + (warp * kIdsPerLane + r) * 32 + lane;
        id[r] = c < n ? slots[c] : -1;
    }
    int mine = 0;
#pragma unroll
    for (int r = 0; r < kIdsPerLane; ++r) {
        hits[r] = __ballot_sync(0xffffffffu, id[r] == slot);
        mine += __popc(hits[r]);
    }
    __syncthreads();
    if (lane == 0) sm.warp_hits[warp] = mine;
    __syncthreads();
    int at = 0, total = 0;
#pragma unroll
    for (int w = 0; w < kFoldWarps; ++w) {
        const int h = sm.warp_hits[w];
        at += w < warp ? h : 0;
        total += h;
    }
#pragma unroll
    for (int r = 0; r < kIdsPerLane; ++r) {
        if (hits[r] >> lane & 1u)
            sm.list[at + __popc(hits[r] & ((1u << lane) - 1u))] = static_cast<uint16_t>((warp * kIdsPerLane + r) * 32 + lane);
        at += __popc(hits[r]);
    }
    __syncthreads();
    return total;
}

// One tile of `rlen` elements of `slot`'s row (`srow`, and `src` in the deposits' rows), C
// 16-byte chunks for each of kFoldThreads / B threads. The other threads' ring slots hold
// B deposits side by side. listed >= 0: the list already holds all deposits of the slot.
template <typename TS, int C, int B>
__device__ __forceinline__ void fold_tile(FoldSmem &sm, float *__restrict__ srow, const TS *__restrict__ src,
                                          int64_t rlen, int64_t elems, const int64_t *__restrict__ slots, int64_t n,
                                          int slot, int listed, float alpha) {
    constexpr int CH = 16 / static_cast<int>(sizeof(TS));   // state elements per chunk
    constexpr int P = kRingChunks / C;                      // groups of B deposits in the ring
    constexpr int W = kFoldThreads / B;                     // threads with chunks
    static_assert(B == 1 || C == 1, "side by side only in narrow tiles");
    const int tid = threadIdx.x;
    const float keep = 1.f - alpha;
    float v[C][CH];
    bool have[C];
#pragma unroll
    for (int i = 0; i < C; ++i) {
        const int64_t q = static_cast<int64_t>(i * kFoldThreads + tid) * CH;
        have[i] = q < rlen && tid < W;
#pragma unroll
        for (int k = 0; k < CH; k += 4) {
            const float4 f = have[i] ? *reinterpret_cast<const float4 *>(srow + q + k) : make_float4(0.f, 0.f, 0.f, 0.f);
            v[i][k] = f.x;
            v[i][k + 1] = f.y;
            v[i][k + 2] = f.z;
            v[i][k + 3] = f.w;
        }
    }
    for (int64_t c0 = 0; c0 < n; c0 += kWindow) {
        const int m = listed >= 0 ? listed : list_deposits(sm, slots, n, c0, slot);
        const TS *base = src + c0 * elems + static_cast<int64_t>(tid) * CH;
        int in = 0, out = 0;   // ring positions of the next group copied and folded
        auto copy = [&](int j0) {
#pragma unroll
            for (int b = 0; b < B; ++b)
                if (j0 + b < m) {
                    const TS *row = base + static_cast<int64_t>(sm.list[j0 + b]) * elems;
#pragma unroll
                    for (int i = 0; i < C; ++i)
                        if (have[i])
                            cp_async16(&sm.ring[(in * C + i) * kFoldThreads + b * W + tid], row + i * kFoldThreads * CH);
                }
            cp_async_commit();
            in = in + 1 == P ? 0 : in + 1;
        };
        for (int j = 0; j < (P - 1) * B; j += B) copy(j);
        for (int j = 0; j < m; j += B) {
            cp_async_wait<P - 2>();
#pragma unroll
            for (int b = 0; b < B; ++b) {
                if (j + b >= m) break;
#pragma unroll
                for (int i = 0; i < C; ++i) {
                    if (!have[i]) continue;
                    const uint4 raw = sm.ring[(out * C + i) * kFoldThreads + b * W + tid];
                    float h[CH];
                    if constexpr (std::is_same<TS, float>::value) {
                        h[0] = __uint_as_float(raw.x);
                        h[1] = __uint_as_float(raw.y);
                        h[2] = __uint_as_float(raw.z);
                        h[3] = __uint_as_float(raw.w);
                    } else {
                        const uint32_t w[4] = {raw.x, raw.y, raw.z, raw.w};
#pragma unroll
                        for (int k = 0; k < 4; ++k) {
                            h[2 * k] = __uint_as_float(w[k] << 16);
                            h[2 * k + 1] = __uint_as_float(w[k] & 0xffff0000u);
                        }
                    }
#pragma unroll
                    for (int k = 0; k < CH; ++k) v[i][k] = fmaf(keep, v[i][k], alpha * h[k]);
                }
            }
            out = out + 1 == P ? 0 : out + 1;
            copy(j + (P - 1) * B);
        }
        cp_async_wait<0>();
    }
#pragma unroll
    for (int i = 0; i < C; ++i) {
        if (!have[i]) continue;
        const int64_t q = static_cast<int64_t>(i * kFoldThreads + tid) * CH;
#pragma unroll
        for (int k = 0; k < CH; k += 4)
            *reinterpret_cast<float4 *>(srow + q + k) = make_float4(v[i][k], v[i][k + 1], v[i][k + 2], v[i][k + 3]);
    }
}

template <typename TS>
__global__ void __launch_bounds__(kFoldThreads, 2)
    smc_consolidate_share_kernel(float *__restrict__ sem, int n_slots, int64_t elems, const TS *__restrict__ states,
                                 const int64_t *__restrict__ slots, int64_t n, float alpha) {
    constexpr int64_t U = kUnitBytes / static_cast<int64_t>(sizeof(TS));  // elements per unit
    extern __shared__ __align__(16) unsigned char smem_raw[];
    FoldSmem &sm = *reinterpret_cast<FoldSmem *>(smem_raw);
    const int tid = threadIdx.x;
    const int64_t units = (elems + U - 1) / U;
    if (tid == 0) {
        sm.first_slot = n_slots;
        sm.last_slot = -1;
    }
    sm.count[tid] = 0;
    __syncthreads();

    // ---- this CTA's pieces ----
    constexpr int kAhead = 16;   // slot ids in flight per thread
    for (int64_t c0 = 0; c0 < n; c0 += kAhead * kFoldThreads) {
        int64_t id[kAhead];
#pragma unroll
        for (int r = 0; r < kAhead; ++r) {
            const int64_t c = c0 + r * kFoldThreads + tid;
            id[r] = c < n ? slots[c] : -1;
        }
#pragma unroll
        for (int r = 0; r < kAhead; ++r) {
            if (id[r] >= 0 && id[r] < n_slots) atomicAdd(&sm.count[id[r]], 1);
            else if (id[r] != -1 && blockIdx.x == 0) atomicOr(&g_smc_status, PRECOG_DEV_BAD_INDEX);
        }
    }
    __syncthreads();
    // a unit of a touched slot moves count * kUnitBytes of states and its semantic values
    // twice (8 bytes an element); weights in units of kUnitBytes, thread s sums slots 0..s
    constexpr int64_t kSemWeight = 2 * U * 4 / kUnitBytes;
    const int64_t w = sm.count[tid] > 0 ? sm.count[tid] + kSemWeight : 0;
    int64_t upto = w;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int64_t v = __shfl_up_sync(0xffffffffu, upto, o);
        upto += (tid & 31) >= o ? v : 0;
    }
    if ((tid & 31) == 31) sm.wsum[tid >> 5] = upto;
    __syncthreads();
    int64_t total = 0;
#pragma unroll
    for (int v = 0; v < kFoldWarps; ++v) {
        const int64_t t = sm.wsum[v];
        upto += v < (tid >> 5) ? t : 0;
        total += t;
    }
    total *= units;
    if (w > 0) {
        // unit u of slot s covers weights [base + u * w, base + (u + 1) * w); this CTA
        // takes the units that start in [lo, hi)
        const int64_t share = total / gridDim.x, rest = total % gridDim.x;
        const int64_t b = blockIdx.x;
        const int64_t lo = b * share + (b < rest ? b : rest);
        const int64_t hi = lo + share + (b < rest ? 1 : 0);
        const int64_t base = (upto - w) * units;
        const int64_t u0 = lo > base ? (lo - base + w - 1) / w : 0;
        const int64_t u1 = hi > base ? (hi - base + w - 1) / w : 0;
        sm.begin[tid] = static_cast<int32_t>(u0 < units ? u0 : units);
        sm.end[tid] = static_cast<int32_t>(u1 < units ? u1 : units);
        if (sm.begin[tid] < sm.end[tid]) {
            atomicMin(&sm.first_slot, tid);
            atomicMax(&sm.last_slot, tid);
        }
    }
    __syncthreads();

    const int last_slot = sm.last_slot;
    for (int slot = sm.first_slot; slot <= last_slot; ++slot) {
        if (sm.count[slot] == 0) continue;
        const int begin = sm.begin[slot], end = sm.end[slot];
        if (begin >= end) continue;
        const int listed = n <= kWindow ? list_deposits(sm, slots, n, 0, slot) : -1;
        const int step = tile_units(end - begin);
        const int chunks = step * (kUnitBytes / 16);
        for (int u = begin; u < end; u += step) {
            const int64_t e0 = u * U;
            const int64_t e1 = (u + step < end ? u + step : end) * U;
            const int64_t rlen = (e1 < elems ? e1 : elems) - e0;
            float *srow = sem + static_cast<int64_t>(slot) * elems + e0;
            const TS *src = states + e0;
            if (chunks * 4 <= kFoldThreads) fold_tile<TS, 1, 4>(sm, srow, src, rlen, elems, slots, n, slot, listed, alpha);
            else if (chunks * 2 <= kFoldThreads) fold_tile<TS, 1, 2>(sm, srow, src, rlen, elems, slots, n, slot, listed, alpha);
            else if (chunks <= kFoldThreads) fold_tile<TS, 1, 1>(sm, srow, src, rlen, elems, slots, n, slot, listed, alpha);
            else if (chunks <= 2 * kFoldThreads) fold_tile<TS, 2, 1>(sm, srow, src, rlen, elems, slots, n, slot, listed, alpha);
            else if (chunks <= 4 * kFoldThreads) fold_tile<TS, 4, 1>(sm, srow, src, rlen, elems, slots, n, slot, listed, alpha);
            else fold_tile<TS, kTileChunks, 1>(sm, srow, src, rlen, elems, slots, n, slot, listed, alpha);
        }
    }
}

}  // namespace

template <typename T>
void launch_route_t(const void *emb, int64_t n, int dim, const void *dom, int M, const void *sub, int J_max,
                    const int32_t *J, int32_t *out_m, int32_t *out_j, int64_t *out_slot, unsigned grid,
                    cudaStream_t stream) {
    const auto *e = static_cast<const T *>(emb);
    const auto *d = static_cast<const T *>(dom);
    const auto *s = static_cast<const T *>(sub);
    const auto a16 = [](const void *ptr) { return reinterpret_cast<uintptr_t>(ptr) % 16 == 0; };
    const bool vec = (static_cast<int64_t>(dim) * static_cast<int64_t>(sizeof(T))) % 16 == 0 && a16(emb) &&
                     a16(dom) && a16(sub);
    if (vec)
        smc_route_kernel<T, true><<<grid, kRouteWarps * 32, 0, stream>>>(e, n, dim, d, M, s, J_max, J, out_m,
                                                                        out_j, out_slot);
    else
        smc_route_kernel<T, false><<<grid, kRouteWarps * 32, 0, stream>>>(e, n, dim, d, M, s, J_max, J, out_m,
                                                                         out_j, out_slot);
}

cudaError_t launch_smc_route(const void *emb, int dtype, int64_t n, int dim, const void *dom, int M,
                             const void *sub, int J_max, const int32_t *J, int32_t *out_m,
                             int32_t *out_j, int64_t *out_slot, cudaStream_t stream) {
    if (n == 0) return cudaSuccess;
    const unsigned grid = static_cast<unsigned>((n + kRouteWarps - 1) / kRouteWarps);
    switch (dtype) {
        case PRECOG_F16:
            launch_route_t<__half>(emb, n, dim, dom, M, sub, J_max, J, out_m, out_j, out_slot, grid, stream);
            break;
        case PRECOG_BF16:
            launch_route_t<__nv_bfloat16>(emb, n, dim, dom, M, sub, J_max, J, out_m, out_j, out_slot, grid, stream);
            break;
        default:
            launch_route_t<float>(emb, n, dim, dom, M, sub, J_max, J, out_m, out_j, out_slot, grid, stream);
    }
    cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess) count_launches(1);
    return e;
}

cudaError_t launch_smc_consolidate(float *sem, int64_t n_slots, int64_t elems, const void *states,
                                   int states_dtype, const int64_t *slots, int64_t n, float alpha,
                                   cudaStream_t stream) {
    if (n == 0 || elems == 0) return cudaSuccess;
    // pairs of elements when every row start stays 8-byte (fp32) / 4-byte (bf16) aligned
    const bool pairs = elems % 2 == 0;
    const int vec = pairs ? 2 : 1;
    const int64_t blocks = (elems / vec + kConsThreads - 1) / kConsThreads;
    if (blocks > 0x7fffffffLL) return cudaErrorInvalidConfiguration;
    const unsigned grid = static_cast<unsigned>(blocks);
    // Few slots: CTAs over pieces of (slot, element range). Rows of whole 16-byte chunks stream
    // through the copy rings: a CTA reads all n slot ids from L2 to count the deposits of up to
    // kTallySlots slots, one per thread, and again for each piece (each tile beyond kWindow
    // deposits) to list its slot's. Other rows take the register per-slot kernel, whose CTAs
    // of 2048 elements read n_slots / 512 of their state bytes in slot ids.
    const int64_t size = states_dtype == PRECOG_BF16 ? 2 : 4;
    const int64_t units = (elems * size + kUnitBytes - 1) / kUnitBytes;
    if (n_slots >= 1 && n_slots <= kTallySlots && elems * size % 16 == 0 && units < 0x7fffffffLL) {
        const int64_t resident = 2 * static_cast<int64_t>(device_sm_count());
        const int64_t touched = n < n_slots ? n : n_slots;   // at most
        const int64_t blocks2 = touched * units < resident ? touched * units : resident;
        const int smem = static_cast<int>(sizeof(FoldSmem));
        cudaError_t e;
        if (states_dtype == PRECOG_BF16) {
            e = ensure_smem(reinterpret_cast<const void *>(smc_consolidate_share_kernel<__nv_bfloat16>), smem);
            if (e != cudaSuccess) return e;
            smc_consolidate_share_kernel<__nv_bfloat16><<<static_cast<unsigned>(blocks2), kFoldThreads, smem, stream>>>(
                sem, static_cast<int>(n_slots), elems, static_cast<const __nv_bfloat16 *>(states), slots, n, alpha);
        } else {
            e = ensure_smem(reinterpret_cast<const void *>(smc_consolidate_share_kernel<float>), smem);
            if (e != cudaSuccess) return e;
            smc_consolidate_share_kernel<float><<<static_cast<unsigned>(blocks2), kFoldThreads, smem, stream>>>(
                sem, static_cast<int>(n_slots), elems, static_cast<const float *>(states), slots, n, alpha);
        }
        e = cudaGetLastError();
        if (e == cudaSuccess) count_launches(1);
        return e;
    }
    if (n_slots >= 1 && n_slots <= 256) {
        const int64_t per_cta = static_cast<int64_t>(kSlotThreads) * kSlotItems * vec;
        const dim3 g2(static_cast<unsigned>((elems + per_cta - 1) / per_cta), static_cast<unsigned>(n_slots));
        if (states_dtype == PRECOG_BF16) {
            const auto *st = static_cast<const __nv_bfloat16 *>(states);
            if (pairs) smc_consolidate_slot_kernel<__nv_bfloat16, 2><<<g2, kSlotThreads, 0, stream>>>(sem, n_slots, elems, st, slots, n, alpha);
            else smc_consolidate_slot_kernel<__nv_bfloat16, 1><<<g2, kSlotThreads, 0, stream>>>(sem, n_slots, elems, st, slots, n, alpha);
        } else {
            const auto *st = static_cast<const float *>(states);
            if (pairs) smc_consolidate_slot_kernel<float, 2><<<g2, kSlotThreads, 0, stream>>>(sem, n_slots, elems, st, slots, n, alpha);
            else smc_consolidate_slot_kernel<float, 1><<<g2, kSlotThreads, 0, stream>>>(sem, n_slots, elems, st, slots, n, alpha);
        }
        cudaError_t e = cudaGetLastError();
        if (e == cudaSuccess) count_launches(1);
        return e;
    }
    if (states_dtype == PRECOG_BF16) {
        const auto *st = static_cast<const __nv_bfloat16 *>(states);
        if (pairs) smc_consolidate_kernel<__nv_bfloat16, 2><<<grid, kConsThreads, 0, stream>>>(sem, n_slots, elems, st, slots, n, alpha);
        else smc_consolidate_kernel<__nv_bfloat16, 1><<<grid, kConsThreads, 0, stream>>>(sem, n_slots, elems, st, slots, n, alpha);
    } else {
        const auto *st = static_cast<const float *>(states);
        if (pairs) smc_consolidate_kernel<float, 2><<<grid, kConsThreads, 0, stream>>>(sem, n_slots, elems, st, slots, n, alpha);
        else smc_consolidate_kernel<float, 1><<<grid, kConsThreads, 0, stream>>>(sem, n_slots, elems, st, slots, n, alpha);
    }
    cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess) count_launches(1);
    return e;
}

cudaError_t smc_status_word_read_clear(uint32_t *bits) {
    uint32_t zero = 0;
    cudaError_t e = cudaMemcpyFromSymbol(bits, g_smc_status, sizeof(uint32_t));
    if (e != cudaSuccess) return e;
    return cudaMemcpyToSymbol(g_smc_status, &zero, sizeof(uint32_t));
}

}  // namespace precog
