// Exact top-1 dot-product retrieval over a flat key index (Sec. 4.2).
//
// fp32 keys, on the CUDA cores (16-bit keys: retrieve_tc.cu). Batches share each row among
// the warps of a CTA (gemm_retrieve_kernel below). The GEMV kernels take a single query's short
// rows and the longest rows: every warp streams whole key rows with
// 16-byte loads (several rows in flight per warp), dots them with a group of
// up to kQB queries held in registers as fp32, and reduces across lanes with
// a fixed butterfly, so a row's score never depends on where the row sits:
// equal rows get equal scores and the lowest row wins a tie. Each
// (score, row) pair is packed into one 64-bit key ordered by score, then by
// lower row; per-CTA maxima go to the workspace and a finalize kernel reduces
// them. A NaN score never enters a key, so it never wins.
#include <algorithm>
#include <type_traits>

#include "../../include/precog.h"
#include "internal.h"
#include "ptx.cuh"

namespace precog {
namespace {

__device__ uint32_t g_retrieve_status;

constexpr int kThreads = 256;
constexpr int kWarps = kThreads / 32;
constexpr int kQB = 4;        // queries per pass over the index
constexpr int kMaxVecsPerRow = 512;  // 16 vectors per lane

// Monotone map of a non-NaN fp32 score to uint32 (-inf -> 0x007fffff > 0).
__device__ __forceinline__ uint32_t ordered_bits(float s) {
    const uint32_t u = __float_as_uint(s + 0.0f);  // -0 -> +0: equal scores, equal keys
    return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}
__device__ __forceinline__ float unordered_float(uint32_t k) {
    return __uint_as_float((k & 0x80000000u) ? (k & 0x7fffffffu) : ~k);
}
// Larger key = higher score, then lower row. Key 0 = "no row".
__device__ __forceinline__ unsigned long long make_key(float s, int64_t row) {
    return (static_cast<unsigned long long>(ordered_bits(s)) << 32) |
           static_cast<unsigned long long>(0xffffffffu - static_cast<uint32_t>(row));
}

// The CUDA-core kernels take fp32 keys (16-bit keys go to the tensor cores).
template <typename T> struct Vec;
template <> struct Vec<float> { static constexpr int n = 4; };

// The products of one 16-byte vector of a row with a query's, and a lane's sum of them. Every
// fp32 kernel sums a row in this order (a lane's vectors l, l+32, ... with even and odd elements
// apart, then the lanes' sums over xor distances 16, 8, 4, 2, 1), so that a score does not depend
// on the kernel that the number of queries or k selects.
__device__ __forceinline__ void dot_step(f2 &acc, const ulonglong2 &x, const f2 (&q)[2]) {
    acc = fma2(x.x, q[0], acc);
    acc = fma2(x.y, q[1], acc);
}
__device__ __forceinline__ float dot_sum(f2 acc) {
    float lo, hi;
    unpack2(acc, lo, hi);
    return lo + hi;
}
// Vector v of a row of floats (zeros where it is not to be read).
__device__ __forceinline__ ulonglong2 load_vec(const float *row, int v, bool in) {
    return in ? __ldg(reinterpret_cast<const ulonglong2 *>(row) + v) : make_ulonglong2(0ull, 0ull);
}

// partial[blockIdx.x * n_queries + q] = best key of this CTA for query q.
// Lane l owns the 16-byte vectors l, l+32, ... of every row (VPL of them) and
// holds the matching query values in registers; RIF rows are loaded before any
// is used, so each lane keeps RIF*VPL 16-byte loads in flight.
// Two vectors per lane keep four CTAs per SM (200,000 x 256 keys 37 us; 78 registers, three: 45).
template <typename T, int QB, int VPL, int RIF>
__global__ void __launch_bounds__(kThreads, QB == 1 && VPL == 2 ? 4 : 1)
    gemv_top1_kernel(const T *__restrict__ index, int64_t M, int dim, const T *__restrict__ queries,
                     int n_queries, int q0, unsigned long long *__restrict__ partial) {
    constexpr int V = Vec<T>::n;
    __shared__ unsigned long long best[QB];
    const int nq = min(QB, n_queries - q0);
    const int lane = threadIdx.x & 31;
    const int warp = threadIdx.x >> 5;
    const int vecs = dim / V;
    f2 qv[QB][VPL][2];
#pragma unroll
    for (int qq = 0; qq < QB; ++qq)
#pragma unroll
        for (int j = 0; j < VPL; ++j) {
            const int v = lane + 32 * j;
            const ulonglong2 raw = load_vec(queries + static_cast<int64_t>(q0 + qq) * dim, v, qq < nq && v < vecs);
            qv[qq][j][0] = raw.x;
            qv[qq][j][1] = raw.y;
        }
    if (threadIdx.x < QB) best[threadIdx.x] = 0ull;
    __syncthreads();

    const int64_t gwarp = static_cast<int64_t>(blockIdx.x) * kWarps + warp;
    const int64_t nwarps = static_cast<int64_t>(gridDim.x) * kWarps;
    unsigned long long mykey[QB];
#pragma unroll
    for (int qq = 0; qq < QB; ++qq) mykey[qq] = 0ull;

    for (int64_t r0 = gwarp * RIF; r0 < M; r0 += nwarps * RIF) {
        ulonglong2 raw[RIF][VPL];
#pragma unroll
        for (int r = 0; r < RIF; ++r)
#pragma unroll
            for (int j = 0; j < VPL; ++j) {
                const int v = lane + 32 * j;
                const int64_t row = r0 + r;
                raw[r][j] = load_vec(index + row * dim, v, v < vecs && row < M);
            }
#pragma unroll
        for (int r = 0; r < RIF; ++r) {
            f2 acc[QB];
#pragma unroll
            for (int qq = 0; qq < QB; ++qq) acc[qq] = 0;
#pragma unroll
            for (int j = 0; j < VPL; ++j)
#pragma unroll
                for (int qq = 0; qq < QB; ++qq) dot_step(acc[qq], raw[r][j], qv[qq][j]);
            const int64_t row = r0 + r;
#pragma unroll
            for (int qq = 0; qq < QB; ++qq) {
                float sc = dot_sum(acc[qq]);
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) sc += __shfl_xor_sync(0xffffffffu, sc, o);
                if (row < M && !isnan(sc)) {
                    const unsigned long long key = make_key(sc, row);
                    mykey[qq] = key > mykey[qq] ? key : mykey[qq];
                }
            }
        }
    }
    if (lane == 0)
        for (int qq = 0; qq < nq; ++qq) atomicMax(&best[qq], mykey[qq]);
    __syncthreads();
    if (threadIdx.x < nq)
        partial[static_cast<int64_t>(blockIdx.x) * n_queries + q0 + threadIdx.x] = best[threadIdx.x];
}

__device__ __forceinline__ unsigned long long shfl_xor_u64(unsigned long long v, int o) {
    const uint32_t lo = __shfl_xor_sync(0xffffffffu, static_cast<uint32_t>(v), o);
    const uint32_t hi = __shfl_xor_sync(0xffffffffu, static_cast<uint32_t>(v >> 32), o);
    return (static_cast<unsigned long long>(hi) << 32) | lo;
}

// A shard's key with its row made global, in signed order: flipping the top bit
// maps the unsigned key order onto int64 order, so keys of different shards combine
// by a signed maximum (an all-reduce MAX over int64); "no row" becomes INT64_MIN.
__device__ __forceinline__ int64_t global_key(unsigned long long k, int64_t row_offset) {
    if (k != 0ull) {
        const int64_t row = row_offset + static_cast<int64_t>(0xffffffffu - static_cast<uint32_t>(k & 0xffffffffu));
        k = (k & 0xffffffff00000000ull) | static_cast<unsigned long long>(0xffffffffu - static_cast<uint32_t>(row));
    }
    return static_cast<int64_t>(k ^ 0x8000000000000000ull);
}

__device__ __forceinline__ void write_best(unsigned long long k, int64_t *best_idx, float *best_score, int64_t q) {
    if (k == 0ull) {
        best_idx[q] = -1;
        if (best_score) best_score[q] = __uint_as_float(0x7fc00000u);
    } else {
        best_idx[q] = static_cast<int64_t>(0xffffffffu - static_cast<uint32_t>(k & 0xffffffffu));
        if (best_score) best_score[q] = unordered_float(static_cast<uint32_t>(k >> 32));
    }
}

// One warp per query: each lane takes the maximum over a strided share of the
// per-CTA keys (independent loads, so many are in flight), then a butterfly.
__global__ void finalize_kernel(const unsigned long long *__restrict__ partial, int n_parts,
                                int n_queries, int64_t *__restrict__ best_idx,
                                float *__restrict__ best_score, int64_t row_offset,
                                int64_t *__restrict__ keys_out) {
    grid_dependency_wait();
    grid_dependency_launch();   // a prefill from the retrieved rows
    const int q = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (q >= n_queries) return;
    unsigned long long k = 0ull;
    for (int i = lane; i < n_parts; i += 32) {
        const unsigned long long v = partial[static_cast<int64_t>(i) * n_queries + q];
        k = v > k ? v : k;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const unsigned long long v = shfl_xor_u64(k, o);
        k = v > k ? v : k;
    }
    if (lane != 0) return;
    if (keys_out) keys_out[q] = global_key(k, row_offset);
    else write_best(k, best_idx, best_score, q);
}

// Signed-order keys (combined over shards) to rows and scores.
__global__ void decode_keys_kernel(const int64_t *__restrict__ keys, int n, int64_t *__restrict__ best_idx,
                                   float *__restrict__ best_score) {
    const int q = blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= n) return;
    write_best(static_cast<unsigned long long>(keys[q]) ^ 0x8000000000000000ull, best_idx, best_score, q);
}

// ---------------------------------------------------------------------------
// Top-k (k <= kListK) for one query per pass: every warp keeps the kListK best
// packed keys seen so far as a sorted list, held identically by all lanes (the
// butterfly leaves the row's score in every lane), so a row costs one compare
// against the list's last entry unless it enters the list. The warps' lists
// are merged per CTA in shared memory; partial[(cta * Q + q) * kListK + j].
constexpr int kListK = 8;

__device__ __forceinline__ void list_insert(unsigned long long (&l)[kListK], unsigned long long v) {
    if (v <= l[kListK - 1]) return;
#pragma unroll
    for (int j = kListK - 1; j > 0; --j) {
        // shift entries below v down by one; v lands in its sorted slot
        const bool shift = v > l[j - 1];
        l[j] = shift ? l[j - 1] : (v > l[j] ? v : l[j]);
    }
    l[0] = v > l[0] ? v : l[0];
}

template <typename T, int VPL>
__global__ void __launch_bounds__(kThreads)
    gemv_topk_kernel(const T *__restrict__ index, int64_t M, int dim, const T *__restrict__ queries,
                     int n_queries, int q, unsigned long long *__restrict__ partial) {
    constexpr int V = Vec<T>::n;
    constexpr int RIF = 4;
    __shared__ unsigned long long lists[kWarps][kListK];
    const int lane = threadIdx.x & 31;
    const int warp = threadIdx.x >> 5;
    const int vecs = dim / V;
    f2 qv[VPL][2];
#pragma unroll
    for (int j = 0; j < VPL; ++j) {
        const int v = lane + 32 * j;
        const ulonglong2 raw = load_vec(queries + static_cast<int64_t>(q) * dim, v, v < vecs);
        qv[j][0] = raw.x;
        qv[j][1] = raw.y;
    }
    unsigned long long l[kListK];
#pragma unroll
    for (int j = 0; j < kListK; ++j) l[j] = 0ull;
    const int64_t gwarp = static_cast<int64_t>(blockIdx.x) * kWarps + warp;
    const int64_t nwarps = static_cast<int64_t>(gridDim.x) * kWarps;
    for (int64_t r0 = gwarp * RIF; r0 < M; r0 += nwarps * RIF) {
        ulonglong2 raw[RIF][VPL];
#pragma unroll
        for (int r = 0; r < RIF; ++r)
#pragma unroll
            for (int j = 0; j < VPL; ++j) {
                const int v = lane + 32 * j;
                const int64_t row = r0 + r;
                raw[r][j] = load_vec(index + row * dim, v, v < vecs && row < M);
            }
#pragma unroll
        for (int r = 0; r < RIF; ++r) {
            f2 sums = 0;
#pragma unroll
            for (int j = 0; j < VPL; ++j) dot_step(sums, raw[r][j], qv[j]);
            float acc = dot_sum(sums);
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
            const int64_t row = r0 + r;
            // acc is the same in every lane (xor butterfly), so the branch is uniform;
            // most rows fall below the list's last key and skip the insertion
            if (row < M && !isnan(acc)) {
                const unsigned long long key = make_key(acc, row);
                if (key > l[kListK - 1]) list_insert(l, key);
            }
        }
    }
    if (lane == 0)
#pragma unroll
        for (int j = 0; j < kListK; ++j) lists[warp][j] = l[j];
    __syncthreads();
    if (threadIdx.x == 0) {
        unsigned long long m[kListK];
#pragma unroll
        for (int j = 0; j < kListK; ++j) m[j] = lists[0][j];
        for (int w = 1; w < kWarps; ++w)
#pragma unroll
            for (int j = 0; j < kListK; ++j) list_insert(m, lists[w][j]);
#pragma unroll
        for (int j = 0; j < kListK; ++j)
            partial[(static_cast<int64_t>(blockIdx.x) * n_queries + q) * kListK + j] = m[j];
    }
}

__device__ __forceinline__ unsigned long long warp_max_u64(unsigned long long v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const unsigned long long w = shfl_xor_u64(v, o);
        v = w > v ? w : v;
    }
    return v;
}

// Merge the per-CTA lists of one query into its k best, one warp per query. The lists'
// 2^log_used leading entries (of kListK) are spread over the lanes, kAhead independent
// loads at a time. The k-th largest of the lanes' largest heads bounds the k-th best from
// below, so few entries reach a lane's sorted list; then k rounds take the warp's largest
// head (keys are unique, so one lane owns it and drops it). One list per lane with
// dependent loads, merged by butterflies, took 25 us for 608 parts.
__global__ void finalize_topk_kernel(const unsigned long long *__restrict__ partial, int n_parts, int log_used,
                                     int n_queries, int k, int64_t *__restrict__ best_idx,
                                     float *__restrict__ best_score) {
    grid_dependency_wait();
    grid_dependency_launch();   // a prefill from the retrieved rows
    constexpr int kAhead = 8;
    const int q = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (q >= n_queries) return;
    auto entry = [&](int part, int j) {
        return partial[(static_cast<int64_t>(part) * n_queries + q) * kListK + j];
    };
    unsigned long long head = 0ull;
    for (int i0 = lane; i0 < n_parts; i0 += 32 * kAhead) {
        unsigned long long v[kAhead];
#pragma unroll
        for (int r = 0; r < kAhead; ++r) v[r] = i0 + 32 * r < n_parts ? entry(i0 + 32 * r, 0) : 0ull;
#pragma unroll
        for (int r = 0; r < kAhead; ++r) head = v[r] > head ? v[r] : head;
    }
    unsigned long long least = 0ull;
    for (int j = 0; j < k; ++j) {
        least = warp_max_u64(head);
        if (head == least) head = 0ull;
    }
    unsigned long long l[kListK];
#pragma unroll
    for (int j = 0; j < kListK; ++j) l[j] = 0ull;
    const int total = n_parts << log_used, mask = (1 << log_used) - 1;
    for (int i0 = lane; i0 < total; i0 += 32 * kAhead) {
        unsigned long long v[kAhead];
#pragma unroll
        for (int r = 0; r < kAhead; ++r) {
            const int i = i0 + 32 * r;
            v[r] = i < total ? entry(i >> log_used, i & mask) : 0ull;
        }
#pragma unroll
        for (int r = 0; r < kAhead; ++r)
            if (v[r] >= least) list_insert(l, v[r]);
    }
    for (int j = 0; j < k; ++j) {
        const unsigned long long key = warp_max_u64(l[0]);
        if (key != 0ull && key == l[0]) {
#pragma unroll
            for (int i = 0; i + 1 < kListK; ++i) l[i] = l[i + 1];
            l[kListK - 1] = 0ull;
        }
        if (lane == 0) write_best(key, best_idx, best_score, static_cast<int64_t>(q) * k + j);
    }
}

// ---------------------------------------------------------------------------
// Batches over an fp32 index: one pass over the keys for up to kGemmWarps * QW queries.
//
// fp32 scores stay on the FMA pipe (the tensor cores would round the keys). A pass per 4
// queries (top-1) or per query (top-k) re-read the index once per pass; here a CTA streams
// tiles of whole key rows through a shared-memory ring (one bulk copy per tile, the rows
// being contiguous) and its kGemmWarps warps share them: WQ groups of QW queries times WR
// shares of the tile's row pairs. A lane owns the 16-byte vectors l, l+32, ... of a row, as
// in the GEMV, with its QW queries' values in registers, so a row costs VPL 16-byte
// shared-memory reads per QW * VPL * 4 multiply-adds (packed, adjacent dims in the halves);
// with QW = 8 shared memory is half as busy as the FMA pipe, with QW = 4 (rows over 384
// dims: the query registers) as busy. The 2 * QW sums of a row pair are added across the
// lanes by halving exchanges (each step sends the half of the sums that the other lane
// keeps): 16 exchanges for 16 sums where separate butterflies take 80, in the same tree for
// every row, so equal rows score equally. Bound: HBM up to about 8 queries, then the FMA
// pipe (59 % busy: three warps per scheduler, exchanges and key updates between the sums).
// Top-1 / top-3, us, before (a pass per 4 queries / per query) -> now:
//   8 queries, 50,021 x 384      53 / 170 ->  24 /  24   (77 MB: 11 us)
//   23                          144 / 449 ->  38 /  42
//   256                        1453 / 4750 -> 301 / 308   (9.8 GFLOP: 122 us)
//   8 queries, 500,000 x 384    419 / 1033 -> 136 / 143   (768 MB: 113 us)
//   8 queries, 300,000 x 768    608 / 1347 -> 158 / 164   (922 MB: 136 us)
constexpr int kGemmWarps = 12;
constexpr int kGemmThreads = kGemmWarps * 32;
constexpr int kGemmStages = 4;
constexpr int kGemmMaxDim = 1024;
constexpr int kGemmStageBytes = 49152;   // at least 24 rows of up to 512 dims, 12 of up to 1024

struct GemmSmem {
    alignas(128) unsigned char ring[kGemmStages][kGemmStageBytes];
    uint64_t full[kGemmStages];
    uint64_t empty[kGemmStages];
    unsigned long long best[kGemmWarps * 8];
};

template <int LIST>
__device__ __forceinline__ void insert_key(unsigned long long (&l)[LIST], unsigned long long v) {
    if (v <= l[LIST - 1]) return;
#pragma unroll
    for (int j = LIST - 1; j > 0; --j) {
        const bool shift = v > l[j - 1];
        l[j] = shift ? l[j - 1] : (v > l[j] ? v : l[j]);
    }
    l[0] = v > l[0] ? v : l[0];
}

// LIST = 1: partial[blockIdx.x * n_queries + q] = best key of this CTA's rows; else the
// LIST best, sorted, in the first LIST of kListK entries of partial[(blockIdx.x *
// n_queries + q) * kListK]. Pass y0 + blockIdx.y takes WQ * QW queries.
template <int VPL, int QW, int LIST>
__global__ void __launch_bounds__(kGemmThreads, 1)
    gemm_retrieve_kernel(const float *__restrict__ index, int64_t M, int dim, const float *__restrict__ queries,
                         int n_queries, int TR, int WQ, int y0, unsigned long long *__restrict__ partial) {
    constexpr int NC = 2 * QW;   // sums of a row pair
    extern __shared__ __align__(128) unsigned char smem_raw[];
    GemmSmem &sm = *reinterpret_cast<GemmSmem *>(smem_raw);
    const int lane = threadIdx.x & 31;
    const int warp = threadIdx.x >> 5;
    const int WR = kGemmWarps / WQ;
    const int wq = warp % WQ, wr = warp / WQ;
    const int q0 = (y0 + static_cast<int>(blockIdx.y)) * WQ * QW;   // first query of the pass
    const int vecs = dim / 4;
    const int64_t ntiles = (M + TR - 1) / TR;
    const int64_t first = blockIdx.x, step = gridDim.x;

    if (threadIdx.x == 0) {
        for (int s = 0; s < kGemmStages; ++s) {
            mbar_init(&sm.full[s], 1);
            mbar_init(&sm.empty[s], kGemmWarps);
        }
        fence_barrier_init();
    }
    if (threadIdx.x < kGemmWarps * 8) sm.best[threadIdx.x] = 0ull;
    __syncthreads();
    auto issue = [&](int64_t k) {   // one thread: this CTA's k-th tile
        const int64_t r0 = (first + k * step) * TR;
        const int64_t rows = M - r0 < TR ? M - r0 : TR;
        const uint32_t bytes = static_cast<uint32_t>(rows * dim * 4);
        const int s = static_cast<int>(k % kGemmStages);
        mbar_arrive_expect_tx(&sm.full[s], bytes);
        bulk_g2s(sm.ring[s], index + r0 * dim, bytes, &sm.full[s]);
    };
    const int64_t mine = first < ntiles ? (ntiles - first + step - 1) / step : 0;
    int64_t issued = 0;
    for (; warp == 0 && issued < kGemmStages && issued < mine; ++issued)
        if (lane == 0) issue(issued);

    f2 qv[QW][VPL][2];
#pragma unroll
    for (int i = 0; i < QW; ++i)
#pragma unroll
        for (int j = 0; j < VPL; ++j) {
            const int v = lane + 32 * j, q = q0 + wq * QW + i;
            const bool in = v < vecs && q < n_queries;
            const ulonglong2 raw =
                in ? __ldg(reinterpret_cast<const ulonglong2 *>(queries + static_cast<int64_t>(q) * dim) + v)
                   : make_ulonglong2(0ull, 0ull);
            qv[i][j][0] = raw.x;
            qv[i][j][1] = raw.y;
        }
    // the sum that this lane ends up with: bit b of the sum's index is lane bit 4 - b
    int sum = 0;
#pragma unroll
    for (int h = NC / 2, o = 16; h > 0; h >>= 1, o >>= 1) sum += (lane & o) ? h : 0;
    const int sum_r = sum / QW;
    unsigned long long l[LIST];
#pragma unroll
    for (int j = 0; j < LIST; ++j) l[j] = 0ull;

    bool ok = true;
    for (int64_t k = 0; k < mine; ++k) {
        const int s = static_cast<int>(k % kGemmStages);
        ok = __all_sync(0xffffffffu, mbar_wait(&sm.full[s], static_cast<uint32_t>((k / kGemmStages) & 1)));
        if (!ok) break;
        const int64_t r0 = (first + k * step) * TR;
        const int rows = static_cast<int>(M - r0 < TR ? M - r0 : TR);
        const unsigned char *tile = sm.ring[s];
        for (int p = wr; 2 * p < rows; p += WR) {
            float a[NC];
#pragma unroll
            for (int r = 0; r < 2; ++r) {
                // an odd tile's last pair reads its row twice; the second sum is dropped
                const int row = 2 * p + r < rows ? 2 * p + r : 2 * p;
                const ulonglong2 *src = reinterpret_cast<const ulonglong2 *>(tile + static_cast<size_t>(row) * dim * 4);
                f2 acc[QW];
#pragma unroll
                for (int i = 0; i < QW; ++i) acc[i] = 0;
#pragma unroll
                for (int j = 0; j < VPL; ++j) {
                    const int v = lane + 32 * j;
                    const ulonglong2 x = v < vecs ? src[v] : make_ulonglong2(0ull, 0ull);
#pragma unroll
                    for (int i = 0; i < QW; ++i) dot_step(acc[i], x, qv[i][j]);
                }
#pragma unroll
                for (int i = 0; i < QW; ++i) a[r * QW + i] = dot_sum(acc[i]);
            }
            int o = 16;
#pragma unroll
            for (int h = NC / 2; h > 0; h >>= 1, o >>= 1) {
                const bool up = (lane & o) != 0;
#pragma unroll
                for (int i = 0; i < h; ++i) {
                    const float keep = up ? a[i + h] : a[i], send = up ? a[i] : a[i + h];
                    a[i] = keep + __shfl_xor_sync(0xffffffffu, send, o);
                }
            }
#pragma unroll
            for (int b = 0; b < 5; ++b)
                if ((16 >> b) <= 16 / NC) a[0] += __shfl_xor_sync(0xffffffffu, a[0], 16 >> b);
            const int64_t row = r0 + 2 * p + sum_r;
            if (2 * p + sum_r < rows && !isnan(a[0])) insert_key<LIST>(l, make_key(a[0], row));
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(&sm.empty[s]);
        // warp 0 refills the stage of the tile before this one: the other warps are done with
        // it or nearly (the whole warp leaves together when a wait runs out)
        if (warp == 0 && k > 0 && issued < mine) {
            const int64_t f = issued - kGemmStages;   // tile k - 1
            ok = __all_sync(0xffffffffu, mbar_wait(&sm.empty[f % kGemmStages], static_cast<uint32_t>((f / kGemmStages) & 1)));
            if (!ok) break;
            if (lane == 0) {
                fence_proxy_async_smem();
                issue(issued);
            }
            ++issued;
        }
    }
    if (!ok) atomicOr(&g_retrieve_status, PRECOG_DEV_TIMEOUT);
    if (threadIdx.x == 0 && !ok)   // issued copies land before the CTA leaves
        for (int64_t f = issued > kGemmStages ? issued - kGemmStages : 0; f < issued; ++f)
            mbar_wait(&sm.full[f % kGemmStages], static_cast<uint32_t>((f / kGemmStages) & 1));
    __syncthreads();
    const bool keeper = (lane & (32 / NC - 1)) == 0;   // one of the lanes that hold the same sum
    if constexpr (LIST == 1) {
        if (keeper && l[0] != 0ull) atomicMax(&sm.best[wq * QW + sum % QW], l[0]);
        __syncthreads();
        const int q = q0 + static_cast<int>(threadIdx.x);
        if (static_cast<int>(threadIdx.x) < WQ * QW && q < n_queries)
            partial[static_cast<int64_t>(blockIdx.x) * n_queries + q] = sm.best[threadIdx.x];
    } else {
        // lists[query][row share and parity][LIST] in the ring, merged by one warp per query (a
        // lane per list, the largest head LIST times) when they are many, else by one thread
        constexpr int kWritten = LIST <= 4 ? 4 : kListK;   // entries that the finalize reads
        unsigned long long *lists = reinterpret_cast<unsigned long long *>(sm.ring);
        if (keeper)
#pragma unroll
            for (int j = 0; j < LIST; ++j)
                lists[((wq * QW + sum % QW) * 2 * WR + 2 * wr + sum_r) * LIST + j] = l[j];
        __syncthreads();
        unsigned long long m[LIST];
        if (WR >= 6) {
            for (int i = warp; i < WQ * QW && q0 + i < n_queries; i += kGemmWarps) {
#pragma unroll
                for (int j = 0; j < LIST; ++j) m[j] = lane < 2 * WR ? lists[(i * 2 * WR + lane) * LIST + j] : 0ull;
                unsigned long long out = 0ull;   // lane j: the j-th best
#pragma unroll
                for (int j = 0; j < LIST; ++j) {
                    const unsigned long long key = warp_max_u64(m[0]);
                    if (lane == j) out = key;
                    if (key == m[0]) {
#pragma unroll
                        for (int h = 0; h + 1 < LIST; ++h) m[h] = m[h + 1];
                        m[LIST - 1] = 0ull;
                    }
                }
                if (lane < kWritten)
                    partial[(static_cast<int64_t>(blockIdx.x) * n_queries + q0 + i) * kListK + lane] = out;
            }
        } else {
            const int i = static_cast<int>(threadIdx.x);
            if (i < WQ * QW && q0 + i < n_queries) {
#pragma unroll
                for (int j = 0; j < LIST; ++j) m[j] = lists[i * 2 * WR * LIST + j];
                for (int r = 1; r < 2 * WR; ++r)
                    for (int j = 0; j < LIST; ++j) {
                        const unsigned long long v = lists[(i * 2 * WR + r) * LIST + j];
                        if (v <= m[LIST - 1]) break;   // sorted: the rest is smaller
                        insert_key<LIST>(m, v);
                    }
#pragma unroll
                for (int j = 0; j < kWritten; ++j)
                    partial[(static_cast<int64_t>(blockIdx.x) * n_queries + q0 + i) * kListK + j] =
                        j < LIST ? m[j < LIST ? j : 0] : 0ull;
            }
        }
    }
}

int num_sms() { return device_sm_count(); }

constexpr int kRowsPerWarpPass = 4;

int gemv_grid(int64_t M) {
    const int64_t rows_per_cta = static_cast<int64_t>(kWarps) * kRowsPerWarpPass;
    const int64_t need = (M + rows_per_cta - 1) / rows_per_cta;
    const int64_t cap = static_cast<int64_t>(num_sms()) * 4;
    return static_cast<int>(need < 1 ? 1 : (need < cap ? need : cap));
}

template <typename T, int QB, int VPL>
cudaError_t launch_gemv_pass(const RetrieveParams &p, int grid, int q0, cudaStream_t stream) {
    constexpr int RIF = QB == 1 ? 4 : 2;
    gemv_top1_kernel<T, QB, VPL, RIF><<<grid, kThreads, 0, stream>>>(
        static_cast<const T *>(p.index), p.M, p.dim, static_cast<const T *>(p.queries), p.n_queries,
        q0, static_cast<unsigned long long *>(p.workspace));
    return cudaGetLastError();
}

// The lengths of rows that reach each kernel (use_gemm): a single query's top-1 up to 512 dims
// or beyond kGemmMaxDim, everything else beyond kGemmMaxDim only.
template <typename T, int QB>
cudaError_t gemv_pass_vpl(const RetrieveParams &p, int grid, int q0, cudaStream_t stream) {
    const int vecs = p.dim / Vec<T>::n;
    const int vpl = (vecs + 31) / 32;
    if constexpr (QB == 1) {
        if (vpl <= 1) return launch_gemv_pass<T, QB, 1>(p, grid, q0, stream);
        if (vpl <= 2) return launch_gemv_pass<T, QB, 2>(p, grid, q0, stream);
        if (vpl <= 3) return launch_gemv_pass<T, QB, 3>(p, grid, q0, stream);
        if (vpl <= 4) return launch_gemv_pass<T, QB, 4>(p, grid, q0, stream);
    }
    return launch_gemv_pass<T, QB, 16>(p, grid, q0, stream);
}

template <typename T>
cudaError_t launch_gemv(const RetrieveParams &p, cudaStream_t stream, int grid, uint64_t *launches) {
    cudaError_t e = cudaSuccess;
    if (p.n_queries == 1) {
        e = gemv_pass_vpl<T, 1>(p, grid, 0, stream);
        ++*launches;
    } else {
        for (int q0 = 0; q0 < p.n_queries && e == cudaSuccess; q0 += kQB, ++*launches)
            e = gemv_pass_vpl<T, kQB>(p, grid, q0, stream);
    }
    return e;
}

// 16-bit indexes go to the tensor cores: one pass over the keys for up to 256 queries,
// streamed by TMA; even a single query's pass is a little faster there (0.246 vs 0.266
// ms over 1M x 768 fp16 keys) than a CUDA-core GEMV, which needs a pass per 4 queries.
// fp32 indexes stay on the CUDA cores (their kernels are instantiated for fp32 keys only).
bool use_tc(const RetrieveParams &p) { return p.dtype != PRECOG_F32; }

template <typename T, int VPL>
cudaError_t launch_topk_pass(const RetrieveParams &p, int grid, int q, cudaStream_t stream) {
    gemv_topk_kernel<T, VPL><<<grid, kThreads, 0, stream>>>(
        static_cast<const T *>(p.index), p.M, p.dim, static_cast<const T *>(p.queries), p.n_queries, q,
        static_cast<unsigned long long *>(p.workspace));
    return cudaGetLastError();
}

template <typename T>
cudaError_t launch_gemv_topk(const RetrieveParams &p, cudaStream_t stream, int grid,
                             uint64_t *launches) {
    const int vpl = (p.dim / Vec<T>::n + 31) / 32;
    cudaError_t e = cudaSuccess;
    for (int q = 0; q < p.n_queries && e == cudaSuccess; ++q, ++*launches)
        e = vpl <= 3 ? launch_topk_pass<T, 3>(p, grid, q, stream) : launch_topk_pass<T, 16>(p, grid, q, stream);
    return e;
}

// fp32 keys of up to kGemmMaxDim dims go to the shared-row kernel. A single query's pass does
// up to 8 queries' arithmetic there, so it goes where that is faster (us, GEMV / shared rows):
// top-1 over rows of more than 512 dims (300,000 x 768: 181 / 139; 200,000 x 256: 37 / 42;
// 300,000 x 384: 71 / 82; 200,000 x 512: 63 / 63); top-k always (50,021 x 384, k = 3: 36 / 24) but
// for long lists over 257 to 384 dims, where insertions stall its few warps (k = 8, 500,000 x
// 384: 141 / 175; 50,021 x 384: 34 / 29).
bool use_gemm(const RetrieveParams &p, bool topk, int k) {
    if (p.dim > kGemmMaxDim) return false;
    if (p.n_queries > 1) return true;
    if (!topk) return p.dim > 512;
    return k <= 3 || p.dim <= 256 || p.dim > 384;
}

// Rows per tile: 24 (12 for rows over 512 dims), and for short rows as many times that as a
// stage holds while every SM still gets a few tiles.
int gemm_tile_rows(int64_t M, int dim) {
    int rows = dim <= 512 ? 24 : 12;
    while (2 * rows * dim * 4 <= kGemmStageBytes && M / (2 * rows) >= 4 * static_cast<int64_t>(num_sms())) rows *= 2;
    return rows;
}

int gemm_grid(int64_t M, int dim) {
    const int rows = gemm_tile_rows(M, dim);
    // no more parts than the workspace is sized for
    return static_cast<int>(std::min<int64_t>(std::min<int64_t>((M + rows - 1) / rows, num_sms()), gemv_grid(M)));
}

template <int VPL, int QW, int LIST>
cudaError_t launch_gemm_vq(const RetrieveParams &p, int grid, cudaStream_t stream, uint64_t *launches) {
    const int groups = (p.n_queries + QW - 1) / QW;
    const int passes = (groups + kGemmWarps - 1) / kGemmWarps;
    int WQ = (groups + passes - 1) / passes;
    while (kGemmWarps % WQ != 0) ++WQ;   // warps split evenly into query groups
    auto kern = gemm_retrieve_kernel<VPL, QW, LIST>;
    const int smem = static_cast<int>(sizeof(GemmSmem));
    cudaError_t e = ensure_smem(reinterpret_cast<const void *>(kern), smem);
    if (e != cudaSuccess) return e;
    const int per_launch = 65535;   // passes per launch (grid y)
    for (int y0 = 0; y0 * WQ < groups; y0 += per_launch) {
        const int left = (groups - y0 * WQ + WQ - 1) / WQ;
        kern<<<dim3(static_cast<unsigned>(grid), static_cast<unsigned>(std::min(left, per_launch))), kGemmThreads, smem,
               stream>>>(static_cast<const float *>(p.index), p.M, p.dim, static_cast<const float *>(p.queries),
                         p.n_queries, gemm_tile_rows(p.M, p.dim), WQ, y0, static_cast<unsigned long long *>(p.workspace));
        e = cudaGetLastError();
        if (e != cudaSuccess) return e;
        ++*launches;
    }
    return cudaSuccess;
}

template <int LIST>
cudaError_t launch_gemm(const RetrieveParams &p, int grid, cudaStream_t stream, uint64_t *launches) {
    const int vpl = (p.dim / 4 + 31) / 32;
    if (vpl <= 1) return launch_gemm_vq<1, 8, LIST>(p, grid, stream, launches);
    if (vpl <= 2) return launch_gemm_vq<2, 8, LIST>(p, grid, stream, launches);
    if (vpl <= 3) return launch_gemm_vq<3, 8, LIST>(p, grid, stream, launches);
    if (vpl <= 4) return launch_gemm_vq<4, 4, LIST>(p, grid, stream, launches);
    if (vpl <= 6) return launch_gemm_vq<6, 4, LIST>(p, grid, stream, launches);
    return launch_gemm_vq<8, 2, LIST>(p, grid, stream, launches);
}

}  // namespace

size_t retrieve_workspace_size(int64_t M, int32_t dim, int32_t n_queries) {
    (void)dim;
    if (n_queries <= 0) return 0;
    const int parts = std::max(gemv_grid(M), retrieve_tc_grid(M, num_sms()));
    return static_cast<size_t>(parts) * n_queries * sizeof(unsigned long long);
}

cudaError_t launch_retrieve(const RetrieveParams &p, cudaStream_t stream) {
    if (p.n_queries == 0) return cudaSuccess;
    const int sz = p.dtype == PRECOG_F32 ? 4 : 2;
    if (p.dim * sz / 16 > kMaxVecsPerRow) return cudaErrorInvalidValue;
    uint64_t launches = 0;
    cudaError_t e = cudaSuccess;
    int parts = 0;  // an empty index has no partial keys: the finalize writes row -1, score NaN
    if (p.M > 0 && use_tc(p)) {
        parts = retrieve_tc_grid(p.M, num_sms());
        e = launch_retrieve_tc(p, parts, stream, &launches);
    } else if (p.M > 0 && use_gemm(p, false, 1)) {
        parts = gemm_grid(p.M, p.dim);
        e = launch_gemm<1>(p, parts, stream, &launches);
    } else if (p.M > 0) {
        parts = gemv_grid(p.M);
        e = launch_gemv<float>(p, stream, parts, &launches);
    }
    if (e == cudaSuccess) {
        e = launch_dependent(finalize_kernel, dim3((p.n_queries + 3) / 4), dim3(128), 0, stream,
                             static_cast<const unsigned long long *>(p.workspace), parts, p.n_queries, p.best_idx,
                             p.best_score, p.row_offset, p.keys_out);
        if (e == cudaSuccess) ++launches;
    }
    count_launches(launches);
    return e;
}

cudaError_t launch_decode_keys(const int64_t *keys, int32_t n, int64_t *best_idx, float *best_score,
                               cudaStream_t stream) {
    if (n == 0) return cudaSuccess;
    decode_keys_kernel<<<(n + 127) / 128, 128, 0, stream>>>(keys, n, best_idx, best_score);
    cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess) count_launches(1);
    return e;
}

size_t retrieve_topk_workspace_size(int64_t M, int32_t dim, int32_t n_queries) {
    (void)dim;
    if (n_queries <= 0) return 0;
    const int parts = std::max(gemv_grid(M), retrieve_tc_grid(M, num_sms()));
    return static_cast<size_t>(parts) * n_queries * kListK * sizeof(unsigned long long);
}

cudaError_t launch_retrieve_topk(const RetrieveParams &p, int k, cudaStream_t stream) {
    if (p.n_queries == 0) return cudaSuccess;
    const int sz = p.dtype == PRECOG_F32 ? 4 : 2;
    if (p.dim * sz / 16 > kMaxVecsPerRow || k < 1 || k > kListK) return cudaErrorInvalidValue;
    uint64_t launches = 0;
    cudaError_t e = cudaSuccess;
    int parts = 0;  // an empty index has no partial lists: the finalize writes rows -1
    int log_used = 3;
    if (p.M > 0 && use_tc(p)) {
        parts = retrieve_tc_grid(p.M, num_sms());
        e = launch_retrieve_tc_topk(p, k, parts, stream, &launches);
        log_used = k <= 2 ? 1 : (k <= 4 ? 2 : 3);   // the tensor-core kernel's list lengths
    } else if (p.M > 0 && use_gemm(p, true, k)) {
        parts = gemm_grid(p.M, p.dim);
        e = k <= 3 ? launch_gemm<3>(p, parts, stream, &launches) : launch_gemm<8>(p, parts, stream, &launches);
        log_used = k <= 3 ? 2 : 3;
    } else if (p.M > 0) {
        parts = gemv_grid(p.M);
        e = launch_gemv_topk<float>(p, stream, parts, &launches);
    }
    if (e == cudaSuccess) {
        e = launch_dependent(finalize_topk_kernel, dim3((p.n_queries + 3) / 4), dim3(128), 0, stream,
                             static_cast<const unsigned long long *>(p.workspace), parts, log_used, p.n_queries, k,
                             p.best_idx, p.best_score);
        if (e == cudaSuccess) ++launches;
    }
    count_launches(launches);
    return e;
}

cudaError_t retrieve_status_word_read_clear(uint32_t *bits) {
    uint32_t zero = 0, tc = 0;
    cudaError_t e = cudaMemcpyFromSymbol(bits, g_retrieve_status, sizeof(uint32_t));
    if (e != cudaSuccess) return e;
    e = cudaMemcpyToSymbol(g_retrieve_status, &zero, sizeof(uint32_t));
    if (e != cudaSuccess) return e;
    e = retrieve_tc_status_word_read_clear(&tc);
    *bits |= tc;
    return e;
}

}  // namespace precog
