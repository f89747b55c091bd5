// Selective-SSM scan with final-state capture (corpus encode) and with an
// injected initial state (query prefill) -- Sec. 3 Eq. 1, Sec. 4.2, Eq. 2.
//
// Work decomposition: one CTA per (layer, chunk, slice of DS channels). Each
// thread owns CPT adjacent channels and keeps their N = 16 fp32 states in
// registers for the whole chunk. The chunk's rows of x and dt (DS channels
// each) and of B (and C) are staged into shared memory TILE tokens at a time
// by the TMA engine, completing on an mbarrier, in a STAGES-deep ring, so the
// time loop only reads shared memory: a whole-row slice is one contiguous 1-D
// bulk copy per tensor; a narrower slice (wide rows) is one tiled tensor-map
// copy of TILE rows per tensor. Captures with few work items share a chunk's
// tokens among the CTAs of a cluster (see combine).
//
// Per token and channel the recurrence is, for the 16 state indices n,
//   h[n] <- alpha_n * h[n] + (dt * x) * B[n],   alpha_n = exp(dt * A[d, n]).
// Three update forms, all in packed fp32x2 arithmetic:
//   kGeneral   one SFU exponential per (d, n);
//   kPower     A[d, n] = (n + 1) * A[d, 0] (stated by the caller, verified per
//              CTA): alpha_n = r^(n+1), r = exp(dt * A[d, 0]), one exponential
//              and a power chain per (t, d); with a readout y the state is
//              updated directly, without one it is accumulated rescaled
//              (see scan_tile_rescaled), which drops the per-n decay multiply.
#include <cfloat>
#include <type_traits>

#include "../../include/precog.h"
#include "internal.h"
#include "ptx.cuh"

namespace precog {
namespace {

__device__ uint32_t g_scan_status;

// Shape of the rescaled capture kernel (channels per thread, tokens per stage,
// stages, resident blocks per SM for the register budget).
#ifndef PRECOG_RESCALED_CPT
#define PRECOG_RESCALED_CPT 4
#endif
#ifndef PRECOG_RESCALED_TILE
#define PRECOG_RESCALED_TILE 16
#endif
#ifndef PRECOG_RESCALED_STAGES
#define PRECOG_RESCALED_STAGES 2
#endif
#ifndef PRECOG_RESCALED_MINB
#define PRECOG_RESCALED_MINB 6
#endif
// Shape of the direct-update kernels with A stated structured (readout, prefill).
#ifndef PRECOG_DIRECT_CPT
#define PRECOG_DIRECT_CPT 4
#endif
#ifndef PRECOG_DIRECT_TILE
#define PRECOG_DIRECT_TILE 16
#endif
#ifndef PRECOG_DIRECT_STAGES
#define PRECOG_DIRECT_STAGES 2
#endif
#ifndef PRECOG_DIRECT_MINB
#define PRECOG_DIRECT_MINB 5
#endif
#ifndef PRECOG_RESCALED_GROUP
#define PRECOG_RESCALED_GROUP 4
#endif


// Tokens whose exponentials the direct update forms ahead: their latency and the loads' then
// overlap the previous tokens' chains. Against one token at a time: readout of 256 chunks x 512
// tokens x 2048 channels 689 -> 652 us, 4 layers x 1000 x 500 1307 -> 1218; trajectories (every
// 8th state of 4 x 128 x 750) 414 -> 340; groups of 2: 670, 1268, 348; of 8: 3 % slower than 4
// in the readouts; of a whole tile 50 % (registers).
constexpr int kDirectGroup = 4;

constexpr int kN = 16;          // state size (N) supported by the kernels
constexpr int kMaxSlice = 256;  // channels per CTA at most (the default slice)
constexpr int kWideSlice = 512; // rows of up to this many channels are staged whole
constexpr int kBarBytes = 128;  // barrier area at the start of shared memory
constexpr float kLog2e = 1.4426950408889634f;
constexpr int kMaxTopk = 8;     // states composed at most by one injection

__device__ __forceinline__ int64_t min64(int64_t a, int64_t b) { return a < b ? a : b; }

enum Mode { kGeneral = 0, kPower = 1 };

// Compile-time shape of one kernel instantiation.
constexpr int kTrajNone = 0, kTrajDirect = 1, kTrajRescaled = 2;

template <typename TIn_, bool HAS_Y_, bool HAS_H0_, int MODE_, int CPT_, int TILE_, int STAGES_,
          int MINB_, int TRAJ_ = kTrajNone, int MAXSLICE_ = kMaxSlice, int FIXDS_ = 0, bool SPLIT_ = false,
          bool PAIRS_ = false>
struct Cfg {
    using TIn = TIn_;
    // Channel slice known at compile time (0: a launch argument). A constant slice turns
    // the shared-memory row offsets of the time loop into immediates.
    static constexpr int FIXDS = FIXDS_;
    // A cluster of CTAs per work item, each with a share of the chunk's tokens (see combine).
    static constexpr bool SPLIT = SPLIT_;
    // 256-channel slices that stand in for 512-channel ones (PAIRS_: the shape of launch_pairs,
    // two channels per thread where other inputs take four): the power statement is verified
    // for the 512 channels together, as by those.
    static constexpr bool WIDE_CHECK = MODE_ == kPower && CPT_ == 2 && (SPLIT_ || PAIRS_ || TRAJ_ != kTrajNone);
    // Widest channel slice of one CTA. Each CTA stages its slice of every token row; a
    // slice narrower than the row turns the row into separate pieces, and HBM serves
    // short scattered pieces far below its streaming rate, so rows up to 512 channels
    // stay whole. MINB counts resident CTAs of kMaxSlice channels (the register budget
    // per thread), whatever the slice.
    static constexpr int MAXSLICE = MAXSLICE_;
    static constexpr int LB_SLICE = FIXDS_ ? FIXDS_ : MAXSLICE_;
    static constexpr int LB_THREADS = LB_SLICE / CPT_;
    static constexpr int LB_BLOCKS = MINB_ * kMaxSlice / LB_SLICE > 0 ? MINB_ * kMaxSlice / LB_SLICE : 1;
    static constexpr bool HAS_Y = HAS_Y_, HAS_H0 = HAS_H0_;
    // keep every stride-th state (K-dial, Sec. 5.2), with the direct or the rescaled update
    static constexpr int TRAJ = TRAJ_;
    static constexpr int MODE = MODE_, CPT = CPT_, TILE = TILE_, STAGES = STAGES_;
    // trajectory states leave through shared memory (see store_trajectory)
    static constexpr bool STAGED = TRAJ_ != kTrajNone && PAIRS_;
    static constexpr bool CONV = !std::is_same<TIn_, float>::value;
    static constexpr int SZ = sizeof(TIn_);
    static constexpr bool RESCALED = MODE_ == kPower && !HAS_Y_ && TRAJ_ != kTrajDirect;
};

// Where the next trajectory state goes: entry index and tokens left until it.
struct TrajCursor {
    int64_t entry;
    int64_t left;
    // the warp's staging buffers, which of them is next, and its channels
    unsigned char *bufs;
    int which, channels, first;
};

// Tensor maps of x and dt for launches whose CTAs take a slice of each row: the tensor is
// viewed as [layer][row][D / inner][inner] (inner = min(slice, 256), the widest box dimension),
// so a box of [1][TILE][slice / inner][inner] is one slice of TILE rows; inner == 0: the
// slices don't divide the row and a box starts at its channel of [layer][row][1][D].
struct SliceMaps {
    CUtensorMap x, dt;
    int32_t valid, inner;
};

struct StageLayout {
    uint32_t xs, dts, bs, cs, bf, cf, bytes;
};

__host__ __device__ inline StageLayout stage_layout(int tile, int DS, int sz, bool has_y, bool conv) {
    StageLayout L;
    uint32_t o = 0;
    L.xs = o;
    o += tile * DS * sz;
    L.dts = o;
    o += tile * DS * sz;
    L.bs = o;
    o += tile * kN * sz;
    L.cs = o;
    if (has_y) o += tile * kN * sz;
    L.bf = o;
    if (conv) o += tile * kN * 4;
    L.cf = o;
    if (conv && has_y) o += tile * kN * 4;
    L.bytes = (o + 127u) & ~127u;
    return L;
}

// CPT adjacent channel values of one token row in shared memory; `neg` gets
// the sign bits of the raw values (nonzero if any is negative).
template <typename TIn, int CPT>
__device__ __forceinline__ void load_chan(const unsigned char *p, float (&v)[CPT], uint32_t &neg) {
    if constexpr (std::is_same<TIn, float>::value) {
        static_assert(CPT == 2, "fp32 inputs: two channels per thread");
        const float2 q = *reinterpret_cast<const float2 *>(p);
        v[0] = q.x;
        v[1] = q.y;
        neg = (__float_as_uint(q.x) | __float_as_uint(q.y)) & 0x80000000u;
    } else {
        uint32_t w[CPT / 2];
        if constexpr (CPT == 2) {
            w[0] = *reinterpret_cast<const uint32_t *>(p);
        } else {
            const uint2 q = *reinterpret_cast<const uint2 *>(p);
            w[0] = q.x;
            w[1] = q.y;
        }
        uint32_t s = 0;
#pragma unroll
        for (int i = 0; i < CPT / 2; ++i) {
            v[2 * i] = __uint_as_float(w[i] << 16);
            v[2 * i + 1] = __uint_as_float(w[i] & 0xffff0000u);
            s |= w[i];
        }
        neg = s & 0x80008000u;
    }
}

__device__ __forceinline__ void load_b(const float *bsrc, int t, f2 (&b)[8]) {
    const ulonglong2 *bv = reinterpret_cast<const ulonglong2 *>(bsrc + t * kN);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const ulonglong2 v = bv[i];
        b[2 * i] = v.x;
        b[2 * i + 1] = v.y;
    }
}

__device__ __forceinline__ void store_state16(void *base, int dtype, int64_t elem_off,
                                              const f2 (&h)[8]) {
    float v[16];
#pragma unroll
    for (int i = 0; i < 8; ++i) unpack2(h[i], v[2 * i], v[2 * i + 1]);
    if (dtype == PRECOG_F32) {
        float4 *dst = reinterpret_cast<float4 *>(static_cast<float *>(base) + elem_off);
#pragma unroll
        for (int i = 0; i < 4; ++i)
            dst[i] = make_float4(v[4 * i], v[4 * i + 1], v[4 * i + 2], v[4 * i + 3]);
    } else {
        uint4 *dst = reinterpret_cast<uint4 *>(static_cast<__nv_bfloat16 *>(base) + elem_off);
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            uint32_t w[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                __nv_bfloat162 b2 = __floats2bfloat162_rn(v[8 * i + 2 * k], v[8 * i + 2 * k + 1]);
                w[k] = *reinterpret_cast<uint32_t *>(&b2);
            }
            dst[i] = make_uint4(w[0], w[1], w[2], w[3]);
        }
    }
}

__device__ __forceinline__ void load_state16(const void *base, int dtype, int64_t elem_off,
                                             f2 (&h)[8]) {
    float v[16];
    if (dtype == PRECOG_F32) {
        const float4 *src = reinterpret_cast<const float4 *>(static_cast<const float *>(base) + elem_off);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const float4 q = src[i];
            v[4 * i] = q.x;
            v[4 * i + 1] = q.y;
            v[4 * i + 2] = q.z;
            v[4 * i + 3] = q.w;
        }
    } else {
        const uint4 *src =
            reinterpret_cast<const uint4 *>(static_cast<const __nv_bfloat16 *>(base) + elem_off);
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            const uint4 q = src[i];
            const uint32_t w[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                v[8 * i + 2 * k] = __uint_as_float(w[k] << 16);
                v[8 * i + 2 * k + 1] = __uint_as_float(w[k] & 0xffff0000u);
            }
        }
    }
#pragma unroll
    for (int i = 0; i < 8; ++i) h[i] = pack2(v[2 * i], v[2 * i + 1]);
}

// p[i] = (r^(2i+1), r^(2i+2)) for i = 0..7
// (x*x, x*x) as one register pair with both halves computed: two multiplies the
// compiler may not merge, instead of one multiply and a register move.
__device__ __forceinline__ f2 sq_pair(float x) {
    float a, b;
    asm volatile("mul.rn.f32 %0, %1, %1;" : "=f"(a) : "f"(x));
    asm volatile("mul.rn.f32 %0, %1, %1;" : "=f"(b) : "f"(x));
    return pack2(a, b);
}

// pow_pairs for the direct update, whose FMA-heavy pipe the moves of duplicated pairs
// saturate (the rescaled capture keeps the move: there the extra multiplies cost more)
__device__ __forceinline__ void pow_pairs_direct(float r, f2 (&p)[8]) {
    const float r2 = r * r;
    p[0] = pack2(r, r2);
    const f2 rr = sq_pair(r);
#pragma unroll
    for (int i = 1; i < 8; ++i) p[i] = mul2(p[i - 1], rr);
}

__device__ __forceinline__ void pow_pairs(float r, f2 (&p)[8]) {
    const float r2 = r * r;
    p[0] = pack2(r, r2);
    const f2 rr = pack2(r2, r2);
#pragma unroll
    for (int i = 1; i < 8; ++i) p[i] = mul2(p[i - 1], rr);
}

// dt * x of the low (high) bf16 halves of two words, exact in fp32 (a product of two
// 8-bit significands), by the mixed-precision FMA with -0 as addend: no widening.
__device__ __forceinline__ float mul_bf16_lo(uint32_t a, uint32_t b) {
    float d;
    asm("{ .reg .b16 al, ah, bl, bh; mov.b32 {al, ah}, %1; mov.b32 {bl, bh}, %2;"
        " fma.rn.f32.bf16 %0, al, bl, %3; }"
        : "=f"(d) : "r"(a), "r"(b), "f"(-0.0f));
    return d;
}
// The same products as volatile statements (not merged with an equal one).
__device__ __forceinline__ float mul_bf16_lo_v(uint32_t a, uint32_t b) {
    float d;
    asm volatile("{ .reg .b16 al, ah, bl, bh; mov.b32 {al, ah}, %1; mov.b32 {bl, bh}, %2;"
                 " fma.rn.f32.bf16 %0, al, bl, %3; }"
                 : "=f"(d) : "r"(a), "r"(b), "f"(-0.0f));
    return d;
}
__device__ __forceinline__ float mul_bf16_hi_v(uint32_t a, uint32_t b) {
    float d;
    asm volatile("{ .reg .b16 al, ah, bl, bh; mov.b32 {al, ah}, %1; mov.b32 {bl, bh}, %2;"
                 " fma.rn.f32.bf16 %0, ah, bh, %3; }"
                 : "=f"(d) : "r"(a), "r"(b), "f"(-0.0f));
    return d;
}
__device__ __forceinline__ float mul_bf16_hi(uint32_t a, uint32_t b) {
    float d;
    asm("{ .reg .b16 al, ah, bl, bh; mov.b32 {al, ah}, %1; mov.b32 {bl, bh}, %2;"
        " fma.rn.f32.bf16 %0, ah, bh, %3; }"
        : "=f"(d) : "r"(a), "r"(b), "f"(-0.0f));
    return d;
}

template <int CPT>
__device__ __forceinline__ void load_words(const unsigned char *p, uint32_t (&w)[CPT / 2]) {
    if constexpr (CPT == 2) {
        w[0] = *reinterpret_cast<const uint32_t *>(p);
    } else {
        const uint2 q = *reinterpret_cast<const uint2 *>(p);
        w[0] = q.x;
        w[1] = q.y;
    }
}

template <int CPT>
__device__ __forceinline__ void widen_words(const uint32_t (&w)[CPT / 2], float (&v)[CPT]) {
#pragma unroll
    for (int i = 0; i < CPT / 2; ++i) {
        v[2 * i] = __uint_as_float(w[i] << 16);
        v[2 * i + 1] = __uint_as_float(w[i] & 0xffff0000u);
    }
}

// ---------------------------------------------------------------------------
// Trajectory states. The states of a warp's channels are adjacent in an entry, but a thread's
// are 32 to 128 bytes apart from its neighbour's, so plain stores of 16 bytes touched 32 lines
// each with half a sector and bound the fine strides. A warp instead lays its states out in a
// shared-memory buffer (rotating the 16-byte pieces by lane, so that the lanes meet different
// banks) and one lane sends them off as a bulk copy; a warp has two buffers of bf16 states or
// one of fp32. With two channels per thread (launch_pairs), 4 layers x 40 chunks x 750 tokens,
// every state bf16 615 -> 476 us and fp32 1253 -> 565, every third (100 chunks) 472 -> 386 and
// 801 -> 538; strides 16 to 100 5 to 25 % (435, 457, 329, 520 with the grouped direct update).
__host__ __device__ constexpr int traj_buffer_bytes(int cpt) { return 2 * 32 * cpt * kN * 2; }   // per warp

template <int CPT>
__device__ __forceinline__ void store_trajectory(unsigned char *bufs, int &which, int lane, int channels, void *base,
                                                 int dtype, int64_t elem_off, const f2 (&h)[CPT][8]) {
    if (channels <= 0) return;   // a warp past the end of the row (uniform)
    // the copy before the last one (fp32: the last one) has left the buffer
    if (lane == 0) {
        if (dtype == PRECOG_F32) bulk_wait_read<0>();
        else bulk_wait_read<1>();
    }
    __syncwarp();
    unsigned char *buf = dtype == PRECOG_F32 ? bufs : bufs + which * (traj_buffer_bytes(CPT) / 2);
    which ^= 1;
    const int rot = (lane >> 1) & 3;
    // blocks of four 16-byte pieces: half a channel's fp32 states twice over, or two channels' bf16
    auto put = [&](int block, int blocks, const uint4 (&p)[4]) {
        uint4 r[4], q[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) r[i] = rot & 1 ? p[(i + 1) & 3] : p[i];
#pragma unroll
        for (int i = 0; i < 4; ++i) q[i] = rot & 2 ? r[(i + 2) & 3] : r[i];
        uint4 *dst = reinterpret_cast<uint4 *>(buf) + (lane * blocks + block) * 4;
#pragma unroll
        for (int i = 0; i < 4; ++i) dst[(i + rot) & 3] = q[i];
    };
    static_assert(CPT % 2 == 0, "two channels per block of bf16 pieces");
    if (dtype == PRECOG_F32) {
#pragma unroll
        for (int j = 0; j < CPT; ++j) {
            uint4 p[4];
#pragma unroll
            for (int i = 0; i < 4; ++i)
                p[i] = make_uint4(static_cast<uint32_t>(h[j][2 * i]), static_cast<uint32_t>(h[j][2 * i] >> 32),
                                  static_cast<uint32_t>(h[j][2 * i + 1]), static_cast<uint32_t>(h[j][2 * i + 1] >> 32));
            put(j, CPT, p);
        }
    } else {
#pragma unroll
        for (int j = 0; j < CPT; j += 2) {
            uint4 p[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                uint32_t w[4];
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    float lo, hi;
                    unpack2(h[j + i / 2][(i & 1) * 4 + k], lo, hi);
                    const __nv_bfloat162 b2 = __floats2bfloat162_rn(lo, hi);
                    w[k] = *reinterpret_cast<const uint32_t *>(&b2);
                }
                p[i] = make_uint4(w[0], w[1], w[2], w[3]);
            }
            put(j / 2, CPT / 2, p);
        }
    }
    fence_proxy_async_smem();
    __syncwarp();
    if (lane == 0) {
        const int sz = dtype == PRECOG_F32 ? 4 : 2;
        bulk_s2g(static_cast<unsigned char *>(base) + elem_off * sz, buf, static_cast<uint32_t>(channels * kN * sz));
        bulk_commit();
    }
}

// ---------------------------------------------------------------------------
// Direct update (any readout): h_n <- alpha_n h_n + u B_n, y = sum_n C_n h_n.
template <class C>
__device__ __forceinline__ void scan_tile_direct(const unsigned char *st, const StageLayout &lay,
                                                 int DS, int dl, int ntok,
                                                 f2 (&h)[C::CPT][8], const float (&kpow)[C::CPT],
                                                 const f2 (&kgen)[C::CPT][8], void *yrow,
                                                 int y_dtype, int64_t y_stride,
                                                 const ScanParams &p, TrajCursor &tc,
                                                 int64_t tok_left, int traj_layer, int dglob,
                                                 float (&tot)[C::CPT]) {
    constexpr int CPT = C::CPT;
    const float *bsrc = reinterpret_cast<const float *>(st + (C::CONV ? lay.bf : lay.bs));
    const float *csrc = reinterpret_cast<const float *>(st + (C::CONV ? lay.cf : lay.cs));
    // dt and x of a token: raw words of 16-bit inputs (u = dt * x is formed from the halves,
    // exactly, and x never widened), else values
    struct Chan {
        uint32_t xw[CPT / 2], dw[CPT / 2];
        float xv[CPT], dv[CPT], r[CPT];
    };
    auto fetch = [&](int t, Chan &c) {
        if constexpr (C::CONV) {
            load_words<CPT>(st + lay.xs + (t * DS + dl) * C::SZ, c.xw);
            load_words<CPT>(st + lay.dts + (t * DS + dl) * C::SZ, c.dw);
            widen_words<CPT>(c.dw, c.dv);
        } else {
            uint32_t neg;
            load_chan<typename C::TIn, CPT>(st + lay.xs + (t * DS + dl) * C::SZ, c.xv, neg);
            load_chan<typename C::TIn, CPT>(st + lay.dts + (t * DS + dl) * C::SZ, c.dv, neg);
        }
        if constexpr (C::MODE == kPower) {
#pragma unroll
            for (int j = 0; j < CPT; ++j) c.r[j] = ex2(c.dv[j] * kpow[j]);
        }
    };
    auto token = [&](int t, const Chan &c) {
        f2 b[8];
        load_b(bsrc, t, b);
        float yv[CPT] = {};
        f2 uu2[CPT];   // (u, u)
        if constexpr (C::CONV) {
            // both halves computed: two products cost less than a product and a move
#pragma unroll
            for (int i = 0; i < CPT / 2; ++i) {
                uu2[2 * i] = pack2(mul_bf16_lo_v(c.dw[i], c.xw[i]), mul_bf16_lo_v(c.dw[i], c.xw[i]));
                uu2[2 * i + 1] = pack2(mul_bf16_hi_v(c.dw[i], c.xw[i]), mul_bf16_hi_v(c.dw[i], c.xw[i]));
            }
        } else {
#pragma unroll
            for (int j = 0; j < CPT; ++j) uu2[j] = pack2(c.dv[j] * c.xv[j], c.dv[j] * c.xv[j]);
        }
        if constexpr (C::SPLIT) {
#pragma unroll
            for (int j = 0; j < CPT; ++j) tot[j] += c.dv[j];
        }
#pragma unroll
        for (int j = 0; j < CPT; ++j) {
            const f2 uu = uu2[j];
            if constexpr (C::MODE == kPower) {
                f2 a[8];
                pow_pairs_direct(c.r[j], a);
#pragma unroll
                for (int i = 0; i < 8; ++i) h[j][i] = fma2(a[i], h[j][i], mul2(uu, b[i]));
            } else {
                const f2 dd = pack2(c.dv[j], c.dv[j]);
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    float e0, e1;
                    unpack2(mul2(dd, kgen[j][i]), e0, e1);
                    h[j][i] = fma2(pack2(ex2(e0), ex2(e1)), h[j][i], mul2(uu, b[i]));
                }
            }
            if constexpr (C::HAS_Y) {
                const ulonglong2 *cv = reinterpret_cast<const ulonglong2 *>(csrc + t * kN);
                f2 acc = 0;
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const ulonglong2 c = cv[i];
                    acc = (i == 0) ? mul2(c.x, h[j][0]) : fma2(c.x, h[j][2 * i], acc);
                    acc = fma2(c.y, h[j][2 * i + 1], acc);
                }
                float lo, hi;
                unpack2(acc, lo, hi);
                yv[j] = lo + hi;
            }
        }
        if constexpr (C::HAS_Y) {
            if (y_dtype == PRECOG_F32) {
                float *dst = static_cast<float *>(yrow) + t * y_stride;
                if constexpr (CPT == 2) {
                    *reinterpret_cast<float2 *>(dst) = make_float2(yv[0], yv[1]);
                } else {
                    *reinterpret_cast<float4 *>(dst) = make_float4(yv[0], yv[1], yv[2], yv[3]);
                }
            } else {
                __nv_bfloat16 *dst = static_cast<__nv_bfloat16 *>(yrow) + t * y_stride;
                __nv_bfloat162 p0 = __floats2bfloat162_rn(yv[0], yv[1]);
                if constexpr (CPT == 2) {
                    *reinterpret_cast<__nv_bfloat162 *>(dst) = p0;
                } else {
                    __nv_bfloat162 p1 = __floats2bfloat162_rn(yv[2], yv[3]);
                    *reinterpret_cast<uint2 *>(dst) = make_uint2(
                        *reinterpret_cast<uint32_t *>(&p0), *reinterpret_cast<uint32_t *>(&p1));
                }
            }
        }
        if constexpr (C::TRAJ == kTrajDirect) {
            // after every stride-th token and after the chunk's last token (uniform)
            if (--tc.left == 0 || t + 1 == tok_left) {
                const int64_t row = (tc.entry * p.L_out + traj_layer) * static_cast<int64_t>(p.D);
                if constexpr (C::STAGED) {
                    store_trajectory<CPT>(tc.bufs, tc.which, threadIdx.x & 31, tc.channels, p.traj, p.traj_dtype,
                                          (row + tc.first) * kN, h);
                } else {
#pragma unroll
                    for (int j = 0; j < CPT; ++j)
                        store_state16(p.traj, p.traj_dtype, (row + dglob + j) * kN, h[j]);
                }
                ++tc.entry;
                tc.left = p.traj_stride;
            }
        }
    };
    constexpr int G = C::MODE == kPower ? kDirectGroup : 1;   // general A: 16 exponentials per token already
    int t = 0;
    if constexpr (G > 1) {
        for (; t + G <= ntok; t += G) {
            Chan c[G];
#pragma unroll
            for (int g = 0; g < G; ++g) fetch(t + g, c[g]);
#pragma unroll
            for (int g = 0; g < G; ++g) token(t + g, c[g]);
        }
    }
    for (; t < ntok; ++t) {
        Chan c;
        fetch(t, c);
        token(t, c);
    }
}

// ---------------------------------------------------------------------------
// Rescaled accumulation (capture without readout, A[d, n] = (n + 1) * a, a <= 0).
// With E_t = 2^(L_t), L_t = sum over the tokens since the last renormalisation
// of dt * (-a * log2 e), the state is h_n = E_t^-(n+1) * G_n and one token adds
//   G_n += (u * E_t^(n+1)) * B_n,     u = dt * x,
// so the per-n decay multiply of the direct update disappears: per token and
// channel one exponential, a packed power chain and 16 FMAs. Whenever some
// lane's L would leave [-kLmax, kLmax] the whole warp renormalises
// (h_n = G_n E^-(n+1), L = 0), which keeps E^(+-16) within 2^(16 * kLmax),
// far from fp32 overflow and underflow. A single token whose own increment is
// outside the window is applied to h directly.
constexpr float kLmax = 6.0f;

__device__ __forceinline__ void renormalise(f2 (&g)[8], float &L) {
    f2 p[8];
    pow_pairs(ex2(-L), p);
#pragma unroll
    for (int i = 0; i < 8; ++i) g[i] = mul2(g[i], p[i]);
    L = 0.f;
}

// G_n += u * E^(n+1) * B_n
__device__ __forceinline__ void accumulate_e(f2 (&g)[8], const f2 (&b)[8], float u, float E) {
    const float w0 = u * E;
    const float E2 = E * E;
    f2 w = pack2(w0, w0 * E);
    const f2 ee = pack2(E2, E2);
    g[0] = fma2(w, b[0], g[0]);
#pragma unroll
    for (int i = 1; i < 8; ++i) {
        w = mul2(w, ee);
        g[i] = fma2(w, b[i], g[i]);
    }
}

// G_n += u * 2^((n+1) * Ln) * B_n
__device__ __forceinline__ void accumulate(f2 (&g)[8], const f2 (&b)[8], float u, float Ln) {
    const float E = ex2(Ln);
    const float w0 = u * E;
    const float E2 = E * E;
    f2 w = pack2(w0, w0 * E);
    const f2 ee = pack2(E2, E2);
    g[0] = fma2(w, b[0], g[0]);
#pragma unroll
    for (int i = 1; i < 8; ++i) {
        w = mul2(w, ee);
        g[i] = fma2(w, b[i], g[i]);
    }
}

// One token with the window check of every lane and channel.
template <int CPT>
__device__ __forceinline__ void token_checked(f2 (&g)[CPT][8], float (&L)[CPT],
                                              const float (&kk)[CPT], const f2 (&b)[8],
                                              const float (&xv)[CPT], const float (&dv)[CPT],
                                              unsigned wmask) {
    float Ln[CPT], u[CPT];
    bool need = false;
#pragma unroll
    for (int j = 0; j < CPT; ++j) {
        Ln[j] = fmaf(dv[j], kk[j], L[j]);
        u[j] = dv[j] * xv[j];
        need |= !(fabsf(Ln[j]) <= kLmax);
    }
    if (__any_sync(wmask, need)) {
#pragma unroll
        for (int j = 0; j < CPT; ++j) {
            renormalise(g[j], L[j]);
            Ln[j] = dv[j] * kk[j];
            if (!(fabsf(Ln[j]) <= kLmax)) {
                f2 a[8];
                pow_pairs(ex2(-Ln[j]), a);
                const f2 uu = pack2(u[j], u[j]);
#pragma unroll
                for (int i = 0; i < 8; ++i) g[j][i] = fma2(a[i], g[j][i], mul2(uu, b[i]));
                Ln[j] = 0.f;
                u[j] = 0.f;
            }
        }
    }
#pragma unroll
    for (int j = 0; j < CPT; ++j) {
        accumulate(g[j], b, u[j], Ln[j]);
        L[j] = Ln[j];
    }
}

// Moves the frame of G to the bottom of the window: h_n = G_n E^-(n+1) is re-expressed
// with L = -kLmax, G_n <- G_n 2^-((n+1)(L + kLmax)). With dt >= 0 the exponent then
// climbs through the whole window [-kLmax, kLmax] before the next renormalisation,
// twice as many tokens as a restart from L = 0. The factor of states 8..15 can fall
// below the fp32 range (s = L + kLmax <= 2 kLmax), so they take it in two multiplies,
// 2^-8s first; every factor and every intermediate stays within 2^(+-16 kLmax).
__device__ __forceinline__ void renorm_floor(f2 (&g)[8], float &L) {
    const float r = ex2(-(L + kLmax));
    const float r2 = r * r;
    f2 p[4];
    p[0] = pack2(r, r2);
    const f2 rr = pack2(r2, r2);
#pragma unroll
    for (int i = 1; i < 4; ++i) p[i] = mul2(p[i - 1], rr);
    float r7, r8;
    unpack2(p[3], r7, r8);
    const f2 q = pack2(r8, r8);
#pragma unroll
    for (int i = 0; i < 4; ++i) g[i] = mul2(g[i], p[i]);
#pragma unroll
    for (int i = 4; i < 8; ++i) g[i] = mul2(mul2(g[i], q), p[i - 4]);
    L = -kLmax;
}

// Tokens go in groups of kGroup. The group's exponents are summed first (one
// serial FMA per token and channel). With dt >= 0 they only grow, so checking
// the group's last exponent covers every token in it. One warp vote per group;
// the fast path then carries no branch, so the power chains of the group's
// tokens can interleave. When some lane's exponent would leave the window, the
// warp renormalises every channel to the bottom of the window before the group
// and takes the fast path all the same; only a negative dt anywhere in the group
// (seen from the sign bits) or a group whose own exponent increment exceeds the
// whole window goes through the per-token check.
constexpr int kGroup = PRECOG_RESCALED_GROUP;

template <class C>
__device__ __forceinline__ void scan_tile_rescaled(const unsigned char *st, const StageLayout &lay,
                                                   const float *bsrc, int DS, int dl, int t0, int ntok,
                                                   f2 (&g)[C::CPT][8], float (&L)[C::CPT],
                                                   const float (&kk)[C::CPT], unsigned wmask,
                                                   float (&tot)[C::CPT]) {
    constexpr int CPT = C::CPT;
    using TIn = typename C::TIn;
    // 16-bit inputs: dt is kept as raw words across the vote, and u = dt * x is formed
    // from the raw halves
    constexpr bool MIX = C::CONV;
    int t = t0;
    for (; t + kGroup <= ntok; t += kGroup) {
        float dvk[kGroup][CPT], Lk[kGroup][CPT];
        uint32_t dw[kGroup][CPT / 2];
        uint32_t neg = 0;
#pragma unroll
        for (int k = 0; k < kGroup; ++k) {
            if constexpr (MIX) {
                load_words<CPT>(st + lay.dts + ((t + k) * DS + dl) * C::SZ, dw[k]);
                widen_words<CPT>(dw[k], dvk[k]);
#pragma unroll
                for (int i = 0; i < CPT / 2; ++i) neg |= dw[k][i];
            } else {
                uint32_t nk;
                load_chan<TIn, CPT>(st + lay.dts + ((t + k) * DS + dl) * C::SZ, dvk[k], nk);
                neg |= nk;
            }
#pragma unroll
            for (int j = 0; j < CPT; ++j) Lk[k][j] = fmaf(dvk[k][j], kk[j], k ? Lk[k - 1][j] : L[j]);
        }
        if constexpr (C::SPLIT) {
#pragma unroll
            for (int j = 0; j < CPT; ++j)
#pragma unroll
                for (int k = 0; k < kGroup; k += 2) tot[j] += dvk[k][j] + dvk[k + 1][j];
        }
        if constexpr (MIX) neg &= 0x80008000u;
        bool up = false;
#pragma unroll
        for (int j = 0; j < CPT; ++j) up |= !(Lk[kGroup - 1][j] <= kLmax);
        bool slow = false;
        if (__any_sync(wmask, up || neg != 0)) {
            slow = __any_sync(wmask, neg != 0);
            if (!slow) {
#pragma unroll
                for (int j = 0; j < CPT; ++j) renorm_floor(g[j], L[j]);
                bool up2 = false;
#pragma unroll
                for (int k = 0; k < kGroup; ++k) {
                    if constexpr (MIX) widen_words<CPT>(dw[k], dvk[k]);
#pragma unroll
                    for (int j = 0; j < CPT; ++j) Lk[k][j] = fmaf(dvk[k][j], kk[j], k ? Lk[k - 1][j] : L[j]);
                }
#pragma unroll
                for (int j = 0; j < CPT; ++j) up2 |= !(Lk[kGroup - 1][j] <= kLmax);
                slow = __any_sync(wmask, up2);
            }
        }
        if (slow) {
            // unrolled so that dvk stays in registers (no dynamic indexing)
#pragma unroll
            for (int k = 0; k < kGroup; ++k) {
                f2 b[8];
                float xv[CPT];
                uint32_t nx;
                load_b(bsrc, t + k, b);
                load_chan<TIn, CPT>(st + lay.xs + ((t + k) * DS + dl) * C::SZ, xv, nx);
                if constexpr (MIX) widen_words<CPT>(dw[k], dvk[k]);
                token_checked<CPT>(g, L, kk, b, xv, dvk[k], wmask);
            }
        } else {
            // the group's exponentials first, so that their latency overlaps the rest
            float Ek[kGroup][CPT];
#pragma unroll
            for (int k = 0; k < kGroup; ++k)
#pragma unroll
                for (int j = 0; j < CPT; ++j) Ek[k][j] = ex2(Lk[k][j]);
#pragma unroll
            for (int k = 0; k < kGroup; ++k) {
                f2 b[8];
                load_b(bsrc, t + k, b);
                float u[CPT];
                if constexpr (MIX) {
                    uint32_t xw[CPT / 2];
                    load_words<CPT>(st + lay.xs + ((t + k) * DS + dl) * C::SZ, xw);
#pragma unroll
                    for (int i = 0; i < CPT / 2; ++i) {
                        u[2 * i] = mul_bf16_lo(dw[k][i], xw[i]);
                        u[2 * i + 1] = mul_bf16_hi(dw[k][i], xw[i]);
                    }
                } else {
                    float xv[CPT];
                    uint32_t nx;
                    load_chan<TIn, CPT>(st + lay.xs + ((t + k) * DS + dl) * C::SZ, xv, nx);
#pragma unroll
                    for (int j = 0; j < CPT; ++j) u[j] = dvk[k][j] * xv[j];
                }
#pragma unroll
                for (int j = 0; j < CPT; ++j) accumulate_e(g[j], b, u[j], Ek[k][j]);
            }
#pragma unroll
            for (int j = 0; j < CPT; ++j) L[j] = Lk[kGroup - 1][j];
        }
    }
    for (; t < ntok; ++t) {
        f2 b[8];
        float xv[CPT], dv[CPT];
        uint32_t n0;
        load_b(bsrc, t, b);
        load_chan<TIn, CPT>(st + lay.xs + (t * DS + dl) * C::SZ, xv, n0);
        load_chan<TIn, CPT>(st + lay.dts + (t * DS + dl) * C::SZ, dv, n0);
        if constexpr (C::SPLIT) {
#pragma unroll
            for (int j = 0; j < CPT; ++j) tot[j] += dv[j];
        }
        token_checked<CPT>(g, L, kk, b, xv, dv, wmask);
    }
}

// ---------------------------------------------------------------------------
// Chunks split over the CTAs of a cluster (captures with few work items). The recurrence is
// linear in the state, so a chunk's final state is the sum over its segments of the
// segment's own final state (from zero) decayed by the tokens after it:
//   h[d, n] = sum_s 2^(A[d, n] log2 e * (dt summed over the segments after s)) h_s[d, n].
// Every CTA leaves its h_s and its sum of dt in its shared memory; the cluster's threads
// share the (channel, 4 states) sums, each from the last segment back, and write the states. Each
// segment's sum is relative to its own tokens, so a factor far below 1 belongs to a state
// that no longer matters and the rounding of its exponent is scaled down with it. Modes that grow
// (a negative sum of dt, or A > 0) may have factors beyond fp32's range where the state is zero or
// small enough to stay finite; those sums are formed again with fma_exp2. (Redoing the rare
// sum costs the usual one nothing, 24 layers x 3 x 500 tokens 30.7 us; a choice per factor
// inside it took 31.9 to 34.8 us.)
struct SplitSmem {
    int32_t dead;      // this CTA gave up on a wait
    int32_t pad[31];
    // followed by float4 h[4][DS] (states 4q..4q+3 of a channel) and float dt_sum[DS]
};

template <class C>
__device__ __forceinline__ void combine(unsigned char *buf, const ScanParams &p, int segs, int DS, int dl, bool dead,
                                        const f2 (&h)[C::CPT][8], const float (&tot)[C::CPT], int64_t chunk,
                                        int layer, int d0) {
    SplitSmem &sm = *reinterpret_cast<SplitSmem *>(buf);
    float4 *hs = reinterpret_cast<float4 *>(buf + sizeof(SplitSmem));
    float *ts = reinterpret_cast<float *>(hs + 4 * DS);
    if (threadIdx.x == 0) sm.dead = dead;
#pragma unroll
    for (int j = 0; j < C::CPT; ++j) {
        ts[dl + j] = tot[j];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            float4 v;
            unpack2(h[j][2 * q], v.x, v.y);
            unpack2(h[j][2 * q + 1], v.z, v.w);
            hs[q * DS + dl + j] = v;
        }
    }
    cluster_sync_all();
    bool any_dead = false;
    for (int s = 0; s < segs; ++s) any_dead |= ld_cluster_u32(mapa_shared(&sm.dead, s)) != 0u;
    const int rank = static_cast<int>(cluster_ctarank()), nthr = blockDim.x;
    const float *Al = p.A + static_cast<int64_t>(layer) * p.D * kN;
    for (int i = rank * nthr + threadIdx.x; i < 4 * DS && !any_dead; i += segs * nthr) {
        const int q = i / DS, ch = i % DS;
        if (d0 + ch >= p.D) continue;
        const float4 a = *reinterpret_cast<const float4 *>(Al + static_cast<int64_t>(d0 + ch) * kN + 4 * q);
        // (finite, so that a mode without memory, A = -inf, times no dt is no decay)
        const auto coeff = [](float x) { return fminf(fmaxf(x * kLog2e, -FLT_MAX), FLT_MAX); };
        const float c[4] = {coeff(a.x), coeff(a.y), coeff(a.z), coeff(a.w)};
        float after = 0.f;   // dt summed over the segments after the current one
        float most = 0.f, least = 0.f;
        float sum[4] = {0.f, 0.f, 0.f, 0.f};
        for (int s = segs - 1; s >= 0; --s) {
            const float4 v = ld_cluster_f4(mapa_shared(&hs[q * DS + ch], s));
            const float hv[4] = {v.x, v.y, v.z, v.w};
            most = fmaxf(most, after);
            least = fminf(least, after);
#pragma unroll
            for (int k = 0; k < 4; ++k) sum[k] = fmaf(ex2(c[k] * after), hv[k], sum[k]);
            after += __uint_as_float(ld_cluster_u32(mapa_shared(&ts[ch], s)));
        }
        const float chigh = fmaxf(fmaxf(c[0], c[1]), fmaxf(c[2], c[3])), clow = fminf(fminf(c[0], c[1]), fminf(c[2], c[3]));
        if (fmaxf(fmaxf(chigh * most, chigh * least), fmaxf(clow * most, clow * least)) > kExp2Near) {
            // once more (the usual sum above has no branches)
            after = sum[0] = sum[1] = sum[2] = sum[3] = 0.f;
#pragma unroll 1
            for (int s = segs - 1; s >= 0; --s) {
                const float4 v = ld_cluster_f4(mapa_shared(&hs[q * DS + ch], s));
                const float hv[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
                for (int k = 0; k < 4; ++k) sum[k] = fma_exp2(hv[k], c[k] * after, sum[k]);
                after += __uint_as_float(ld_cluster_u32(mapa_shared(&ts[ch], s)));
            }
        }
        const int64_t off = ((chunk * p.L_out + p.layer0 + layer) * static_cast<int64_t>(p.D) + d0 + ch) * kN + 4 * q;
        if (p.state_dtype == PRECOG_F32) {
            *reinterpret_cast<float4 *>(static_cast<float *>(p.states) + off) = make_float4(sum[0], sum[1], sum[2], sum[3]);
        } else {
            __nv_bfloat162 lo = __floats2bfloat162_rn(sum[0], sum[1]), hi = __floats2bfloat162_rn(sum[2], sum[3]);
            *reinterpret_cast<uint2 *>(static_cast<__nv_bfloat16 *>(p.states) + off) =
                make_uint2(*reinterpret_cast<uint32_t *>(&lo), *reinterpret_cast<uint32_t *>(&hi));
        }
    }
    cluster_sync_all();   // no CTA leaves while another may still read its shared memory
}

template <class C>
__global__ void __launch_bounds__(C::LB_THREADS, C::LB_BLOCKS)
    scan_kernel(const ScanParams p, const int DS_arg, const int slices, const __grid_constant__ SliceMaps maps) {
    if constexpr (C::HAS_H0) grid_dependency_wait();
    using TIn = typename C::TIn;
    const int DS = C::FIXDS ? C::FIXDS : DS_arg;
    constexpr int CPT = C::CPT, TILE = C::TILE, STAGES = C::STAGES, SZ = C::SZ;
    extern __shared__ __align__(128) unsigned char smem[];
    uint64_t *full = reinterpret_cast<uint64_t *>(smem);
    unsigned char *stage0 = smem + kBarBytes;
    const StageLayout lay = stage_layout(TILE, DS, SZ, C::HAS_Y, C::CONV);
    const int tid = threadIdx.x;
    const int nthr = blockDim.x;

    // ---- work item ----
    int64_t item = C::SPLIT ? blockIdx.x / p.segments : blockIdx.x;
    const int slice = static_cast<int>(item % slices);
    item /= slices;
    const int64_t chunk = p.order ? p.order[item % p.n_chunks] : item % p.n_chunks;
    if (chunk < 0 || chunk >= p.n_chunks) {  // an order entry outside the chunks: skipped
        if (threadIdx.x == 0) atomicOr(&g_scan_status, PRECOG_DEV_BAD_INDEX);
        return;
    }
    const int layer = static_cast<int>(item / p.n_chunks);
    // a last slice narrower than the others leaves its upper threads without channels
    const bool live = C::FIXDS || slice * DS + static_cast<int>(threadIdx.x) * CPT < p.D;
    // this thread's rows of A first (16 floats each, 16-byte loads): their latency overlaps
    // the chunk's offsets below
    float a_rows[CPT][kN];
    {
        const float *Al0 = p.A + static_cast<int64_t>(layer) * p.D * kN;
#pragma unroll
        for (int j = 0; j < CPT; ++j) {
            const float4 *a4 = reinterpret_cast<const float4 *>(
                Al0 + static_cast<int64_t>(slice * DS + static_cast<int>(threadIdx.x) * CPT + j) * kN);
#pragma unroll
            for (int q = 0; q < kN / 4; ++q) {
                const float4 v = live ? a4[q] : make_float4(0.f, 0.f, 0.f, 0.f);
                a_rows[j][4 * q] = v.x;
                a_rows[j][4 * q + 1] = v.y;
                a_rows[j][4 * q + 2] = v.z;
                a_rows[j][4 * q + 3] = v.w;
            }
        }
    }
    int64_t start, len;
    if (p.use_fixed) {
        start = chunk * p.fixed_len;
        len = p.fixed_len;
    } else {
        start = p.offsets[chunk];
        const int64_t end = p.offsets[chunk + 1];
        if (start < 0 || end < start || end > p.T_tot) {
            if (tid == 0) atomicOr(&g_scan_status, PRECOG_DEV_BAD_OFFSETS);
            return;
        }
        len = end - start;
    }
    if constexpr (C::SPLIT) {
        // this CTA's share of the chunk: whole tiles (the cluster's CTAs left together above)
        const int64_t share = ((len + TILE - 1) / TILE + p.segments - 1) / p.segments * TILE;
        const int64_t skip = share * cluster_ctarank();
        start += skip;
        len = len > skip ? min64(len - skip, share) : 0;
    }
    TrajCursor tcur{};
    if constexpr (C::TRAJ) {
        // chunk c keeps ceil(len / stride) states starting at entry traj_offsets[c]
        const int64_t e0 = p.traj_offsets[chunk], e1 = p.traj_offsets[chunk + 1];
        if (e1 - e0 != (len + p.traj_stride - 1) / p.traj_stride) {
            if (tid == 0) atomicOr(&g_scan_status, PRECOG_DEV_BAD_OFFSETS);
            return;
        }
        tcur.entry = e0;
        tcur.left = p.traj_stride;
        const int wc = 32 * CPT, w0 = slice * DS + tid / 32 * wc;   // the warp's channels
        const int row_end = p.D - slice * DS < DS ? p.D : slice * DS + DS;
        tcur.first = w0;
        tcur.channels = row_end - w0 < wc ? row_end - w0 : wc;
        tcur.bufs = stage0 + STAGES * lay.bytes + tid / 32 * traj_buffer_bytes(CPT);
    }
    const int d0 = slice * DS;
    const int dl = tid * CPT;
    const int D = p.D;
    const TIn *xl = static_cast<const TIn *>(p.x) + layer * p.ls_xd;
    const TIn *dtl = static_cast<const TIn *>(p.dt) + layer * p.ls_xd;
    const TIn *Bl = static_cast<const TIn *>(p.B) + layer * p.ls_bc;
    const TIn *Cl = C::HAS_Y ? static_cast<const TIn *>(p.C) + layer * p.ls_bc : nullptr;

    // ---- coefficients; kPower verifies the structure (A[d, n] = (n + 1) A[d, 0] <= 0) ----
    float kpow[CPT];      // A[d, 0] * log2 e
    f2 kgen[CPT][8];      // (A[d, n] * log2 e) pairs, kGeneral only
    bool a_ok = true;
#pragma unroll
    for (int j = 0; j < CPT; ++j) {
        const float (&a)[kN] = a_rows[j];
        kpow[j] = a[0] * kLog2e;
        if constexpr (C::MODE == kGeneral) {
#pragma unroll
            for (int i = 0; i < 8; ++i) kgen[j][i] = pack2(a[2 * i] * kLog2e, a[2 * i + 1] * kLog2e);
        } else {
            a_ok &= a[0] <= 0.f;
#pragma unroll
            for (int n = 1; n < kN; ++n) a_ok &= a[n] == static_cast<float>(n + 1) * a[0];
        }
    }
    if constexpr (C::WIDE_CHECK) {
        if (DS == kMaxSlice && D % kWideSlice == 0) {
            const float4 *a4 = reinterpret_cast<const float4 *>(
                p.A + (static_cast<int64_t>(layer) * D + (slice ^ 1) * DS + dl) * kN);
#pragma unroll
            for (int j = 0; j < CPT; ++j) {
                const float a0 = a4[j * (kN / 4)].x;
                a_ok &= a0 <= 0.f;
#pragma unroll
                for (int q = 0; q < kN / 4; ++q) {
                    const float4 v = a4[j * (kN / 4) + q];
                    const float n = static_cast<float>(4 * q + 1);
                    a_ok &= v.x == n * a0 && v.y == (n + 1.f) * a0 && v.z == (n + 2.f) * a0 && v.w == (n + 3.f) * a0;
                }
            }
        }
    }
    if constexpr (C::MODE == kPower) {
        if (!__syncthreads_and(a_ok)) {
            if (tid == 0) atomicOr(&g_scan_status, PRECOG_DEV_BAD_A);
            return;
        }
    }

    // ---- pipeline start: barrier init, first STAGES tiles in flight ----
    const int64_t ntiles = (len + TILE - 1) / TILE;
    if (tid == 0) {
        for (int s = 0; s < STAGES; ++s) mbar_init(&full[s], 1);
        fence_barrier_init();
    }
    __syncthreads();
    auto issue = [&](int64_t k) {  // thread 0 only
        const int s = static_cast<int>(k % STAGES);
        unsigned char *st = stage0 + s * lay.bytes;
        const int64_t row0 = start + k * TILE;
        const int ntok = static_cast<int>(min64(TILE, len - k * TILE));
        const uint32_t rowb = DS * SZ;
        const uint32_t bytes = ntok * rowb * 2 + ntok * kN * SZ * (C::HAS_Y ? 2 : 1);
        if (DS == D) {
            mbar_arrive_expect_tx(&full[s], bytes);
            bulk_g2s(st + lay.xs, xl + row0 * D, ntok * rowb, &full[s]);
            bulk_g2s(st + lay.dts, dtl + row0 * D, ntok * rowb, &full[s]);
        } else if (maps.valid) {
            // the slice of TILE rows as one tensor-map copy per tensor (a box always moves
            // TILE rows; rows past the end of the tensor arrive as zeros)
            mbar_arrive_expect_tx(&full[s], bytes + (TILE - ntok) * rowb * 2);
            const bool even = C::FIXDS || maps.inner;
            const int c0 = even ? 0 : d0, c1 = even ? d0 / maps.inner : 0;
            tma_load_4d(st + lay.xs, &maps.x, c0, c1, static_cast<int32_t>(row0), layer, &full[s]);
            tma_load_4d(st + lay.dts, &maps.dt, c0, c1, static_cast<int32_t>(row0), layer, &full[s]);
        } else {
            const uint32_t ownb = !C::FIXDS && D - d0 < DS ? (D - d0) * SZ : rowb;   // the slice's part of the row
            mbar_arrive_expect_tx(&full[s], bytes - ntok * (rowb - ownb) * 2);
            for (int r = 0; r < ntok; ++r) {
                bulk_g2s(st + lay.xs + r * rowb, xl + (row0 + r) * D + d0, ownb, &full[s]);
                bulk_g2s(st + lay.dts + r * rowb, dtl + (row0 + r) * D + d0, ownb, &full[s]);
            }
        }
        bulk_g2s(st + lay.bs, Bl + row0 * kN, ntok * kN * SZ, &full[s]);
        if (C::HAS_Y) bulk_g2s(st + lay.cs, Cl + row0 * kN, ntok * kN * SZ, &full[s]);
    };
    if (tid == 0)
        for (int64_t k = 0; k < min64(STAGES, ntiles); ++k) issue(k);

    // ---- initial state (overlaps the first copies) ----
    f2 h[CPT][8];
    bool h0_valid = false;
    int64_t h0_row = 0;
    if constexpr (C::HAS_H0) {
        if (p.topk <= 1) {
            h0_row = p.idx ? p.idx[chunk] : chunk;
            h0_valid = h0_row >= 0 && h0_row < p.bank_entries;
            if (!h0_valid && !(p.idx && h0_row == -1) && tid == 0)
                atomicOr(&g_scan_status, PRECOG_DEV_BAD_INDEX);
        }
    }
#pragma unroll
    for (int j = 0; j < CPT; ++j) {
        if (C::HAS_H0 && h0_valid && live) {
            const int64_t off =
                ((h0_row * p.L_bank + p.layer0 + layer) * static_cast<int64_t>(D) + d0 + dl + j) * kN;
            load_state16(p.bank, p.bank_dtype, off, h[j]);
        } else {
#pragma unroll
            for (int i = 0; i < 8; ++i) h[j][i] = 0;
        }
    }
    if constexpr (C::HAS_H0) {
        if (p.topk > 1) {
            // Top-k composition (Sec. 4.4, Eq. smc-fusion): h_init = sum_j w_j bank[row_j],
            // w = softmax(score / temperature) over the valid rows (row -1 or a NaN score:
            // weight 0; a row outside the bank: weight 0 and PRECOG_DEV_BAD_INDEX).
            const int64_t *rows = p.idx + chunk * p.topk;
            const float *sc = p.topk_scores + chunk * p.topk;
            float w[kMaxTopk];
            float smax = -__int_as_float(0x7f800000);
#pragma unroll
            for (int k = 0; k < kMaxTopk; ++k) {
                w[k] = -__int_as_float(0x7f800000);
                if (k < p.topk) {
                    const int64_t r = rows[k];
                    const bool in_bank = r >= 0 && r < p.bank_entries;
                    if (!in_bank && r != -1 && tid == 0) atomicOr(&g_scan_status, PRECOG_DEV_BAD_INDEX);
                    const float z = sc[k] * p.inv_temp;
                    if (in_bank && !isnan(z)) {
                        w[k] = z;
                        smax = fmaxf(smax, z);
                    }
                }
            }
            float wsum = 0.f;
#pragma unroll
            for (int k = 0; k < kMaxTopk; ++k) {
                w[k] = (w[k] == -__int_as_float(0x7f800000)) ? 0.f : ex2((w[k] - smax) * kLog2e);
                wsum += w[k];
            }
#pragma unroll
            for (int k = 0; k < kMaxTopk; ++k) {
                if (k >= p.topk || w[k] == 0.f) continue;
                const float wk = w[k] / wsum;
                const f2 ww = pack2(wk, wk);
#pragma unroll
                for (int j = 0; live && j < CPT; ++j) {
                    f2 hk[8];
                    const int64_t off = ((rows[k] * p.L_bank + p.layer0 + layer) * static_cast<int64_t>(D) +
                                         d0 + dl + j) * kN;
                    load_state16(p.bank, p.bank_dtype, off, hk);
#pragma unroll
                    for (int i = 0; i < 8; ++i) h[j][i] = fma2(ww, hk[i], h[j][i]);
                }
            }
        }
    }
    const unsigned wmask = __activemask();
    float Lw[CPT], kk[CPT], tot[CPT];
    bool dead = false;
#pragma unroll
    for (int j = 0; j < CPT; ++j) {
        tot[j] = 0.f;
        Lw[j] = 0.f;
        kk[j] = -kpow[j];
    }

    // ---- time loop ----
    void *yrow = nullptr;
    const int64_t y_stride = D;
    if (C::HAS_Y) {
        const int64_t off = (static_cast<int64_t>(layer) * p.T_tot + start) * D + d0 + dl;
        yrow = (p.y_dtype == PRECOG_F32) ? static_cast<void *>(static_cast<float *>(p.y) + off)
                                         : static_cast<void *>(static_cast<__nv_bfloat16 *>(p.y) + off);
    }
    for (int64_t k = 0; k < ntiles; ++k) {
        const int s = static_cast<int>(k % STAGES);
        const uint32_t par = static_cast<uint32_t>((k / STAGES) & 1);
        unsigned char *st = stage0 + s * lay.bytes;
        const int ntok = static_cast<int>(min64(TILE, len - k * TILE));
        const bool ok = mbar_wait(&full[s], par);
        if (C::CONV && ok) {
            const TIn *bsrc = reinterpret_cast<const TIn *>(st + lay.bs);
            float *bdst = reinterpret_cast<float *>(st + lay.bf);
            if constexpr (std::is_same<TIn, __nv_bfloat16>::value) {
                // four values per thread and step: one 8-byte read, one 16-byte write
                for (int i = tid * 4; i < ntok * kN; i += nthr * 4) {
                    const uint2 w = *reinterpret_cast<const uint2 *>(bsrc + i);
                    *reinterpret_cast<float4 *>(bdst + i) =
                        make_float4(__uint_as_float(w.x << 16), __uint_as_float(w.x & 0xffff0000u),
                                    __uint_as_float(w.y << 16), __uint_as_float(w.y & 0xffff0000u));
                }
            } else {
                for (int i = tid; i < ntok * kN; i += nthr) bdst[i] = to_f32(bsrc[i]);
            }
            if (C::HAS_Y) {
                const TIn *csrc = reinterpret_cast<const TIn *>(st + lay.cs);
                float *cdst = reinterpret_cast<float *>(st + lay.cf);
                if constexpr (std::is_same<TIn, __nv_bfloat16>::value) {
                    for (int i = tid * 4; i < ntok * kN; i += nthr * 4) {
                        const uint2 w = *reinterpret_cast<const uint2 *>(csrc + i);
                        *reinterpret_cast<float4 *>(cdst + i) =
                            make_float4(__uint_as_float(w.x << 16), __uint_as_float(w.x & 0xffff0000u),
                                        __uint_as_float(w.y << 16), __uint_as_float(w.y & 0xffff0000u));
                    }
                } else {
                    for (int i = tid; i < ntok * kN; i += nthr) cdst[i] = to_f32(csrc[i]);
                }
            }
        }
        if (!__syncthreads_and(ok)) {
            // Give up on this chunk: record it, let issued copies land, leave.
            if (tid == 0) {
                atomicOr(&g_scan_status, PRECOG_DEV_TIMEOUT);
                for (int64_t k2 = k; k2 < min64(k + STAGES, ntiles); ++k2)
                    mbar_wait(&full[k2 % STAGES], static_cast<uint32_t>((k2 / STAGES) & 1));
            }
            if constexpr (C::STAGED) {
                if ((tid & 31) == 0) bulk_wait_all();
            }
            if constexpr (!C::SPLIT) return;
            dead = true;   // the cluster's other CTAs still expect this one at their barriers
            break;
        }
        if constexpr (C::RESCALED && C::TRAJ == kTrajRescaled) {
            // segments end at the trajectory points; there the state is brought back
            // to h (renormalised, L = 0), stored, and the accumulation continues
            int t = 0;
            while (t < ntok) {
                const int seg = static_cast<int>(min64(ntok - t, tcur.left));
                scan_tile_rescaled<C>(st, lay, reinterpret_cast<const float *>(st + (C::CONV ? lay.bf : lay.bs)), DS, dl, t,
                                      t + seg, h, Lw, kk, wmask, tot);
                t += seg;
                tcur.left -= seg;
                if (tcur.left == 0 || k * TILE + t == len) {
#pragma unroll
                    for (int j = 0; j < CPT; ++j) renormalise(h[j], Lw[j]);
                    const int64_t row = (tcur.entry * p.L_out + p.layer0 + layer) * static_cast<int64_t>(D);
                    if constexpr (C::STAGED) {
                        store_trajectory<CPT>(tcur.bufs, tcur.which, tid & 31, tcur.channels, p.traj, p.traj_dtype,
                                              (row + tcur.first) * kN, h);
                    } else {
#pragma unroll
                        for (int j = 0; live && j < CPT; ++j)
                            store_state16(p.traj, p.traj_dtype, (row + d0 + dl + j) * kN, h[j]);
                    }
                    ++tcur.entry;
                    tcur.left = p.traj_stride;
                }
            }
        } else if constexpr (C::RESCALED) {
            scan_tile_rescaled<C>(st, lay, reinterpret_cast<const float *>(st + (C::CONV ? lay.bf : lay.bs)), DS, dl, 0,
                                  ntok, h, Lw, kk, wmask, tot);
        } else if (C::STAGED || live) {   // (the branch around the loop: in it, it kept tokens apart)
            scan_tile_direct<C>(st, lay, DS, dl, ntok, h, kpow, kgen, yrow, p.y_dtype, y_stride, p, tcur,
                                len - k * TILE, p.layer0 + layer, d0 + dl, tot);
        }
        if (C::HAS_Y) {
            yrow = (p.y_dtype == PRECOG_F32)
                       ? static_cast<void *>(static_cast<float *>(yrow) + TILE * y_stride)
                       : static_cast<void *>(static_cast<__nv_bfloat16 *>(yrow) + TILE * y_stride);
        }
        fence_proxy_async_smem();
        __syncthreads();
        if (tid == 0 && k + STAGES < ntiles) issue(k + STAGES);
    }

    // ---- state capture ----
    if constexpr (C::STAGED) {
        if ((tid & 31) == 0) bulk_wait_all();   // the last states are on their way out of shared memory
        return;
    }
    if constexpr (C::RESCALED) {
#pragma unroll
        for (int j = 0; j < CPT; ++j) renormalise(h[j], Lw[j]);
    }
    if constexpr (C::SPLIT) {
        __syncthreads();
        combine<C>(stage0, p, p.segments, DS, dl, dead, h, tot, chunk, layer, d0);
        return;
    }
    if (p.states && live) {
#pragma unroll
        for (int j = 0; j < CPT; ++j) {
            const int64_t off =
                ((chunk * p.L_out + p.layer0 + layer) * static_cast<int64_t>(D) + d0 + dl + j) * kN;
            store_state16(p.states, p.state_dtype, off, h[j]);
        }
    }
}

// Channel slice of one CTA: the widest of 512 (if maxslice allows it), 256 and 128 channels that
// divides the row; else the whole row if it fits, whatever its length, or the fewest slices of up
// to 256, of equal width up to whole warps of two channels per thread (the last one is narrower:
// its upper threads have no channels). Slices had to be a power of two that divides D, so D = 1000
// or 712 ran 125 or 89 CTAs of two threads per chunk: 2 layers x 400 chunks x 200 tokens bf16,
// D = 1000: capture 3654 -> 225 us, readout 7035 -> 421 us, general A (fp32) 2593 -> 540 us; D = 456:
// 1678 -> 128, 3219 -> 229, 1189 -> 275 us. Equal slices against 256 and a rest: general fp32
// readout of 2 layers x 138 x 687 tokens, D = 320, 298 us against 364. `narrow`: 64 channels.
// For a general A or trajectories in launches that leave SMs idle, so that more SMs share the
// exponentials or the stores (every 8th state of 1 x 40 x 200 tokens, general fp32, D = 320, 37 us,
// equal slices 43; every state of 2 x 3 x 153, bf16 power form, D = 712, 39 us, 101), and for all
// trajectories of a general A, whose deep ring leaves one fp32 CTA of 256 channels to an SM
// (2 x 138 x 687, D = 448, 397 and 557).
int pick_slice(int D, int maxslice, bool narrow) {
    for (int ds = kWideSlice; ds >= 128; ds /= 2)
        if (ds <= maxslice && D % ds == 0) return ds;
    if (D <= maxslice) return D;
    if (narrow) return 64;
    const int n = (D + kMaxSlice - 1) / kMaxSlice, width = (D + n - 1) / n;
    return (width + 63) / 64 * 64;
}

// True when a full-width launch would have fewer CTAs than the device has SMs.
bool few_items(const ScanParams &p) {
    const int sms = device_sm_count();
    const int64_t slices = (p.D + kMaxSlice - 1) / kMaxSlice;
    return static_cast<int64_t>(p.n_layers) * p.n_chunks * slices < sms;
}

// The same by channels, whatever the number of CTAs they make.
bool few_channels(const ScanParams &p) {
    return static_cast<int64_t>(p.n_layers) * p.n_chunks * p.D < static_cast<int64_t>(device_sm_count()) * kMaxSlice;
}

// Whether trajectories with the rescaled update (16-bit inputs) go four channels per thread and
// store plainly, in the captures' shape, or two and staged (launch_pairs), whose tokens cost 5 %
// more. Plain stores pay from strides of 64 with bf16 states and 128 (100 in slices of other than
// 256 channels) with fp32 ones. A CTA of 256 channels is two warps in the first
// shape: an odd number of them per SM leaves two of its four schedulers a warp behind, while
// the second's four warps load all alike; in CTAs of one warp (rows that 128 divides but not
// 256) it is the last round that counts. us, every 250th fp32 state, 152 n CTAs of 256 channels,
// first / second shape: n = 6 (700 tokens) 234 / 245, 7 301 / 281, 12 438 / 462, 20 (420 tokens)
// 435 / 460, 27 (311) 454 / 462; stride 64, n = 8 (600) 297 / 282, bf16 270 / 278. Second / first of
// D = 128: n = 7 0.97, 11 1.02, 21 1.06; D = 64: 0.61; 192: 0.92; 320: 1.03.
bool fits_quads(const ScanParams &p) {
    if (p.D < 256 && p.D % 128 != 0) return false;   // dead lanes
    const int ds = pick_slice(p.D, kWideSlice, false);
    if (p.traj_stride < (p.traj_dtype != PRECOG_F32 ? 64 : ds == 256 ? 128 : 100)) return false;
    const int64_t items = (static_cast<int64_t>(p.n_layers) * p.n_chunks * p.D + kMaxSlice - 1) / kMaxSlice;
    const int64_t per_sm = (items + device_sm_count() - 1) / device_sm_count();
    return ds % 256 == 0 ? per_sm > 2 && 200 * ((per_sm + 1) / 2) <= 105 * per_sm : per_sm > 8;
}

template <class C>
cudaError_t launch_cfg(const ScanParams &p, cudaStream_t stream) {
    const bool idle = !C::SPLIT && (C::MODE == kGeneral || C::TRAJ != kTrajNone) && few_channels(p);
    const int DS = C::FIXDS ? C::FIXDS : pick_slice(p.D, C::MAXSLICE, idle || (C::MODE == kGeneral && C::TRAJ != kTrajNone));
    if (DS % C::CPT != 0 || (C::FIXDS && p.D % DS != 0)) return cudaErrorInvalidValue;
    const int slices = (p.D + DS - 1) / DS;
    const StageLayout lay = stage_layout(C::TILE, DS, C::SZ, C::HAS_Y, C::CONV);
    const int warps = (DS / C::CPT + 31) / 32;
    const size_t smem = kBarBytes + static_cast<size_t>(C::STAGES) * lay.bytes +
                        (C::STAGED ? warps * traj_buffer_bytes(C::CPT) : 0);
    const int64_t items = static_cast<int64_t>(p.n_layers) * p.n_chunks * slices;
    if (items == 0) return cudaSuccess;
    if (items > 0x7fffffffLL) return cudaErrorInvalidConfiguration;
    SliceMaps maps{};
    if (DS < p.D) {
        // slices that divide the row: [layer][row][D / inner][inner], a box of whole inner rows;
        // else [layer][row][1][D], a box from channel d0 (channels past the row arrive as zeros)
        const bool even = p.D % DS == 0;
        const int inner = even ? (DS < 256 ? DS : 256) : p.D;
        const cuuint64_t rows = static_cast<cuuint64_t>(p.T_tot);
        const cuuint64_t dims[4] = {static_cast<cuuint64_t>(inner), static_cast<cuuint64_t>(p.D / inner), rows,
                                    static_cast<cuuint64_t>(p.n_layers)};
        const cuuint64_t lstride = static_cast<cuuint64_t>(p.n_layers > 1 ? p.ls_xd : rows * p.D) * C::SZ;
        const cuuint64_t strides[3] = {static_cast<cuuint64_t>(inner) * C::SZ, static_cast<cuuint64_t>(p.D) * C::SZ,
                                       lstride};
        const cuuint32_t box[4] = {static_cast<cuuint32_t>(DS < 256 ? DS : 256), static_cast<cuuint32_t>(even ? DS / inner : 1),
                                   static_cast<cuuint32_t>(C::TILE), 1};
        const CUtensorMapDataType dt = C::SZ == 4 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT32 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16;
        maps.valid = encode_tiled_map(&maps.x, dt, 4, p.x, dims, strides, box, CU_TENSOR_MAP_SWIZZLE_NONE) &&
                     encode_tiled_map(&maps.dt, dt, 4, p.dt, dims, strides, box, CU_TENSOR_MAP_SWIZZLE_NONE);
        maps.inner = even ? inner : 0;
    }
    auto kern = scan_kernel<C>;
    cudaError_t e = ensure_smem(reinterpret_cast<const void *>(kern), static_cast<int>(smem));
    if (e != cudaSuccess) return e;
    if constexpr (C::SPLIT) {
        if (items * p.segments > 0x7fffffffLL) return cudaErrorInvalidConfiguration;
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(static_cast<unsigned>(items * p.segments));
        cfg.blockDim = dim3(static_cast<unsigned>(DS / C::CPT));
        cfg.dynamicSmemBytes = smem;
        cfg.stream = stream;
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = static_cast<unsigned>(p.segments);
        attr[0].val.clusterDim.y = 1;
        attr[0].val.clusterDim.z = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        e = cudaLaunchKernelEx(&cfg, kern, p, DS, slices, maps);
    } else if constexpr (C::HAS_H0) {
        // a prefill, usually behind the retrieval of its rows
        e = launch_dependent(kern, dim3(static_cast<unsigned>(items)), dim3(DS / C::CPT), smem, stream, p, DS, slices, maps);
    } else {
        kern<<<static_cast<unsigned>(items), DS / C::CPT, smem, stream>>>(p, DS, slices, maps);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) count_launches(1);
    return e;
}

// CTAs per chunk of a capture (8 or 4; 1: not split). One CTA takes 0.09 (fp32) to 0.14 us per
// token whatever else runs, so a launch that leaves SMs without a CTA or with one is as long as its
// chunks. A split launch has `segs` times the CTAs, each with its ring, its rows of A and its
// part of the combination, and with fp32 inputs only three of them fit an SM; so the chunks must
// be the longer, the more CTAs an SM would get: at least kPerChannels tokens per 256
// channels and kPerCta per CTA on an SM, and 80. us, unsplit / split as chosen (bf16 power):
// 24 layers x 3 chunks x 500 tokens 70 / 27, 1 x 1 x 4096 517 / 60, 24 x 9 x 500 72 / 60, but
// 24 x 9 x 128 23 / 25 in four shares; fp32 24 x 5 x 80 12.4 / 22.5, general fp32 4 layers x 9 x
// 80 tokens x 1000 channels 14.5 / 26.4: not split. Of 760 sizes of each kind (1 to 48 layers of
// 8 to 2048 channels, 80 to 1000 tokens) 6 to 16 take longer than unsplit now, by at most 18 to
// 37 %, where a threshold of 80 tokens for all made it 78 to 244, up to 2.7 times.
template <class C>
int split_segments(const ScanParams &p) {
    constexpr bool f32 = std::is_same<typename C::TIn, float>::value;
    constexpr int64_t kPerChannels = C::MODE == kGeneral ? 40 : f32 ? 70 : 30, kPerCta = C::MODE == kPower && !f32 ? 5 : 15;
    const int64_t sms = device_sm_count();
    const int DS = pick_slice(p.D, C::MAXSLICE, false);
    const int64_t pieces = static_cast<int64_t>(p.n_layers) * p.n_chunks;
    const int64_t ctas = pieces * ((p.D + DS - 1) / DS), full = (pieces * p.D + kMaxSlice - 1) / kMaxSlice;
    const int64_t tokens = p.T_tot / p.n_chunks;   // of a chunk on average: the offsets are on the device
    if (tokens < 80 || 2 * full > 3 * sms) return 1;
    for (int segs = 8; segs >= 4; segs /= 2)
        if (full * segs <= 6 * sms && tokens >= segs * C::TILE && tokens * sms >= (kPerChannels * full + kPerCta * ctas) * segs)
            return segs;
    return 1;
}

// Two channels per thread: power-form A with fp32 inputs, and trajectories that fill the SMs. The
// ring of 256 fp32 channels takes 68 KB, so three CTAs share an SM whatever their registers, and
// with two channels per thread they are 12 warps instead of 6: 1 layer x 500 chunks x 1000 tokens
// capture 274 -> 231 us, 1 x 100 x 300 x 2048 144 -> 112; readout 24 x 30 x 500 370 -> 290,
// 1 x 100 x 300 x 2048 276 -> 215. The buffers of staged trajectories leave two CTAs of fp32 inputs
// and four of bf16 ones (16 warps, 122 registers). bf16 captures and readouts keep four channels per
// thread (in this shape 215 -> 234 us and 190 -> 209).
template <typename TIn, bool HAS_Y, bool HAS_H0, int TRAJ>
cudaError_t launch_pairs(const ScanParams &p, cudaStream_t stream) {
    if (p.D % kMaxSlice == 0)
        return launch_cfg<Cfg<TIn, HAS_Y, HAS_H0, kPower, 2, 16, 2, 4, TRAJ, kMaxSlice, kMaxSlice, false, true>>(p, stream);
    return launch_cfg<Cfg<TIn, HAS_Y, HAS_H0, kPower, 2, 16, 2, 4, TRAJ, kMaxSlice, 0, false, true>>(p, stream);
}

// Shapes: the rescaled capture kernel (the corpus-encode hot loop) and the
// direct kernels (readout, prefill, general A).
template <typename TIn, bool HAS_Y, bool HAS_H0, int MODE, int TRAJ = kTrajNone>
cudaError_t launch_t(const ScanParams &p, cudaStream_t stream) {
    if constexpr (TRAJ != kTrajNone) {
        // power form: the rescaled or (short strides) the direct update, in the fp32 shape but
        // for wide strides of 16-bit inputs where the captures' shape is faster (fits_quads)
        if constexpr (MODE == kPower) {
            if constexpr (TRAJ == kTrajRescaled && !std::is_same<TIn, float>::value)
                if (fits_quads(p))
                    return p.D % 256 == 0 && p.D % 512 != 0
                               ? launch_cfg<Cfg<TIn, false, false, kPower, PRECOG_RESCALED_CPT, PRECOG_RESCALED_TILE,
                                                PRECOG_RESCALED_STAGES, PRECOG_RESCALED_MINB, TRAJ, kWideSlice, 256>>(p, stream)
                               : launch_cfg<Cfg<TIn, false, false, kPower, PRECOG_RESCALED_CPT, PRECOG_RESCALED_TILE,
                                                PRECOG_RESCALED_STAGES, PRECOG_RESCALED_MINB, TRAJ, kWideSlice>>(p, stream);
            // (launches that do not fill the SMs store plainly: each staged state adds to the
            // chain of a lone warp, 24 x 1 x 250 x 64, every state: 57 us, 71)
            if (few_channels(p)) return launch_cfg<Cfg<TIn, false, false, MODE, 2, 16, 2, 5, TRAJ, kMaxSlice>>(p, stream);
            return launch_pairs<TIn, false, false, TRAJ>(p, stream);
        } else {
            if (p.D % 256 == 0)
                return launch_cfg<Cfg<TIn, false, false, MODE, 2, 16, 4, 3, kTrajDirect, kMaxSlice, 256>>(p, stream);
            return launch_cfg<Cfg<TIn, false, false, MODE, 2, 16, 4, 3, kTrajDirect>>(p, stream);
        }
    } else if constexpr (MODE == kPower && !HAS_Y) {
        if constexpr (std::is_same<TIn, float>::value) {
            return launch_pairs<TIn, HAS_Y, HAS_H0, kTrajNone>(p, stream);
        } else {
            // the corpus encode of 256- and 512-channel slices (the paper's layer width, the
            // ragged and wide workloads' slices) gets the slice fixed at compile time
            if constexpr (!HAS_H0) {
                const int ds = pick_slice(p.D, kWideSlice, false);
                if (ds == 256 && p.D % 256 == 0)
                    return launch_cfg<Cfg<TIn, false, false, MODE, PRECOG_RESCALED_CPT, PRECOG_RESCALED_TILE,
                                          PRECOG_RESCALED_STAGES, PRECOG_RESCALED_MINB, kTrajNone, kWideSlice, 256>>(
                        p, stream);
                if (ds == 512)
                    return launch_cfg<Cfg<TIn, false, false, MODE, PRECOG_RESCALED_CPT, PRECOG_RESCALED_TILE,
                                          PRECOG_RESCALED_STAGES, PRECOG_RESCALED_MINB, kTrajNone, kWideSlice, 512>>(
                        p, stream);
            }
            return launch_cfg<Cfg<TIn, HAS_Y, HAS_H0, MODE, PRECOG_RESCALED_CPT, PRECOG_RESCALED_TILE,
                                  PRECOG_RESCALED_STAGES, PRECOG_RESCALED_MINB, kTrajNone, kWideSlice>>(p, stream);
        }
    } else {
        if constexpr (MODE == kPower) {
            // Fewer work items than SMs (a single query's prefill: one CTA per layer) is a
            // latency-bound launch: the latency-shaped kernel splits every channel's states
            // over four threads; shapes it does not take run two channels per thread.
            if (few_items(p)) {
                if (scan_latency_eligible(p)) return launch_scan_latency(p, stream);
                return launch_cfg<Cfg<TIn, HAS_Y, HAS_H0, MODE, 2, 16, 2, 3>>(p, stream);
            }
            if constexpr (std::is_same<TIn, float>::value) {
                return launch_pairs<TIn, HAS_Y, HAS_H0, kTrajNone>(p, stream);
            } else {
                // 16-bit rows: 256- and 512-channel slices fixed at compile time
                const int ds = pick_slice(p.D, kWideSlice, false);
                if (ds == 256 && p.D % 256 == 0)
                    return launch_cfg<Cfg<TIn, HAS_Y, HAS_H0, MODE, PRECOG_DIRECT_CPT, PRECOG_DIRECT_TILE,
                                          PRECOG_DIRECT_STAGES, PRECOG_DIRECT_MINB, kTrajNone, kWideSlice, 256>>(
                        p, stream);
                if (ds == 512)
                    return launch_cfg<Cfg<TIn, HAS_Y, HAS_H0, MODE, PRECOG_DIRECT_CPT, PRECOG_DIRECT_TILE,
                                          PRECOG_DIRECT_STAGES, PRECOG_DIRECT_MINB, kTrajNone, kWideSlice, 512>>(
                        p, stream);
                return launch_cfg<Cfg<TIn, HAS_Y, HAS_H0, MODE, PRECOG_DIRECT_CPT, PRECOG_DIRECT_TILE,
                                      PRECOG_DIRECT_STAGES, PRECOG_DIRECT_MINB, kTrajNone, kWideSlice>>(p, stream);
            }
        } else {
            // general A keeps 16 exponent coefficients per channel: 2 channels per thread. The
            // more CTAs share an SM's SFU (the bound: 16 exponentials per channel-token) the better:
            // with two stages and 128 registers four of bf16 inputs and three of fp32 ones (68 KB
            // rings), with four stages three (readouts two) and one. 4 layers x 1000 chunks x 500
            // tokens fp32 1524 -> 1070 us, bf16 1096 -> 1032, with readout 2126 -> 1419 and 1721 ->
            // 1443. Launches that do not fill the SMs keep the deeper ring and the registers (bf16
            // readout 24 x 3 x 500: 93 us, 102; state-only prefill 24 x 1 x 500 x 64 channels: 59, 65;
            // fp32 capture 24 x 7 x 79 x 64: 13.4, 14.4).
            if (few_channels(p))
                return p.D % 256 == 0
                           ? launch_cfg<Cfg<TIn, HAS_Y, HAS_H0, MODE, 2, 16, 4, 3, kTrajNone, kMaxSlice, 256>>(p, stream)
                           : launch_cfg<Cfg<TIn, HAS_Y, HAS_H0, MODE, 2, 16, 4, 3>>(p, stream);
            if (p.D % 256 == 0)
                return launch_cfg<Cfg<TIn, HAS_Y, HAS_H0, MODE, 2, 16, 2, 4, kTrajNone, kMaxSlice, 256>>(p, stream);
            return launch_cfg<Cfg<TIn, HAS_Y, HAS_H0, MODE, 2, 16, 2, 4>>(p, stream);
        }
    }
}

template <typename TIn, int MODE>
cudaError_t launch_mode(const ScanParams &p, cudaStream_t stream) {
    if (p.traj != nullptr) {
        // strides of at least a few token groups amortise the renormalisation at each
        // trajectory point, so they take the rescaled accumulation
        if constexpr (MODE == kPower)
            if (p.traj_stride >= 4 * kGroup) return launch_t<TIn, false, false, MODE, kTrajRescaled>(p, stream);
        return launch_t<TIn, false, false, MODE, kTrajDirect>(p, stream);
    }
    const bool has_y = p.y != nullptr;
    const bool has_h0 = p.bank != nullptr;
    if (!has_y && !has_h0) {
        using Split = Cfg<TIn, false, false, MODE, 2, 16, 2, MODE == kGeneral ? 4 : 5, kTrajNone, kMaxSlice, 0, true>;
        const int segs = split_segments<Split>(p);
        if (segs > 1) {
            ScanParams q = p;
            q.segments = segs;
            return launch_cfg<Split>(q, stream);
        }
    }
    if (has_y)
        return has_h0 ? launch_t<TIn, true, true, MODE>(p, stream)
                      : launch_t<TIn, true, false, MODE>(p, stream);
    return has_h0 ? launch_t<TIn, false, true, MODE>(p, stream)
                  : launch_t<TIn, false, false, MODE>(p, stream);
}

template <typename TIn>
cudaError_t launch_in(const ScanParams &p, cudaStream_t stream) {
    return p.a_kind == PRECOG_A_POWER ? launch_mode<TIn, kPower>(p, stream)
                                      : launch_mode<TIn, kGeneral>(p, stream);
}

}  // namespace

cudaError_t launch_scan(const ScanParams &p, cudaStream_t stream) {
    if (p.in_dtype == PRECOG_F32) return launch_in<float>(p, stream);
    return launch_in<__nv_bfloat16>(p, stream);
}

cudaError_t scan_status_word_read_clear(uint32_t *bits) {
    uint32_t zero = 0;
    cudaError_t e = cudaMemcpyFromSymbol(bits, g_scan_status, sizeof(uint32_t));
    if (e != cudaSuccess) return e;
    return cudaMemcpyToSymbol(g_scan_status, &zero, sizeof(uint32_t));
}

}  // namespace precog
