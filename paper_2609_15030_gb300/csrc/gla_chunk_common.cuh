// Device pieces of the tensor-core prefill (gla_chunked_tc.cu): constants, the shared-memory
// and TMEM maps, the fast path's operand build, state pass, causal mask and output epilogue,
// the exact path's steps, the per-token short segments, and the MMA groups each path issues.
//
// Notation (per head, one segment of L <= 64 tokens inside one 64-token chunk of the
// absolute position grid, cumulative log2-decay Lam_i = log2(e) sum_{s<=i} a_s per key dim):
//   Q~_i = q_i 2^{Lam_i},  K~_j = k_j 2^{-Lam_j},  A_ij = [j <= i] Q~_i . K~_j,
//   o_i = Q~_i S + sum_j A_ij v_j,  S' = diag(2^{Lam_last}) (S + K~^T V)   (fast path)
//   S' = diag(2^{Lam_last}) S + K^^T V,  K^_j = k_j 2^{Lam_last - Lam_j}   (exact path)
#pragma once

#include <cuda.h>
#include <cudaTypedefs.h>
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include "hs_internal.cuh"
#include "sm100_ptx.cuh"

namespace hs {
namespace gck {

using namespace ptx;

constexpr int CH = 64;    // chunk length (absolute grid)
constexpr int NB = 256;   // operand builders (warps 0..7): cumulative gates, Q~, K~, V^T
constexpr int NW = 256;   // state warps (warps 8..15): state passes, masks, epilogues
constexpr int NT = NB + NW;
constexpr int kLoader = 0;   // the first builder thread issues the copies outside a run of fast
                             // segments; inside one a lane of warp 1 does
constexpr int kIssuer = NB + 64;  // the state thread that waits and arrives for its group; its warp's
                                  // elected lane issues every MMA.  In TMEM lane quarter 2, which
                                  // has no part in the masking of A
constexpr int kShort = 8; // segments of at most this many tokens run token by token
constexpr float kLog2e = 1.4426950408889634f;
// exact path: log-gates below this are taken at this value.  2^(kGateFloor * log2 e) = 2^-144
// is flushed to 0 by ex2.approx.ftz, so such a gate still zeroes the state, while the
// cumulative log2-decay after it stays small enough (|Lam| of a few hundred, not ~1.4e4 for
// a gate of -1e4) for the differences Lam_i - Lam_j of later tokens to keep their precision.
constexpr float kGateFloor = -100.0f;
constexpr float kF16Lim = 32768.0f;         // fast-path fp16 operands stay below 2^15
// a decision taken mid-run bounds the state it starts from (the measured |S| of the previous
// segment's start plus that segment's largest update); the bound is scaled by this margin so
// that whenever it passes, the measured state (what a run resumed at that segment checks)
// passes too: rounding can put the computed state a few ulps above the exact-arithmetic bound
constexpr float kBoundMargin = 1.00390625f; // 1 + 2^-8
constexpr float kLamRange = 10.0f;          // fast path: a segment's total log2-decay >= -10, so
                                            // Q~ = q 2^Lam stays far from fp16's subnormals
constexpr uint64_t kTimeoutNs = 1000000000ull;
// decision words of a run (fast path or not), in turn by segment.  Two: builder threads read the
// one of segment k - 1 after the barrier that follows its wait, and the first of them may already
// hand segment k over, whose decision must not land in the word the others are still to read; the
// decision after that needs a hand-over which comes after every builder thread passed its next wait.
constexpr int kDecisions = 2;
// segments requested into L2 ahead of the staged one.  One, since a segment is staged while the
// one two before it is still in work: two cost 256-token tails 26.6 us instead of 25.3 (their
// last segments competed with the first), three cost 4 x 32 heads of 16,384 tokens 992 us
// instead of 960, none 1,037.
constexpr int kPrefetch = 1;

// shared memory map (offsets from a 1024-byte aligned base), sized for the head width
// D = d_k = d_v = 128 (a D = 64 head uses the first part of each region).  Operands are
// K-major with the 128-byte swizzle.
constexpr uint32_t SET_BYTES = 40960;   // one of three fast operand sets:
constexpr uint32_t S_QH = 0;            //   Q~  fp16 [64 tok i][D]                     16 KiB
constexpr uint32_t S_KH = 16384;        //   K~  fp16 [64 tok j][D]                     16 KiB
constexpr uint32_t S_AH = 32768;        //   A   fp16 [64 tok i][64 tok j]                8 KiB
constexpr uint32_t X_QT = 0;            // exact path (over the sets): Q~ tf32 [64][D]         32 KiB
constexpr uint32_t X_LAM = 32768;       //   Lam f32 [64 tok][D] (see lam_at)                    32 KiB
constexpr uint32_t X_B2 = 65536;        //   [A ; K^^T] tf32 [64 i + D][64 tok j]               48 KiB
constexpr uint32_t OFF_SQ = 122880;     // staged q  bf16 [64][D]                  16 KiB
constexpr uint32_t OFF_SK = 139264;     // staged k                                 16 KiB
constexpr uint32_t OFF_SG = 155648;     // staged log-gates f32 [64][D]             32 KiB
constexpr uint32_t OFF_SV = 188416;     // staged v, two buffers by chunk parity    32 KiB
constexpr uint32_t OFF_GAM = 221184;    // 2^{Lam_last} per key dim, four slots by chunk number   2 KiB
constexpr uint32_t OFF_TOT = 223232;    // partial log2-decay totals [token groups][D]        2 KiB
constexpr uint32_t OFF_RED = 225280;    // three sets of [8 warps][8]: builders' max |q|, fast-path
                                        //   flag, max |k|, max |v| (0..3; with the operand sets);
                                        //   state warps' max |S| (4; two sets, a pass each in turn)
constexpr uint32_t OFF_BAR = 226048;    // 6 mbarriers
constexpr uint32_t OFF_MISC = 226112;   // TMEM base address, abort flag, decision, run result
constexpr uint32_t OFF_DG = 226176;     // diagonal of A in float32, with the operand sets:
                                        //   [set][key-dim half][64 tokens] partial sums  1.5 KiB
constexpr uint32_t SMEM_BYTES = 227712 + 1024;

// tensor memory: D_O alternates between two buffers by chunk parity, placed on
// either side of S^T.  Every MMA has M = 128 (TMEM lanes = value dim e, or query row i for D_A):
// with D = 64 the lanes 64..127 of the state-side products are computed and never read.
constexpr uint32_t TMEM_COLS = 512;
constexpr uint32_t TM_O0 = 0;           // D_O of even chunks (lane e, col i), 64 cols
constexpr uint32_t TM_S = 64;           // S^T  float32, 128 lanes x D cols
constexpr uint32_t TM_SH = 256;         // S^T fp16 copy, two key dims per column      D/2 cols
constexpr uint32_t TM_A = 320;          // D_A, 128 lanes x 64 cols (lanes 0..63 used)
constexpr uint32_t TM_V = 384;          // V^T: fast, fp16 pairs 3 x 32 cols (with the operand sets);
                                        // exact, f32 64 cols
// exact path (no fast-path data live): S^T as two tf32 parts for S^T Q~^T, hi in the D
// columns right of S^T (D_O1 and, for D = 128, the fp16 copy), lo in the columns of D_A and
// of the third V^T buffer (key dims 0..63, 64..127)
constexpr uint32_t TM_SLO0 = 320;
constexpr uint32_t TM_SLO1 = 448;

constexpr uint32_t IDF_N64 = idesc_f16(128, 64);
constexpr uint32_t IDT_N64 = idesc_tf32(128, 64, 0, 0);

// what depends on the head width D (64 or 128)
template <int D>
struct Geo {
    static_assert(D == 64 || D == 128, "head width");
    static constexpr int DP = D / 2;              // builder threads per token group (key-dim pairs)
    static constexpr int NQ = NB / DP;            // token groups of the build: 4 or 8
    static constexpr int TPG = CH / NQ;           // tokens per group: 16 or 8
    static constexpr int CW = D / 2;              // state columns per state thread: 64 or 32
    static constexpr int NG = D / 16;             // short segments: partial sums over 16 key rows
    static constexpr int ROWS = 64 + D;           // rows of the exact path's [A ; K^^T] operand
    static constexpr uint32_t O1 = TM_S + D;      // D_O of odd chunks, right of S^T
    static constexpr uint32_t SHI = TM_S + D;     // exact path: hi part of S^T
    static constexpr uint32_t IDF_ST = idesc_f16(128, D, 1);       // S^T += V^T K~ (K~ read MN-major)
    static constexpr uint32_t IDT_ST = idesc_tf32(128, D, 0, 0);   // exact: S^T += V^T K^
    static constexpr uint32_t STAGE = 3 * CH * D * 2 + CH * D * 4;  // staged q, k, v, log-gates
};

struct TmaMaps {
    CUtensorMap q, k, v, g;
};

// byte offset of 16-bit element (row, col) of a K-major operand with `rows` rows
// (64 columns = 128 bytes per row and slab)
__device__ __forceinline__ uint32_t h_off(int rows, int row, int col)
{
    return (uint32_t)((col >> 6) * rows * 128 + row * 128 + ((((col & 63) >> 3) ^ (row & 7)) << 4) +
                      ((col & 7) << 1));
}

// byte offset of 32-bit element (row, col) of a K-major operand (32 columns per slab)
__device__ __forceinline__ uint32_t t_off(int rows, int row, int col)
{
    return (uint32_t)((col >> 5) * rows * 128 + row * 128 + ((((col & 31) >> 2) ^ (row & 7)) << 4) +
                      ((col & 3) << 2));
}

// barriers among the builder warps (id 1) and among the state warps (id 2)
__device__ __forceinline__ void bar_builders()
{
    asm volatile("bar.sync 1, 256;" ::: "memory");
}

__device__ __forceinline__ void bar_staters()
{
    asm volatile("bar.sync 2, 256;" ::: "memory");
}

// named barrier `id` over 256 threads that also returns the OR of `pred` over them, so
// every thread of the group takes the same branch after it
__device__ __forceinline__ bool bar_or(int id, bool pred)
{
    uint32_t r;
    asm volatile(
        "{\n\t.reg .pred p, q;\n\t"
        "setp.ne.u32 p, %1, 0;\n\t"
        "bar.red.or.pred q, %2, 256, p;\n\t"
        "selp.u32 %0, 1, 0, q;\n\t}"
        : "=r"(r)
        : "r"((uint32_t)pred), "r"(id)
        : "memory");
    return r != 0;
}

__device__ __forceinline__ float warp_max(float v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
        v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}

// warp sums of eight per-lane values as a transposing butterfly: every lane returns the sum
// over the warp's 32 lanes of value x = (lane >> 2) & 7, added in the same order in every
// lane that holds it
__device__ __forceinline__ float warp_sum8(const float (&v)[8], int lane)
{
    const bool h4 = (lane & 16) != 0, h3 = (lane & 8) != 0, h2 = (lane & 4) != 0;
    float w[4], y[2];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const float send = h4 ? v[j] : v[j + 4];
        w[j] = (h4 ? v[j + 4] : v[j]) + __shfl_xor_sync(0xffffffffu, send, 16);
    }
#pragma unroll
    for (int j = 0; j < 2; ++j) {
        const float send = h3 ? w[j] : w[j + 2];
        y[j] = (h3 ? w[j + 2] : w[j]) + __shfl_xor_sync(0xffffffffu, send, 8);
    }
    const float send = h2 ? y[0] : y[1];
    float z = (h2 ? y[1] : y[0]) + __shfl_xor_sync(0xffffffffu, send, 4);
    z += __shfl_xor_sync(0xffffffffu, z, 2);
    z += __shfl_xor_sync(0xffffffffu, z, 1);
    return z;
}

__device__ __forceinline__ float bf16f(uint16_t x)
{
    return __uint_as_float(((uint32_t)x) << 16);
}

// two floats -> fp16x2 (round to nearest even), the first in the low half
__device__ __forceinline__ uint32_t pack_h2(float lo, float hi)
{
    const __half2 h = __floats2half2_rn(lo, hi);
    return *reinterpret_cast<const uint32_t *>(&h);
}

// running elementwise maxima of |x| over fp16 / bf16 pairs (NaN propagates)
__device__ __forceinline__ __half2 hmax_abs(__half2 acc, uint32_t pair)
{
    return __hmax2_nan(acc, __habs2(*reinterpret_cast<const __half2 *>(&pair)));
}

__device__ __forceinline__ __nv_bfloat162 bmax_abs(__nv_bfloat162 acc, uint32_t pair)
{
    return __hmax2_nan(acc, __habs2(*reinterpret_cast<const __nv_bfloat162 *>(&pair)));
}

__device__ __forceinline__ float hmax_of(__half2 m)
{
    return fmaxf(__low2float(m), __high2float(m));
}

__device__ __forceinline__ float bmax_of(__nv_bfloat162 m)
{
    return fmaxf(__low2float(m), __high2float(m));
}

// 2^x, one MUFU op (relative error ~2^-22)
__device__ __forceinline__ float ex2(float x)
{
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// round to tf32 (nearest, ties away from zero) with integer ops; low 13 bits cleared.  A NaN stays
// one: CUDA's, 0x7FFFFFFF, would carry into the sign and become -0, hiding what the inputs did
__device__ __forceinline__ float rna_tf32(float x)
{
    return x == x ? __uint_as_float((__float_as_uint(x) + 0x1000u) & 0xFFFFE000u) : x;
}


// threadIdx.x, not known to be a constant of the loop over the segments: the exact path's
// address arithmetic then stays in the exact path.  Hoisted out of the loop it was spilled
// around the fast path, which runs at the register limit (256-token tails 33.2 us, not 29.8).
__device__ __forceinline__ int thread_id()
{
    int t;
    asm volatile("mov.u32 %0, %%tid.x;" : "=r"(t));
    return t;
}

// the staged v of the segment in v buffer vb
__device__ __forceinline__ const uint16_t *staged_v(const uint8_t *smem, int vb)
{
    return reinterpret_cast<const uint16_t *>(smem + OFF_SV + vb * 16384);
}

// zero the staged rows past a segment of L < 64 tokens (all threads, or the builder
// warps only)
template <int D>
__device__ __forceinline__ void zero_tail(uint8_t *smem, int L, int vb, bool builders_only)
{
    const int tid = threadIdx.x;
    constexpr int QV = D / 8, RV = 5 * D / 8;   // 16-byte vectors per q/k/v row, per token

    if (L < CH) {
        const int nthr = builders_only ? NB : NT;
        for (int idx = tid; idx < (CH - L) * RV; idx += nthr) {
            const int row = L + idx / RV, c = idx % RV;
            uint4 *dst;
            if (c < QV)
                dst = reinterpret_cast<uint4 *>(smem + OFF_SQ + row * 2 * D) + c;
            else if (c < 2 * QV)
                dst = reinterpret_cast<uint4 *>(smem + OFF_SK + row * 2 * D) + (c - QV);
            else if (c < 3 * QV)
                dst = reinterpret_cast<uint4 *>(smem + OFF_SV + vb * 16384 + row * 2 * D) + (c - 2 * QV);
            else
                dst = reinterpret_cast<uint4 *>(smem + OFF_SG + row * 4 * D) + (c - 3 * QV);
            *dst = make_uint4(0u, 0u, 0u, 0u);
        }
        fence_proxy_async_smem();   // the next copies overwrite these rows
        if (builders_only)
            bar_builders();
        else
            __syncthreads();
    }
}


// ---- fast operands of a staged long segment into set iset (builder warps).  Thread
// (dp, qt) owns key dims 2dp, 2dp+1 for the TPG tokens of group qt (16 tokens x 4 groups at
// D = 128, 8 x 8 at D = 64): it sums their log2-gates, then runs the cumulative sum again
// from the earlier groups' totals (shared memory; 2^{Lam_last} into gam slot `gslot`) while
// it writes Q~ and K~ (token-major), fp16, with 4-byte stores.  Its two key dims are a register
// pair: their sums and products are f32x2 instructions, the roundings those of the scalar ones
// (with the state pass's decay: 4 x 32 heads of 16,384 tokens 957.5 us, now 950).  Per warp:
// max |q|, |k| and per thread whether its operands fit fp16 (for the guard).  The diagonal
// A_ii = q_i . k_i (no decay between a token and itself) is summed in float32 from the bf16
// inputs, each warp's 64 key dims by a butterfly, into the set's diagonal partials: fp16 Q~ and K~
// would round the terms of that dot product to 11 bits, which a token whose own q . k cancels
// cannot afford.
//
// A segment that the guard is sure to send to the exact path for its gates alone (one above
// 0, or a total log2-decay below -kLamRange) stops after the totals and returns false: the
// staged inputs are untouched, so the exact path starts from them without another copy.
template <int D>
__device__ __forceinline__ bool build_fast(uint8_t *smem, int L, int vb, int iset, int gslot,
                                           float &mq, float &mk, bool &ok)
{
    using G = Geo<D>;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const uint16_t *sQ = reinterpret_cast<const uint16_t *>(smem + OFF_SQ);
    const uint16_t *sK = reinterpret_cast<const uint16_t *>(smem + OFF_SK);
    const float *sG = reinterpret_cast<const float *>(smem + OFF_SG);
    float *sTot = reinterpret_cast<float *>(smem + OFF_TOT);
    float *sGam = reinterpret_cast<float *>(smem + OFF_GAM);

    zero_tail<D>(smem, L, vb, true);
    const int dp = tid % G::DP, qt = tid / G::DP;
    float amax = -INFINITY;
    {
        // group totals
        uint64_t r = 0;
#pragma unroll
        for (int x = 0; x < G::TPG; ++x) {
            const uint64_t a = *reinterpret_cast<const uint64_t *>(sG + (G::TPG * qt + x) * D + 2 * dp);
            amax = fmaxf(amax, fmaxf(unpair(a).x, unpair(a).y));
            r = fma2(a, pair(kLog2e, kLog2e), r);
        }
        *reinterpret_cast<uint64_t *>(sTot + qt * D + 2 * dp) = r;
    }
    bar_builders();
    // the running sums start from the earlier groups' totals
    float run0 = 0.f, run1 = 0.f;
    bool lam_ok;
    {
        float t0 = 0.f, t1 = 0.f;
#pragma unroll
        for (int u = 0; u < G::NQ; ++u) {
            const float2 t = *reinterpret_cast<const float2 *>(sTot + u * D + 2 * dp);
            if (u < qt) {
                run0 += t.x;
                run1 += t.y;
            }
            t0 += t.x;
            t1 += t.y;
        }
        if (qt == 0)
            *reinterpret_cast<float2 *>(sGam + gslot * D + 2 * dp) = make_float2(ex2(t0), ex2(t1));
        lam_ok = t0 >= -kLamRange && t1 >= -kLamRange;
    }
    if (bar_or(1, !(amax <= 0.f && lam_ok)))
        return false;
    uint8_t *set = smem + iset * SET_BYTES;
    __nv_bfloat162 bq = __float2bfloat162_rn(0.f), bk = bq;   // max |q|, |k|
    __half2 hq = __float2half2_rn(0.f), hk = hq;                 // max |Q~|, |K~| (fp16)
    // runs of 8 tokens; within a run, token pairs: Q~ and K~ as fp16 pairs of key dims
    float *sDg = reinterpret_cast<float *>(smem + OFF_DG) + iset * 128 + (dp >> 5) * 64;
    uint64_t run = pair(run0, run1);
#pragma unroll 1
    for (int grp = 0; grp < G::TPG / 8; ++grp) {
        const int j0 = G::TPG * qt + 8 * grp;
        // the eight tokens' inputs first: the compiler cannot move a load over the operand stores
        uint64_t a[8];
        uint32_t q2[8], k2[8];
#pragma unroll
        for (int t = 0; t < 8; ++t) {
            a[t] = *reinterpret_cast<const uint64_t *>(sG + (j0 + t) * D + 2 * dp);
            q2[t] = *reinterpret_cast<const uint32_t *>(sQ + (j0 + t) * D + 2 * dp);
            k2[t] = *reinterpret_cast<const uint32_t *>(sK + (j0 + t) * D + 2 * dp);
        }
        float pd[8];   // q . k over this thread's two key dims, tokens 8 grp + 0..7 of its group
#pragma unroll
        for (int t = 0; t < 8; ++t) {
            run = fma2(a[t], pair(kLog2e, kLog2e), run);
            const float2 lam = unpair(run);
            const float q0 = __uint_as_float(q2[t] << 16), q1 = __uint_as_float(q2[t] & 0xFFFF0000u);
            const float k0 = __uint_as_float(k2[t] << 16), k1 = __uint_as_float(k2[t] & 0xFFFF0000u);
            const float2 qs = unpair(mul2(pair(q0, q1), pair(ex2(lam.x), ex2(lam.y))));
            const float2 ks = unpair(mul2(pair(k0, k1), pair(ex2(-lam.x), ex2(-lam.y))));
            const uint32_t qp = pack_h2(qs.x, qs.y);
            const uint32_t kp = pack_h2(ks.x, ks.y);
            pd[t] = fmaf(q1, k1, q0 * k0);
            *reinterpret_cast<uint32_t *>(set + S_QH + h_off(64, j0 + t, 2 * dp)) = qp;
            *reinterpret_cast<uint32_t *>(set + S_KH + h_off(64, j0 + t, 2 * dp)) = kp;
            bq = bmax_abs(bq, q2[t]);
            bk = bmax_abs(bk, k2[t]);
            hq = hmax_abs(hq, qp);
            hk = hmax_abs(hk, kp);
        }
        const float dsum = warp_sum8(pd, lane);
        if ((lane & 3) == 0)
            sDg[j0 + ((lane >> 2) & 7)] = dsum;
    }
    mq = warp_max(bmax_of(bq));
    mk = warp_max(bmax_of(bk));
    ok = hmax_of(hq) < kF16Lim && hmax_of(hk) < kF16Lim;
    return true;
}

// ... then V^T (buffer iset), thread (e, half) packing tokens [32 half, 32 half + 32) of value dim
// e, and the guard words (set iset; `built`: whether build_fast went through; if not, a failing
// flag only)
template <int D>
__device__ __forceinline__ void build_values(uint8_t *smem, uint32_t tmem, int vb, int iset, bool built,
                                             float mq, float mk, bool ok)
{
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const uint32_t lrow = (uint32_t)((warp & 3) * 32) << 16;   // this warp's TMEM lane quarter
    const int e_own = (warp & 3) * 32 + lane;                  // TMEM lane = value dim e
    const int th = warp >> 2;
    const uint16_t *sV = staged_v(smem, vb);
    float *sRed = reinterpret_cast<float *>(smem + OFF_RED) + iset * 64;
    if (!built) {
        if (lane == 0)
            sRed[warp * 8 + 1] = 0.f;
        return;
    }
    __nv_bfloat162 bv = __float2bfloat162_rn(0.f);
    {
        uint32_t vpk[16];
#pragma unroll
        for (int m = 0; m < 16; ++m) {
            const int i = 32 * th + 2 * m;
            uint32_t w = 0;
            if (e_own < D)
                w = (uint32_t)sV[i * D + e_own] | ((uint32_t)sV[(i + 1) * D + e_own] << 16);
            bv = bmax_abs(bv, w);
            vpk[m] = pack_h2(__uint_as_float(w << 16), __uint_as_float(w & 0xFFFF0000u));
        }
        tmem_st16(tmem + lrow + TM_V + 32 * iset + 16 * th, vpk);
    }
    const float mv = warp_max(bmax_of(bv));
    // non-increasing Lam (|Q~| <= |q|, |A| <= D max|q| max|k|), a total decay of at most
    // 2^-10 (Q~ of the segment's last tokens keeps its precision) and every fp16 operand below
    // 2^15; NaN fails
    ok = __all_sync(0xffffffffu, ok && mv < kF16Lim);
    if (lane == 0) {
        sRed[warp * 8 + 0] = mq;
        sRed[warp * 8 + 1] = ok ? 1.f : 0.f;
        sRed[warp * 8 + 2] = mk;
        sRed[warp * 8 + 3] = mv;
    }
    tmem_wait_st();
}


// ---- state pass (state warps): decay by gam slot gpar (gpar < 0: none), checkpoint slot,
// fp16 copy of S^T for the next S^T Q~^T, and the largest |S| (into maxima set mset)
template <int D>
__device__ __forceinline__ void state_pass(uint8_t *smem, uint32_t tmem, int gpar, float *slot, bool copy,
                                           int mset)
{
    constexpr int CW = Geo<D>::CW;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const bool worker = warp >= 8;
    const uint32_t lrow = (uint32_t)((warp & 3) * 32) << 16;   // this warp's TMEM lane quarter
    const int colhalf = (warp >> 2) & 1;
    const int e_own = (warp & 3) * 32 + lane;                  // TMEM lane = value dim e
    const float *sGam = reinterpret_cast<const float *>(smem + OFF_GAM);
    float *sRed = reinterpret_cast<float *>(smem + OFF_RED) + mset * 64;

    if (!worker)
        return;
    float m = 0.f;
    if (e_own < D) {
        // 32 columns at a time; at d = 128 the issuing warp, which also issues D_A meanwhile, takes
        // a quarter of its lanes' columns and its partner three
        const int d0 = D == 128 && warp == kIssuer / 32 + 4 ? 32 : colhalf * CW;
        const int d1 = D == 128 && warp == kIssuer / 32 ? 32 : colhalf * CW + CW;
        __half2 hm = __float2half2_rn(0.f);
#pragma unroll 1
        for (int db = d0; db < d1; db += 32) {
            float r[32];
            tmem_ld32(tmem + lrow + TM_S + db, r);
            tmem_wait_ld();
            if (gpar >= 0) {
                const float *gam = sGam + gpar * D + db;
#pragma unroll
                for (int c = 0; c < 8; ++c) {
                    const float4 g4 = *reinterpret_cast<const float4 *>(gam + 4 * c);
                    const float2 x = unpair(mul2(pair(r[4 * c], r[4 * c + 1]), pair(g4.x, g4.y)));
                    const float2 y = unpair(mul2(pair(r[4 * c + 2], r[4 * c + 3]), pair(g4.z, g4.w)));
                    r[4 * c] = x.x;
                    r[4 * c + 1] = x.y;
                    r[4 * c + 2] = y.x;
                    r[4 * c + 3] = y.y;
                }
                tmem_st32(tmem + lrow + TM_S + db, r);
            }
            if (slot != nullptr) {
#pragma unroll
                for (int x = 0; x < 32; ++x)
                    slot[(int64_t)(db + x) * D + e_own] = r[x];
            }
            if (copy) {
                // the fp16 copy, two key dims per column; its largest magnitude (inf past fp16)
                uint32_t u[16];
#pragma unroll
                for (int c = 0; c < 16; ++c) {
                    u[c] = pack_h2(r[2 * c], r[2 * c + 1]);
                    hm = hmax_abs(hm, u[c]);
                }
                tmem_st16(tmem + lrow + TM_SH + db / 2, u);
            } else {
#pragma unroll
                for (int x = 0; x < 32; ++x)
                    m = fmaxf(m, fabsf(r[x]));
            }
        }
        if (copy)
            m = hmax_of(hm);
        tmem_wait_st();
    }
    m = warp_max(m);
    if (lane == 0)
        sRed[(warp & 7) * 8 + 4] = m;
}


// ---- the causally masked intra-chunk matrix A (D_A) -> operand set iset's A
// (state warps of TMEM lane quarters 0 and 1)
template <int D>
__device__ __forceinline__ void a_build(uint8_t *smem, uint32_t tmem, int iset)
{
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const bool worker = warp >= 8;
    const uint32_t lrow = (uint32_t)((warp & 3) * 32) << 16;

    if (!(worker && (warp & 3) < 2))
        return;
    const int i = (warp & 3) * 32 + lane;      // TMEM lane = query row
    const int jb = ((warp >> 2) & 1) * 32;      // this warp's 32 key columns
    float r[32];
    tmem_ld32(tmem + lrow + TM_A + jb, r);
    // the diagonal from the builders' float32 partials (one per 64 key dims)
    const float *sDg = reinterpret_cast<const float *>(smem + OFF_DG) + iset * 128;
    const float dg = (i >= jb && i < jb + 32) ? (D == 128 ? sDg[i] + sDg[64 + i] : sDg[i]) : 0.f;
    tmem_wait_ld();
    uint8_t *set = smem + iset * SET_BYTES;
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        uint32_t w[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int j0 = jb + 8 * c + 2 * u;
            const float x0 = j0 == i ? dg : (j0 <= i ? r[8 * c + 2 * u] : 0.f);
            const float x1 = j0 + 1 == i ? dg : (j0 + 1 <= i ? r[8 * c + 2 * u + 1] : 0.f);
            w[u] = pack_h2(x0, x1);
        }
        *reinterpret_cast<uint4 *>(set + S_AH + h_off(64, i, jb + 8 * c)) =
            make_uint4(w[0], w[1], w[2], w[3]);
    }
}


// ---- output epilogue of a processed segment (state warps): D_O buffer `par` -> o (lane e,
// 32 rows per warp)
template <int D>
__device__ __forceinline__ void out_epilogue(uint32_t tmem, float *ob, int64_t tstride, int L, int par)
{
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const bool worker = warp >= 8;
    const uint32_t lrow = (uint32_t)((warp & 3) * 32) << 16;   // this warp's TMEM lane quarter
    const int colhalf = (warp >> 2) & 1;
    const int e_own = (warp & 3) * 32 + lane;                  // TMEM lane = value dim e

    if (!worker || e_own >= D)
        return;
#pragma unroll 1
    for (int ib = colhalf * 32; ib < colhalf * 32 + 32; ib += 16) {
        uint32_t r[16];
        tmem_ld16(tmem + lrow + (par ? Geo<D>::O1 : TM_O0) + ib, r);
        tmem_wait_ld();
        float *op = ob + (int64_t)ib * tstride + e_own;
        if (L == CH) {
#pragma unroll
            for (int x = 0; x < 16; ++x)
                __stcs(op + (int64_t)x * tstride, __uint_as_float(r[x]));
        } else {
#pragma unroll
            for (int x = 0; x < 16; ++x)
                if (ib + x < L)
                    __stcs(op + (int64_t)x * tstride, __uint_as_float(r[x]));
        }
    }
}


// ---- the state between global memory ([d][e], row = key dim) and TMEM (S^T, lane e) ----

// (state warps) load a state into TMEM and record its largest |S| (float32) for the guard
template <int D>
__device__ __forceinline__ void state_load(uint8_t *smem, uint32_t tmem, const float *src, int mset)
{
    constexpr int CW = Geo<D>::CW;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (warp < 8)
        return;
    const uint32_t lrow = (uint32_t)((warp & 3) * 32) << 16;
    const int colhalf = (warp >> 2) & 1;
    const int e_own = (warp & 3) * 32 + lane;
    float *sRed = reinterpret_cast<float *>(smem + OFF_RED) + mset * 64;
    float r[32];
    float m = 0.f;
    if (e_own < D) {
#pragma unroll
        for (int c0 = 0; c0 < CW; c0 += 32) {
            const int d0 = colhalf * CW + c0;
#pragma unroll
            for (int x = 0; x < 32; ++x) {
                r[x] = src[(int64_t)(d0 + x) * D + e_own];
                m = fmaxf(m, fabsf(r[x]));
            }
            tmem_st32(tmem + lrow + TM_S + d0, r);
        }
        tmem_wait_st();
    }
    m = warp_max(m);
    if (lane == 0)
        sRed[(warp & 7) * 8 + 4] = m;
}

// (state warps) store the state in TMEM to global memory
template <int D>
__device__ __forceinline__ void state_store(uint32_t tmem, float *dst)
{
    constexpr int CW = Geo<D>::CW;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int e_own = (warp & 3) * 32 + lane;
    if (warp < 8 || e_own >= D)
        return;
    const uint32_t lrow = (uint32_t)((warp & 3) * 32) << 16;
    const int colhalf = (warp >> 2) & 1;
    float r[32];
#pragma unroll
    for (int c0 = 0; c0 < CW; c0 += 32) {
        const int d0 = colhalf * CW + c0;
        tmem_ld32(tmem + lrow + TM_S + d0, r);
        tmem_wait_ld();
#pragma unroll
        for (int x = 0; x < 32; ++x)
            dst[(int64_t)(d0 + x) * D + e_own] = r[x];
    }
}

// ---- exact path pieces (every thread of the 512-thread CTA takes part) ----

// element (token, key dim) of X_LAM, in floats: token-major, the 16-byte chunks of odd tokens
// swapped in pairs so that the fragment loads of exact_square (16 bytes from each of two
// neighbouring rows per quarter-warp) meet no bank twice
template <int D>
__device__ __forceinline__ int lam_at(int row, int d)
{
    return row * D + (d ^ ((row & 1) << 2));
}

// cumulative log2-gates of a staged segment (16 tokens of a key dim per thread, into X_LAM;
// gates below kGateFloor taken at the floor), Q~ = q 2^{Lam} (tf32, X_QT) and 2^{Lam_last} into
// gam slot 0.  Returns (uniformly) whether some gate is above 0.
template <int D>
__device__ __forceinline__ bool exact_decay(uint8_t *smem, int L, int vb)
{
    const int tid = thread_id(), warp = tid >> 5, lane = tid & 31;
    const int d = (warp & 3) * 32 + lane;
    const bool worker = d < D;
    const int t0 = (warp >> 2) * 16;           // this thread's 16 tokens
    const uint16_t *sQ = reinterpret_cast<const uint16_t *>(smem + OFF_SQ);
    const float *sG = reinterpret_cast<const float *>(smem + OFF_SG);
    float *sTot = reinterpret_cast<float *>(smem + OFF_TOT);
    float *sGam = reinterpret_cast<float *>(smem + OFF_GAM);
    float *sLam = reinterpret_cast<float *>(smem + X_LAM);
    zero_tail<D>(smem, L, vb, false);
    float lam[16];
    bool up = false;
    if (worker) {
        float run = 0.f;
#pragma unroll
        for (int x = 0; x < 16; ++x) {
            const float g = fmaxf(sG[(t0 + x) * D + d], kGateFloor);
            up = up || g > 0.f;
            run = fmaf(g, kLog2e, run);
            lam[x] = run;
        }
        sTot[(warp >> 2) * D + d] = run;
    }
    up = __syncthreads_or(up) != 0;
    if (worker) {
        float before = 0.f, last = 0.f;        // Lam before this thread's tokens, Lam_last
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            if (u == (warp >> 2))
                before = last;
            last += sTot[u * D + d];
        }
        if (t0 == 0)
            sGam[d] = ex2(last);
#pragma unroll
        for (int x = 0; x < 16; ++x) {
            const float l = before + lam[x];
            sLam[lam_at<D>(t0 + x, d)] = l;
            *reinterpret_cast<float *>(smem + X_QT + t_off(64, t0 + x, d)) =
                rna_tf32(bf16f(sQ[(t0 + x) * D + d]) * ex2(l));
        }
    }
    return up;
}

// (builder warps) K^^T = k 2^{Lam_last - Lam} (tf32, rows 64.. of X_B2) and V^T float32 into TMEM
template <int D>
__device__ __forceinline__ void exact_keys_values(uint8_t *smem, uint32_t tmem, int vb)
{
    const int warp = thread_id() >> 5, lane = thread_id() & 31;
    const int d = (warp & 3) * 32 + lane;      // key dim, and value dim = TMEM lane of V^T
    if (warp >= 8 || d >= D)
        return;
    const uint32_t lrow = (uint32_t)((warp & 3) * 32) << 16;
    const uint16_t *sK = reinterpret_cast<const uint16_t *>(smem + OFF_SK);
    const uint16_t *sV = staged_v(smem, vb);
    const float *sLam = reinterpret_cast<const float *>(smem + X_LAM);
    const float last = sLam[lam_at<D>(CH - 1, d)];
#pragma unroll 1
    for (int t0 = (warp >> 2) * 32; t0 < (warp >> 2) * 32 + 32; t0 += 16) {
        uint32_t vtr[16];
#pragma unroll
        for (int g = 0; g < 4; ++g) {
            float4 w;
            float *wv = &w.x;
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int i = t0 + 4 * g + u;
                wv[u] = rna_tf32(bf16f(sK[i * D + d]) * ex2(last - sLam[lam_at<D>(i, d)]));
                vtr[4 * g + u] = __float_as_uint(bf16f(sV[i * D + d]));
            }
            *reinterpret_cast<float4 *>(smem + X_B2 + t_off(Geo<D>::ROWS, 64 + d, t0 + 4 * g)) = w;
        }
        tmem_st16(tmem + lrow + TM_V + t0, vtr);
    }
    tmem_wait_st();
}

// (state warps) the state as two tf32 parts for S^T Q~^T (an A operand from TMEM is read as
// tf32): hi = S with its low 13 mantissa bits cleared (exact in tf32), lo = S - hi (exact in
// fp32, at most 13 significant bits), so the product keeps the state to ~2^-20 instead of a
// 2^-10 truncation.  S itself is then left decayed by gam slot 0 for the state update.
template <int D>
__device__ __forceinline__ void exact_split_state(const uint8_t *smem, uint32_t tmem)
{
    constexpr int CW = Geo<D>::CW;
    const int warp = thread_id() >> 5, lane = thread_id() & 31;
    if (warp < 8 || (warp & 3) * 32 + lane >= D)
        return;
    const uint32_t lrow = (uint32_t)((warp & 3) * 32) << 16;
    const int colhalf = (warp >> 2) & 1;
    // 16 columns at a time: 32 took the kernel past its registers
#pragma unroll 1
    for (int c0 = 0; c0 < CW; c0 += 16) {
        const int d0 = colhalf * CW + c0;
        const float *gam = reinterpret_cast<const float *>(smem + OFF_GAM) + d0;
        uint32_t r[16], x2[16];
        tmem_ld16(tmem + lrow + TM_S + d0, r);
        tmem_wait_ld();
#pragma unroll
        for (int x = 0; x < 16; ++x)
            x2[x] = r[x] & 0xFFFFE000u;
        tmem_st16(tmem + lrow + Geo<D>::SHI + d0, x2);
#pragma unroll
        for (int x = 0; x < 16; ++x)
            x2[x] = __float_as_uint(__uint_as_float(r[x]) - __uint_as_float(x2[x]));
        tmem_st16(tmem + lrow + (d0 < 64 ? TM_SLO0 + d0 : TM_SLO1 + (d0 - 64)), x2);
#pragma unroll
        for (int x = 0; x < 16; ++x)
            r[x] = __float_as_uint(__uint_as_float(r[x]) * gam[x]);
        tmem_st16(tmem + lrow + TM_S + d0, r);
    }
    tmem_wait_st();
}

// ---- exact path: A_ij = sum_d q_id k_jd 2^{Lam_id - Lam_jd}, j <= i < L, as exact as float32 sums
// over pairs, then rounded to tf32 into rows 0..63 of X_B2 (zeros above the diagonal).
//
// Taken pair by pair that is 262,144 exponentials at d = 128 and, with one thread per pair, a
// 32-way bank conflict on every operand.  When no gate is above 0 the 64 x 64 triangle is cut
// in halves instead: the lower left H x H square of every block of 2 H tokens (H = 32, 16, 8)
// factors at the token R that ends the block's first half, 2^{Lam_i - Lam_j} =
// 2^{Lam_i - Lam_R} 2^{Lam_R - Lam_j} with j <= R < i, so both exponents are <= 0: no overflow,
// and a power that underflows stands for a power 2^{Lam_i - Lam_j} that does.  The factors are formed in
// registers as matrix fragments and split into two tf32 parts each, three tf32 products for one
// (see squares_mma).  The eight 8 x 8 triangles left on the diagonal
// are taken pair by pair.  The tasks (one warp each, drawn from a shared counter, the long ones
// first) are halves of the key dims of four 16 x 16 units (a square of H = 16, or two of H = 8),
// quarters of those of each half of the 32 x 32 square, and 64 key dims of a triangle.  Meanwhile the
// issuing thread's warp feeds S^T Q~^T to the tensor core, a chain of dependent products under the
// tasks.  Tails of 475 tokens of 9 x 16 heads with every segment on this path: 507 us taken pair
// by pair, 125 us with the squares' products on CUDA cores, 94 us as tf32 fragments, 87 us with
// the builders looking one segment ahead, and 90.7 us since the fragments are rounded and summed
// as exactly as pairs and infinities and NaN are kept: ~23 k cycles a segment, the decays, operands,
// scores, update and outputs one after another (a segment's exponentials alone are ~2,300 warp
// instructions, 4.6 k cycles of the special-function units).
// Segments with a gate above 0 keep the pairwise form (exact_scores_pairs), and segments with a
// score that comes out infinite or NaN fall back to it.

// a 16 x 16 unit's rows: query rows r0.. and r1.. (8 each), key rows c0.. and c1.., and the
// tokens R that (r0, c0) and (r1, c1) factor at; units 2 and 3 hold two squares of H = 8, in
// the quadrants (r0, c0) and (r1, c1)
struct SquareUnit {
    int r0, r1, c0, c1, ref0, ref1;
};

__device__ __forceinline__ SquareUnit square_unit(int u)
{
    SquareUnit m;
    m.c0 = 32 * (u & 1);
    m.r0 = m.c0 + (u < 2 ? 16 : 8);
    m.c1 = m.c0 + (u < 2 ? 8 : 16);
    m.r1 = m.c0 + 24;
    m.ref0 = m.c0 + (u < 2 ? 15 : 7);
    m.ref1 = m.c0 + (u < 2 ? 15 : 23);
    return m;
}

// partial sums of the tasks, in the staged log-gates' area (free by then)
constexpr uint32_t X_P32 = OFF_SG;             // 32 x 32 square [4 quarters][32][32]     16 KiB
constexpr uint32_t X_P16 = OFF_SG + 16384;     // units [4][2 halves][16][16]              8 KiB
constexpr uint32_t X_PTR = OFF_SG + 24576;     // triangles [8][d / 64][40]              2.5 KiB

// four factors x 2^{+-(l - lr)} of one row (key dims kk..kk+3): x in bf16 and the powers, lr given
struct Factors {
    uint2 w;
    float e[4];

    __device__ __forceinline__ float x(int i) const
    {
        const uint32_t u = i < 2 ? w.x : w.y;
        return __uint_as_float((i & 1) ? u & 0xFFFF0000u : u << 16);
    }
};

template <int D, int SIGN>
__device__ __forceinline__ Factors factors4(const uint8_t *smem, uint32_t off, int row, const float4 &r,
                                            int kk)
{
    const float *sLam = reinterpret_cast<const float *>(smem + X_LAM);
    const float4 l = *reinterpret_cast<const float4 *>(sLam + lam_at<D>(row, kk));
    const float s = (float)SIGN;
    return {*reinterpret_cast<const uint2 *>(smem + off + (row * D + kk) * 2),
            {ex2(s * (l.x - r.x)), ex2(s * (l.y - r.y)), ex2(s * (l.z - r.z)), ex2(s * (l.w - r.w))}};
}

template <int D>
__device__ __forceinline__ float4 lam4(const uint8_t *smem, int row, int kk)
{
    return *reinterpret_cast<const float4 *>(reinterpret_cast<const float *>(smem + X_LAM) +
                                             lam_at<D>(row, kk));
}

// NT8 tiles of 16 x 8 scores += fragments a (rows g and g + 8) and b, each four consecutive key dims
// per lane: a k step of the products takes two of them (any assignment of key dims to k will
// do, as long as both operands share it).  The matrix instruction truncates its sums, so each
// step's three products have an accumulator of their own, which float32 additions (to nearest)
// collect.  Root mean square error of cancelling scores relative to the sum of their terms'
// magnitudes: 1.7e-8 at d = 128 and 2.3e-8 at d = 64 (taken pair by pair 2.0e-8 and 2.3e-8); with
// parts split by truncation and one accumulator throughout 4.1e-8 and 4.9e-8, at 87.5 us instead of
// 90.6 for tails of 475 tokens of 9 x 16 heads.
template <int NT8>
__device__ __forceinline__ void squares_mma(float (&acc)[NT8][4], const Factors (&a)[2],
                                            const Factors (&b)[NT8])
{
#pragma unroll
    for (int x = 0; x < 4; x += 2) {
        uint32_t ah[4], al[4], bh[NT8][2], bl[NT8][2];
        float c[NT8][4];
#pragma unroll
        for (int n = 0; n < NT8; ++n) {
            split_tf32(b[n].x(x), b[n].e[x], bh[n][0], bl[n][0]);
            split_tf32(b[n].x(x + 1), b[n].e[x + 1], bh[n][1], bl[n][1]);
        }
        split_tf32(a[0].x(x), a[0].e[x], ah[0], al[0]);
        split_tf32(a[1].x(x), a[1].e[x], ah[1], al[1]);
        split_tf32(a[0].x(x + 1), a[0].e[x + 1], ah[2], al[2]);
        split_tf32(a[1].x(x + 1), a[1].e[x + 1], ah[3], al[3]);
#pragma unroll
        for (int n = 0; n < NT8; ++n)
            mma_m16n8k8_tf32_new(c[n], al, bh[n]);
#pragma unroll
        for (int n = 0; n < NT8; ++n)
            mma_m16n8k8_tf32(c[n], ah, bl[n]);
#pragma unroll
        for (int n = 0; n < NT8; ++n)
            mma_m16n8k8_tf32(c[n], ah, bh[n]);
#pragma unroll
        for (int n = 0; n < NT8; ++n)
#pragma unroll
            for (int y = 0; y < 4; ++y)
                acc[n][y] += c[n][y];
    }
}

// (one warp) a quarter of the key dims of one half (queries 32 + 16 mh..) of the 32 x 32 square
// (queries 32..63, keys 0..31, factored at token 31)
template <int D>
__device__ __forceinline__ void exact_square32(uint8_t *smem, int mh, int quarter)
{
    const int lane = thread_id() & 31, g = lane >> 2, t = lane & 3;
    float acc[4][4] = {};
#pragma unroll 1
    for (int k0 = quarter * (D / 4); k0 < (quarter + 1) * (D / 4); k0 += 16) {
        const int kk = k0 + 4 * t;
        const float4 r = lam4<D>(smem, 31, kk);
        Factors a[2], b[4];
#pragma unroll
        for (int x = 0; x < 2; ++x)
            a[x] = factors4<D, 1>(smem, OFF_SQ, 32 + 16 * mh + 8 * x + g, r, kk);
#pragma unroll
        for (int x = 0; x < 4; ++x)
            b[x] = factors4<D, -1>(smem, OFF_SK, 8 * x + g, r, kk);
        squares_mma<4>(acc, a, b);
    }
    float *dst = reinterpret_cast<float *>(smem + X_P32) + quarter * 1024 + (16 * mh + g) * 32 + 2 * t;
#pragma unroll
    for (int n = 0; n < 4; ++n) {
        *reinterpret_cast<float2 *>(dst + 8 * n) = make_float2(acc[n][0], acc[n][1]);
        *reinterpret_cast<float2 *>(dst + 8 * 32 + 8 * n) = make_float2(acc[n][2], acc[n][3]);
    }
}

// (one warp) half of unit u's key dims
template <int D>
__device__ __forceinline__ void exact_square16(uint8_t *smem, int u, int half)
{
    const int lane = thread_id() & 31, g = lane >> 2, t = lane & 3;
    const SquareUnit m = square_unit(u);
    float acc[2][4] = {};
#pragma unroll 1
    for (int k0 = half * (D / 2); k0 < (half + 1) * (D / 2); k0 += 32) {
        Factors a[2][2], b[2][2];
#pragma unroll
        for (int y = 0; y < 2; ++y) {
            const int kk = k0 + 16 * y + 4 * t;
            const float4 ra = lam4<D>(smem, m.ref0, kk), rb = lam4<D>(smem, m.ref1, kk);
            a[y][0] = factors4<D, 1>(smem, OFF_SQ, m.r0 + g, ra, kk);
            a[y][1] = factors4<D, 1>(smem, OFF_SQ, m.r1 + g, rb, kk);
            b[y][0] = factors4<D, -1>(smem, OFF_SK, m.c0 + g, ra, kk);
            b[y][1] = factors4<D, -1>(smem, OFF_SK, m.c1 + g, rb, kk);
        }
        squares_mma<2>(acc, a[0], b[0]);
        squares_mma<2>(acc, a[1], b[1]);
    }
    float *dst = reinterpret_cast<float *>(smem + X_P16) + (2 * u + half) * 256;
#pragma unroll
    for (int n = 0; n < 2; ++n) {
        float *p = dst + g * 16 + 8 * n + 2 * t;
        *reinterpret_cast<float2 *>(p) = make_float2(acc[n][0], acc[n][1]);
        *reinterpret_cast<float2 *>(p + 8 * 16) = make_float2(acc[n][2], acc[n][3]);
    }
}

// (one warp) the 8 x 8 triangle of tokens 8 blk.. over 64 key dims (part `part`), two per lane:
// 36 products each, then warp sums into X_PTR
template <int D>
__device__ __forceinline__ void exact_triangle(uint8_t *smem, int blk, int part)
{
    const int lane = thread_id() & 31, d = part * 64 + 2 * lane;
    const float *sLam = reinterpret_cast<const float *>(smem + X_LAM);
    float *dst = reinterpret_cast<float *>(smem + X_PTR) + (blk * (D / 64) + part) * 40;
    float2 l[8];
    uint32_t k[8];
#pragma unroll
    for (int x = 0; x < 8; ++x) {
        l[x] = *reinterpret_cast<const float2 *>(sLam + lam_at<D>(8 * blk + x, d));
        k[x] = *reinterpret_cast<const uint32_t *>(smem + OFF_SK + ((8 * blk + x) * D + d) * 2);
    }
    float v[8];
    // product n = i (i + 1) / 2 + j, eight at a time
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const uint32_t w = *reinterpret_cast<const uint32_t *>(smem + OFF_SQ + ((8 * blk + i) * D + d) * 2);
        const float2 q = make_float2(__uint_as_float(w << 16), __uint_as_float(w & 0xFFFF0000u));
#pragma unroll
        for (int j = 0; j <= i; ++j) {
            const int n = i * (i + 1) / 2 + j;
            const float k0 = __uint_as_float(k[j] << 16), k1 = __uint_as_float(k[j] & 0xFFFF0000u);
            v[n % 8] = j == i ? fmaf(q.y, k1, q.x * k0)
                              : fmaf(q.y * k1, ex2(l[i].y - l[j].y), q.x * k0 * ex2(l[i].x - l[j].x));
            if (n % 8 == 7 || n == 35) {
                if (n == 35) {
#pragma unroll
                    for (int x = 4; x < 8; ++x)
                        v[x] = 0.f;
                }
                const float sum = warp_sum8(v, lane);
                if ((lane & 3) == 0)
                    dst[(n & ~7) + (lane >> 2)] = sum;
            }
        }
    }
}

constexpr int kSquareTasks = 8 + 8;

// (one warp) the task-th of kSquareTasks + 8 (D / 64) score tasks
template <int D>
__device__ __forceinline__ void exact_task(uint8_t *smem, int task)
{
    if (task < 8)
        exact_square16<D>(smem, task >> 1, task & 1);
    else if (task < kSquareTasks)
        exact_square32<D>(smem, task & 1, (task - 8) >> 1);
    else
        exact_triangle<D>(smem, (task - kSquareTasks) / (D / 64), (task - kSquareTasks) % (D / 64));
}

// (builder warps) whether the gates of a staged segment alone send it to the exact path: the
// first step of build_fast, with its arithmetic and its verdict (uniform over the builders)
template <int D>
__device__ __forceinline__ bool gates_exact(uint8_t *smem, int L, int vb)
{
    using G = Geo<D>;
    const int tid = thread_id(), dp = tid % G::DP, qt = tid / G::DP;
    const float *sG = reinterpret_cast<const float *>(smem + OFF_SG);
    float *sTot = reinterpret_cast<float *>(smem + OFF_TOT);
    zero_tail<D>(smem, L, vb, true);
    float amax = -INFINITY, r0 = 0.f, r1 = 0.f;
#pragma unroll
    for (int x = 0; x < G::TPG; ++x) {
        const float2 a = *reinterpret_cast<const float2 *>(sG + (G::TPG * qt + x) * D + 2 * dp);
        amax = fmaxf(amax, fmaxf(a.x, a.y));
        r0 = fmaf(a.x, kLog2e, r0);
        r1 = fmaf(a.y, kLog2e, r1);
    }
    *reinterpret_cast<float2 *>(sTot + qt * D + 2 * dp) = make_float2(r0, r1);
    bar_builders();
    float t0 = 0.f, t1 = 0.f;
#pragma unroll
    for (int u = 0; u < G::NQ; ++u) {
        const float2 t = *reinterpret_cast<const float2 *>(sTot + u * D + 2 * dp);
        t0 += t.x;
        t1 += t.y;
    }
    return bar_or(1, !(amax <= 0.f && t0 >= -kLamRange && t1 >= -kLamRange));
}

// (builder warps) zeros above the diagonal, in 16-byte pieces; pieces that cross the diagonal
// belong to the triangles
template <int D>
__device__ __forceinline__ void exact_zeros(uint8_t *smem)
{
#pragma unroll
    for (int x = 0; x < CH * CH / 4 / NB; ++x) {
        const int e = thread_id() + x * NB;
        const int i = e >> 4, j = (e & 15) * 4;
        if (j > i)
            *reinterpret_cast<float4 *>(smem + X_B2 + t_off(Geo<D>::ROWS, i, j)) =
                make_float4(0.f, 0.f, 0.f, 0.f);
    }
}

// the partial sums added up: every score on and below the diagonal, and the triangles' zeros.
// Returns whether one of this thread's scores is infinite or NaN.
template <int D>
__device__ __forceinline__ bool exact_scores_sum(uint8_t *smem)
{
    const int tid = thread_id();
    bool bad = false;
    auto put = [&](int i, int j, float a) {
        bad = bad || !(fabsf(a) < INFINITY);
        *reinterpret_cast<float *>(smem + X_B2 + t_off(Geo<D>::ROWS, i, j)) = rna_tf32(a);
    };
#pragma unroll
    for (int x = 0; x < 2; ++x) {
        const int e = tid + x * NT;
        const float *src = reinterpret_cast<const float *>(smem + X_P32) + e;
        put(32 + (e >> 5), e & 31, (src[0] + src[1024]) + (src[2048] + src[3072]));
    }
#pragma unroll
    for (int x = 0; x < 2; ++x) {
        const int e = tid + x * NT, u = e >> 8, r = (e >> 4) & 15, c = e & 15;
        const float *src = reinterpret_cast<const float *>(smem + X_P16) + 2 * u * 256 + (e & 255);
        const SquareUnit m = square_unit(u);
        if (u < 2 || (r >> 3) == (c >> 3))
            put(r < 8 ? m.r0 + r : m.r1 + r - 8, c < 8 ? m.c0 + c : m.c1 + c - 8, src[0] + src[256]);
    }
    {
        constexpr int NP = D / 64;
        const int blk = tid >> 6, i = (tid >> 3) & 7, j = tid & 7, n = i * (i + 1) / 2 + j;
        const float *src = reinterpret_cast<const float *>(smem + X_PTR) + blk * NP * 40;
        float a = 0.f;
        if (j <= i) {
#pragma unroll
            for (int x = 0; x < NP; ++x)
                a += src[x * 40 + n];
        }
        put(8 * blk + i, 8 * blk + j, a);
    }
    return bad;
}

// pair by pair, for segments with a gate above 0 or a score that is not finite: one float32 chain per
// score, a thread each.  Four key dims a step, since a warp's 32 keys lie in as many rows of the same
// banks: by single elements tails of 512 tokens of 9 x 16 heads, every segment here, took 928 us, now
// 517 (same bits).  A call, not inlined: inlined it left the output pass at d = 128 with 28 bytes of
// spills (4,608 tokens of 16 heads 93.5 us instead of 92.45).
template <int D>
__device__ __noinline__ void exact_scores_pairs(uint8_t *smem, int L)
{
    const int tid = thread_id();
    const float *lg = reinterpret_cast<const float *>(smem + X_LAM);
    for (int idx = tid; idx < CH * CH; idx += NT) {
        const int i = idx >> 6, j = idx & 63;
        float acc = 0.f;
        if (j <= i && i < L) {
#pragma unroll 1
            for (int dd = 0; dd < D; dd += 4) {
                const uint2 q = *reinterpret_cast<const uint2 *>(smem + OFF_SQ + (i * D + dd) * 2);
                const uint2 k = *reinterpret_cast<const uint2 *>(smem + OFF_SK + (j * D + dd) * 2);
                const float4 li = *reinterpret_cast<const float4 *>(lg + lam_at<D>(i, dd));
                const float4 lj = *reinterpret_cast<const float4 *>(lg + lam_at<D>(j, dd));
                acc = fmaf(__uint_as_float(q.x << 16) * __uint_as_float(k.x << 16), ex2(li.x - lj.x), acc);
                acc = fmaf(__uint_as_float(q.x & 0xFFFF0000u) * __uint_as_float(k.x & 0xFFFF0000u),
                           ex2(li.y - lj.y), acc);
                acc = fmaf(__uint_as_float(q.y << 16) * __uint_as_float(k.y << 16), ex2(li.z - lj.z), acc);
                acc = fmaf(__uint_as_float(q.y & 0xFFFF0000u) * __uint_as_float(k.y & 0xFFFF0000u),
                           ex2(li.w - lj.w), acc);
            }
        }
        *reinterpret_cast<float *>(smem + X_B2 + t_off(Geo<D>::ROWS, i, j)) = rna_tf32(acc);
    }
}

// (issuing thread) S^T Q~^T into D_O (TM_O0): the hi part, then the lo part
template <int D>
__device__ __forceinline__ void exact_issue_sq(uint32_t tmem, uint32_t sb)
{
#pragma unroll 1
    for (int kk = 0; kk < D / 8; ++kk) {
        const uint32_t koff = (kk >> 2) * 8192 + (kk & 3) * 32;
        mma_tf32_ts(tmem + TM_O0, tmem + Geo<D>::SHI + kk * 8, sdesc_sw128(sb + X_QT + koff, 16, 1024),
                    IDT_N64, kk > 0);
    }
#pragma unroll 1
    for (int kk = 0; kk < D / 8; ++kk) {
        const uint32_t koff = (kk >> 2) * 8192 + (kk & 3) * 32;
        const uint32_t lo = kk < 8 ? TM_SLO0 + kk * 8 : TM_SLO1 + (kk - 8) * 8;
        mma_tf32_ts(tmem + TM_O0, tmem + lo, sdesc_sw128(sb + X_QT + koff, 16, 1024), IDT_N64, 1);
    }
}

// Every operand of an exact segment, and S^T Q~^T issued: from staged inputs to A and K^^T in
// X_B2, V^T and the decayed state in TMEM, visible to the tensor core.  `next` is a word of
// shared memory (the task counter).  The state warps split the state and start S^T Q~^T while
// the builders form K^ and V^T; then both draw score tasks.
template <int D>
__device__ __forceinline__ void exact_operands(uint8_t *smem, uint32_t tmem, int L, int vb, int *next)
{
    constexpr int TASKS = kSquareTasks + 8 * (D / 64);
    if (thread_id() == 0)
        *next = 0;
    const bool up = exact_decay<D>(smem, L, vb);
    fence_proxy_async_smem();
    __syncthreads();
    if (thread_id() < NB) {
        if (!up)
            exact_zeros<D>(smem);
        exact_keys_values<D>(smem, tmem, vb);
    } else {
        exact_split_state<D>(smem, tmem);
        tc_fence_before();
        bar_staters();
        if (uniform(thread_id() >> 5) == kIssuer / 32) {
            tc_fence_after();
            if (elect_one())
                exact_issue_sq<D>(tmem, smem_u32(smem));
        }
        __syncwarp();
    }
    bool pairs = up;
    if (!up) {
        while (true) {
            int task = 0;
            if ((thread_id() & 31) == 0)
                task = atomicAdd(next, 1);
            task = __shfl_sync(0xffffffffu, task, 0);
            if (task >= TASKS)
                break;
            exact_task<D>(smem, task);
        }
        __syncthreads();
        const bool bad = exact_scores_sum<D>(smem);
        fence_proxy_async_smem();
        tc_fence_before();
        // an infinite q or k has no split into two parts (an infinity less itself is NaN)
        pairs = __syncthreads_or(bad) != 0;
    }
    if (pairs) {
        exact_scores_pairs<D>(smem, L);
        fence_proxy_async_smem();
        tc_fence_before();
        __syncthreads();
    }
}

// (issuing thread) D_O += V^T A^T and S^T += V^T K^ (S^T decayed before), 8 tokens per step.  Two
// accumulators of N = 64 and N = D columns: S^T Q~^T is not waited for, and products execute in
// issue order only on the same accumulator with the same shape.  (As one accumulator [D_O | S^T] of
// N = 64 + D after a wait for S^T Q~^T: tails of 475 tokens of 9 x 16 heads 87.8 us, one segment of
// two d = 64 heads 11.0 us; so 86.5 and 10.5.)
template <int D>
__device__ __forceinline__ void exact_issue_update(uint32_t tmem, uint32_t sb)
{
#pragma unroll 1
    for (int kk = 0; kk < CH / 8; ++kk) {
        const uint32_t koff = (kk >> 2) * (Geo<D>::ROWS * 128) + (kk & 3) * 32;
        mma_tf32_ts(tmem + TM_O0, tmem + TM_V + kk * 8, sdesc_sw128(sb + X_B2 + koff, 16, 1024), IDT_N64, 1);
        mma_tf32_ts(tmem + TM_S, tmem + TM_V + kk * 8, sdesc_sw128(sb + X_B2 + 8192 + koff, 16, 1024),
                    Geo<D>::IDT_ST, 1);
    }
}

// ---- fast path MMA groups (issuing thread) ----

// D_A = Q~ K~^T of an operand set
template <int D>
__device__ __forceinline__ void fast_issue_scores(uint32_t tmem, uint32_t sb, int iset)
{
    const uint32_t setb = sb + (uint32_t)iset * SET_BYTES;
#pragma unroll
    for (int kk = 0; kk < D / 16; ++kk) {
        const uint32_t koff = (kk >> 2) * 8192 + (kk & 3) * 32;
        mma_f16_ss(tmem + TM_A, sdesc_sw128(setb + S_QH + koff, 16, 1024),
                   sdesc_sw128(setb + S_KH + koff, 16, 1024), IDF_N64, kk > 0);
    }
}

// D_O = S^T Q~^T (A operand: the fp16 copy of S^T; the update product accumulates onto it)
template <int D>
__device__ __forceinline__ void fast_issue_sq(uint32_t tmem, uint32_t sb, int par, int iset)
{
    const uint32_t setb = sb + (uint32_t)iset * SET_BYTES;
#pragma unroll
    for (int kk = 0; kk < D / 16; ++kk) {
        const uint32_t koff = (kk >> 2) * 8192 + (kk & 3) * 32;
        mma_f16_ts(tmem + (par ? Geo<D>::O1 : TM_O0), tmem + TM_SH + kk * 8,
                   sdesc_sw128(setb + S_QH + koff, 16, 1024), IDF_N64, kk > 0);
    }
}

// D_O += V^T A^T and S^T += V^T K~, 16 tokens per step.  K~ is stored token-major for D_A
// (K-major there, K = key dim); read with N = key dim contiguous it is the MN-major B operand
// of the state update: 64-dim blocks 8 KiB apart (leading byte offset), 8-token row groups
// 1 KiB apart (stride byte offset), 16 tokens = 2 KiB per step.
// (WITH_STATE false: D_O only, for launches that discard the state)
template <int D, bool WITH_STATE = true>
__device__ __forceinline__ void fast_issue_update(uint32_t tmem, uint32_t sb, int par, int iset)
{
    const uint32_t setb = sb + (uint32_t)iset * SET_BYTES;
    const uint32_t vt = tmem + TM_V + 32 * iset;
#pragma unroll
    for (int kk = 0; kk < CH / 16; ++kk) {
        mma_f16_ts(tmem + (par ? Geo<D>::O1 : TM_O0), vt + kk * 8,
                   sdesc_sw128(setb + S_AH + kk * 32, 16, 1024), IDF_N64, 1);
        if (WITH_STATE)
            mma_f16_ts(tmem + TM_S, vt + kk * 8, sdesc_sw128(setb + S_KH + kk * 2048, 8192, 1024),
                       Geo<D>::IDF_ST, 1);
    }
}

// ---- short segments (<= kShort tokens): the per-token recurrence with the recurrent kernel's
// exact operation order (fma chains over groups of 16 key rows, group partials summed left to
// right).  The state part (every thread; gates exponentiated in place, then the state warps
// update S in TMEM, write the slot and the largest |S|, and leave each token's group partials
// in the operand sets) ...
template <int D>
__device__ __forceinline__ void short_state(uint8_t *smem, uint32_t tmem, int L, int vb, float *slot,
                                            int mset)
{
    constexpr int CW = Geo<D>::CW, NG = Geo<D>::NG;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int e_own = (warp & 3) * 32 + lane;
    const bool worker = warp >= 8 && e_own < D;
    const uint32_t lrow = (uint32_t)((warp & 3) * 32) << 16;
    const int colhalf = (warp >> 2) & 1;
    const uint16_t *sQ = reinterpret_cast<const uint16_t *>(smem + OFF_SQ);
    const uint16_t *sK = reinterpret_cast<const uint16_t *>(smem + OFF_SK);
    const uint16_t *sV = staged_v(smem, vb);
    float *sG = reinterpret_cast<float *>(smem + OFF_SG);
    float *sRed = reinterpret_cast<float *>(smem + OFF_RED) + mset * 64;
    for (int idx = tid; idx < L * D; idx += NT)
        sG[idx] = expf(sG[idx]);
    __syncthreads();
    float *part = reinterpret_cast<float *>(smem);   // [kShort][D/16 groups][D] in the operand sets
    if (warp >= 8) {
        float m = 0.f;
        if (worker) {
            float S[CW];
#pragma unroll
            for (int c0 = 0; c0 < CW; c0 += 32)
                tmem_ld32(tmem + lrow + TM_S + colhalf * CW + c0, *reinterpret_cast<float(*)[32]>(&S[c0]));
            tmem_wait_ld();
            for (int i = 0; i < L; ++i) {
                const float ve = bf16f(sV[i * D + e_own]);
#pragma unroll
                for (int mm = 0; mm < CW / 16; ++mm) {
                    float acc = 0.f;
#pragma unroll
                    for (int r = 16 * mm; r < 16 * mm + 16; ++r) {
                        const int dd = colhalf * CW + r;
                        S[r] = fmaf(sG[i * D + dd], S[r], bf16f(sK[i * D + dd]) * ve);
                        acc = fmaf(bf16f(sQ[i * D + dd]), S[r], acc);
                    }
                    part[(i * NG + colhalf * (NG / 2) + mm) * D + e_own] = acc;
                }
            }
#pragma unroll
            for (int c0 = 0; c0 < CW; c0 += 32)
                tmem_st32(tmem + lrow + TM_S + colhalf * CW + c0, *reinterpret_cast<float(*)[32]>(&S[c0]));
#pragma unroll
            for (int r = 0; r < CW; ++r) {
                m = fmaxf(m, fabsf(S[r]));
                if (slot != nullptr)
                    slot[(int64_t)(colhalf * CW + r) * D + e_own] = S[r];
            }
            tmem_wait_st();
        }
        m = warp_max(m);
        if (lane == 0)
            sRed[(warp & 7) * 8 + 4] = m;
    }
    fence_proxy_async_smem();
    __syncthreads();
}

// ... and the outputs (every thread): each token's output is the left-to-right sum of its
// eight group partials
template <int D>
__device__ __forceinline__ void short_outputs(const uint8_t *smem, int L, float *ob, int64_t tstride)
{
    constexpr int NG = Geo<D>::NG;
    const float *part = reinterpret_cast<const float *>(smem);
    for (int idx = threadIdx.x; idx < L * D; idx += NT) {
        const int i = idx / D, e = idx % D;
        float sum = part[(i * NG) * D + e];
#pragma unroll
        for (int g = 1; g < NG; ++g)
            sum += part[(i * NG + g) * D + e];
        ob[(int64_t)i * tstride + e] = sum;
    }
}

// ---- operands of a segment's state from the zero state, dS = sum_j K^_j^T v_j with K^_j =
// k_j 2^{Lam_last - Lam_j} (gla_dstate_kernel).  A
// thread of NWARPS warps owns key dim and value dim (warp mod 4) * 32 + lane and 64 / NWARPS * 4
// tokens, in groups of 16: Lam_last - Lam_j is the sum of the later groups' log2-decay and a
// running sum backwards through the group, so strong decay costs no precision.  K^ (tf32)
// goes to `op`, K-major [D][64 tokens], four tokens per store; V^T (bf16 values, exact in tf32) to
// the 64 TMEM columns at `vt`; the segment's decay G_d = 2^{Lam_last} to g[d * gstride] (device
// memory).  All inputs are loaded before the first store: with one thread per key dim walking
// the 64 tokens and storing as it went, each shared-memory load waited for the store before it
// (4,608 tokens of 16 heads through hs_linattn_prefill_scan: 112 us, now 106.5; a 512-token
// tail 18.6 us, now 17.2).  Holds one CTA-wide barrier; the caller makes the operands visible to
// the tensor core.
template <int D, int NWARPS>
__device__ __forceinline__ void dstate_operands(uint8_t *op, const uint16_t *sK, const uint16_t *sV,
                                                const float *sG, float *sTot, uint32_t tmem, uint32_t vt,
                                                float *g, int64_t gstride)
{
    constexpr int PER = 16 / NWARPS;           // token groups per thread
    const int warp = thread_id() >> 5, lane = thread_id() & 31;
    const int d = (warp & 3) * 32 + lane;
    const int g0 = (warp >> 2) * PER;
    if (d < D) {
#pragma unroll
        for (int y = 0; y < PER; ++y) {
            float run = 0.f;
#pragma unroll
            for (int x = 15; x >= 0; --x)
                run = fmaf(sG[(16 * (g0 + y) + x) * D + d], kLog2e, run);
            sTot[(g0 + y) * D + d] = run;
        }
    }
    __syncthreads();
    if (d >= D)
        return;
#pragma unroll 1
    for (int y = 0; y < PER; ++y) {
        const int t0 = 16 * (g0 + y);
        float a[16], k[16];
        uint32_t v[16];
#pragma unroll
        for (int x = 0; x < 16; ++x) {
            a[x] = sG[(t0 + x) * D + d];
            k[x] = bf16f(sK[(t0 + x) * D + d]);
            v[x] = (uint32_t)sV[(t0 + x) * D + d] << 16;
        }
        float later = 0.f;                     // log2-decay of the later groups
#pragma unroll
        for (int u = 3; u > 0; --u)
            if (u > g0 + y)
                later += sTot[u * D + d];
        float run = 0.f;
#pragma unroll
        for (int x = 15; x >= 0; --x) {
            k[x] = rna_tf32(k[x] * ex2(later + run));
            run = fmaf(a[x], kLog2e, run);
        }
        if (t0 == 0)
            g[d * gstride] = ex2(later + run);
#pragma unroll
        for (int x = 0; x < 16; x += 4)
            *reinterpret_cast<float4 *>(op + t_off(D, d, t0 + x)) =
                make_float4(k[x], k[x + 1], k[x + 2], k[x + 3]);
        tmem_st16(tmem + ((uint32_t)((warp & 3) * 32) << 16) + vt + t0, v);
    }
    tmem_wait_st();
}

// (one thread) dS^T = V^T K^ of those operands into the D TMEM columns at `dst`
template <int D>
__device__ __forceinline__ void dstate_issue(uint32_t tmem, uint32_t op, uint32_t vt, uint32_t dst)
{
#pragma unroll
    for (int kk = 0; kk < CH / 8; ++kk)
        mma_tf32_ts(tmem + dst, tmem + vt + kk * 8,
                    sdesc_sw128(op + (kk >> 2) * (D * 128) + (kk & 3) * 32, 16, 1024),
                    idesc_tf32(128, D, 0, 0), kk > 0);
}

// ---- tensor maps of the q / k / v / log-gate rows ([rows][n_heads * 128], one 64-row x
// 128-element box per head and segment) ----

inline PFN_cuTensorMapEncodeTiled_v12000 encode_fn()
{
    // resolved once per process from the driver; a pure function pointer
    static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
    if (fn == nullptr) {
        void *ptr = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &ptr, 12000,
                                             cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(ptr);
    }
    return fn;
}

template <int D>
inline bool encode_rows(CUtensorMap *m, CUtensorMapDataType dt, const void *base, uint64_t inner,
                        uint64_t rows, uint32_t elem)
{
    auto fn = encode_fn();
    if (fn == nullptr)
        return false;
    cuuint64_t gdim[2] = {inner, rows};
    cuuint64_t gstride[1] = {inner * elem};
    cuuint32_t box[2] = {(cuuint32_t)D, (cuuint32_t)CH};
    cuuint32_t estr[2] = {1, 1};
    return fn(m, dt, 2, const_cast<void *>(base), gdim, gstride, box, estr,
              CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
              CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}


}  // namespace gck
}  // namespace hs
