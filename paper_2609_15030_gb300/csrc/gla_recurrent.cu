// Gated linear attention, one token at a time on CUDA cores:
//     S_t = diag(g_t) S_{t-1} + k_t v_t^T,   o_t = q_t S_t,   g_t = exp(a_t).
// (The paper runs its linear layers on FLA kernels and prints no recurrence;
// this is the form the library implements.)
//
// One CTA owns 64 value columns of one (problem, head) and keeps that part of the d x d
// float32 state in registers for the whole call, as 16 x 2 blocks (16 key rows, 2 value
// columns) per thread; a warp's lanes are column pairs, so every state load and store of a
// warp is 256 contiguous bytes of one row.  The kernel is bound by the state's bytes (a short
// call reads and writes 64 KiB per head and computes a few tokens in between), so what matters
// is that the loads of one CTA overlap the arithmetic and stores of others: 256 threads of 64
// registers (8 bytes spilled) over 32 KiB of state put four CTAs on an SM.  72 problems of 16 heads and 2-8
// tokens (160 MB): 29.5 us = 5.4 TB/s; 31.7 without the later CTAs' states requested into L2, 35.1
// without the CTA's own lines requested first either (its tokens' alone: 32.9), and 38.2 us with
// whole heads (16 x 4 blocks, 125 registers, two CTAs per SM) then.  Tokens are staged eight at a
// time in shared memory, and their rows of q, k and g are read back 16 bytes at a time, one
// broadcast per four rows.  A thread's two columns go through one f32x2 instruction (scalar
// instructions cost 1.3 us more; with each value stored twice in shared memory, so that a load
// gives the pair, 3.7 us more, from the 43 KiB it takes).
//
// Per token the arithmetic is fixed: g = expf(a); every element becomes
// fmaf(g_d, S[d][e], k_d * v_e); partial dot products over each group of 16
// consecutive key rows run as one sequential fma chain in increasing row
// order; o_e is the left-to-right sum of the d/16 group partials.  The chunked
// tensor-core kernel computes short segments with exactly these operations
// (d = 128), so the two kernels agree bit for bit on them.  The order depends
// only on each token's inputs and the incoming state, so resuming from any
// checkpoint reproduces a full recomputation bit for bit.
#include "hs_internal.cuh"
#include "sm100_ptx.cuh"

namespace hs {
namespace {

using namespace ptx;

constexpr int kTokBlock = 8;

// four values of a bf16 row
__device__ __forceinline__ float4 bf16x4(const uint16_t *p)
{
    const uint2 w = *reinterpret_cast<const uint2 *>(p);
    return make_float4(__uint_as_float(w.x << 16), __uint_as_float(w.x & 0xFFFF0000u),
                       __uint_as_float(w.y << 16), __uint_as_float(w.y & 0xFFFF0000u));
}

constexpr int kCols = 64;             // value columns of a CTA

// CTA = (problem, head, block of 64 columns).  Thread (cg, rg) holds rows [16*rg, 16*rg+16) and
// the CTA's columns 2*cg, 2*cg+1.
template <int D>
__global__ void __launch_bounds__((kCols / 2) * (D / 16), D == 128 ? 4 : 7)
gla_recurrent_kernel(const __grid_constant__ GlaParams p, unsigned ahead)
{
    constexpr int NCG = kCols / 2;    // column pairs (lanes)
    constexpr int NRG = D / 16;       // row groups of 16
    constexpr int NTH = NCG * NRG;
    constexpr int NCB = D / kCols;    // column blocks per head
    __shared__ __align__(16) float sq[kTokBlock][D], sk[kTokBlock][D], sg[kTokBlock][D];
    __shared__ __align__(16) float sv[kTokBlock][kCols];
    __shared__ __align__(16) float spart[kTokBlock][NRG][kCols];

    const int bh = blockIdx.x / NCB;
    const int e0 = (blockIdx.x - bh * NCB) * kCols;
    const int b = bh / p.n_heads;
    const int h = bh - b * p.n_heads;
    const int n = p.n_tokens[b];
    if (n <= 0)
        return;
    const int tid = threadIdx.x;
    {
        // the first tokens' rows and the state into L2, while the kernel before finishes and ahead of
        // the loads below (a prefetch moves no data into this SM, so it is safe even if that kernel
        // writes them): the tokens' loads, needed first, are issued last, and waited a whole trip to
        // memory behind the state's
        constexpr int LB = D / 64;   // 128-byte lines of one bf16 row (a float row is 2 LB)
        const int t = tid / (5 * LB), l = tid % (5 * LB);
        if (t < min(n, kTokBlock)) {
            const int64_t at = (((int64_t)p.row0[b] + t) * p.n_heads + h) * D;
            const char *src = l < LB       ? reinterpret_cast<const char *>(p.q + at) + 128 * l
                              : l < 2 * LB ? reinterpret_cast<const char *>(p.k + at) + 128 * (l - LB)
                              : l < 3 * LB ? reinterpret_cast<const char *>(p.v + at) + 128 * (l - 2 * LB)
                                           : reinterpret_cast<const char *>(p.log_g + at) + 128 * (l - 3 * LB);
            asm volatile("prefetch.global.L2 [%0];" ::"l"(src));
        }
    }
    // the CTA's 64 columns of a state row are two lines
    if (tid < 2 * D)
        asm volatile("prefetch.global.L2 [%0];" ::"l"(p.state + ((int64_t)b * p.n_heads + h) * D * D +
                                                      (tid >> 1) * D + e0 + (tid & 1) * 32));
    pdl_wait_and_release();
    // the state of a CTA that starts about when this one ends (see the launch)
    const unsigned nx = blockIdx.x + ahead;
    if (tid < 2 * D && nx < gridDim.x) {
        const unsigned nbh = nx / NCB;
        if (p.n_tokens[nbh / p.n_heads] > 0)
            asm volatile("prefetch.global.L2 [%0];" ::"l"(p.state + (int64_t)nbh * D * D + (tid >> 1) * D +
                                                          (nx - nbh * NCB) * kCols + (tid & 1) * 32));
    }
    const int cg = tid % NCG;
    const int rg = tid / NCG;
    int next_ck = p.first_ck[b];      // tokens up to the next checkpoint, and its slot
    int ck = p.ck_base[b];

    // this thread's first element of a state
    const int64_t elem = (int64_t)h * D * D + 16 * rg * D + e0 + 2 * cg;
    float *st = p.state + (int64_t)b * p.n_heads * D * D + elem;
    uint64_t S[16];   // S[r] = state row 16*rg + r, columns e0 + 2*cg, + 1
#pragma unroll
    for (int r = 0; r < 16; ++r)
        S[r] = *reinterpret_cast<const uint64_t *>(st + r * D);

    for (int t0 = 0; t0 < n; t0 += kTokBlock) {
        const int tb = min(kTokBlock, n - t0);
        const int64_t row0 = ((int64_t)p.row0[b] + t0) * p.n_heads + h;
        for (int idx = tid; idx < tb * (D / 4); idx += NTH) {
            const int tt = idx / (D / 4), d = (idx % (D / 4)) * 4;
            const int64_t at = (row0 + (int64_t)tt * p.n_heads) * D + d;
            const float4 a = *reinterpret_cast<const float4 *>(p.log_g + at);
            *reinterpret_cast<float4 *>(&sq[tt][d]) = bf16x4(p.q + at);
            *reinterpret_cast<float4 *>(&sk[tt][d]) = bf16x4(p.k + at);
            *reinterpret_cast<float4 *>(&sg[tt][d]) = make_float4(expf(a.x), expf(a.y), expf(a.z), expf(a.w));
        }
        for (int idx = tid; idx < tb * (kCols / 4); idx += NTH) {
            const int tt = idx / (kCols / 4), e = (idx % (kCols / 4)) * 4;
            *reinterpret_cast<float4 *>(&sv[tt][e]) =
                bf16x4(p.v + (row0 + (int64_t)tt * p.n_heads) * D + e0 + e);
        }
        __syncthreads();
#pragma unroll 1
        for (int tt = 0; tt < tb; ++tt) {
            const uint64_t v2 = *reinterpret_cast<const uint64_t *>(&sv[tt][2 * cg]);
            uint64_t acc = 0;
#pragma unroll
            for (int r4 = 0; r4 < 16; r4 += 4) {
                const int i = 16 * rg + r4;
                const float4 g4 = *reinterpret_cast<const float4 *>(&sg[tt][i]);
                const float4 k4 = *reinterpret_cast<const float4 *>(&sk[tt][i]);
                const float4 q4 = *reinterpret_cast<const float4 *>(&sq[tt][i]);
                const float g[4] = {g4.x, g4.y, g4.z, g4.w}, kk[4] = {k4.x, k4.y, k4.z, k4.w},
                            qq[4] = {q4.x, q4.y, q4.z, q4.w};
#pragma unroll
                for (int x = 0; x < 4; ++x) {
                    uint64_t &s = S[r4 + x];
                    s = fma2(pair(g[x], g[x]), s, mul2(pair(kk[x], kk[x]), v2));
                    acc = fma2(pair(qq[x], qq[x]), s, acc);
                }
            }
            *reinterpret_cast<uint64_t *>(&spart[tt][rg][2 * cg]) = acc;
            if (t0 + tt + 1 == next_ck) {
                float *slot = p.ckpt_slots[ck++];
                next_ck = next_ck <= n - p.ckpt_interval ? next_ck + p.ckpt_interval : 0;
                if (slot == nullptr) {
                    if (tid == 0)
                        report(p.d_err, HS_DEVERR_NULL);
                } else if ((reinterpret_cast<uintptr_t>(slot) & 15u) != 0) {
                    if (tid == 0)
                        report(p.d_err, HS_DEVERR_MISALIGNED);
                } else {
                    slot += elem;
#pragma unroll
                    for (int r = 0; r < 16; ++r)
                        *reinterpret_cast<uint64_t *>(slot + r * D) = S[r];
                }
            }
        }
        if (t0 + tb >= n) {
            // final state out before the output reduction, so the store drains behind it
#pragma unroll
            for (int r = 0; r < 16; ++r)
                *reinterpret_cast<uint64_t *>(st + r * D) = S[r];
        }
        __syncthreads();
        for (int idx = tid; idx < tb * kCols; idx += NTH) {
            const int tt = idx / kCols, e = idx % kCols;
            float sum = spart[tt][0][e];
#pragma unroll
            for (int g = 1; g < NRG; ++g)
                sum += spart[tt][g][e];
            p.o[(row0 + (int64_t)tt * p.n_heads) * D + e0 + e] = sum;
        }
        __syncthreads();
    }
}

}  // namespace

cudaError_t launch_gla_recurrent(const GlaParams &p, int d, int sm_count, cudaStream_t s)
{
    const unsigned grid = (unsigned)p.batch * (unsigned)p.n_heads * (unsigned)(d / kCols);
    // each CTA requests the state three CTAs per SM further on at d = 128 (an SM holds four), five at
    // d = 64 (seven).  d = 128, 72 problems of 16 heads, 2-8 tokens: 31.7 us without, 29.9 two, 29.5
    // three, 30.2 four, 31.7 five, 32.6 eight further; 32 problems of 32 heads, 1-2 tokens: 24.6, 22.7,
    // 22.7, 22.8, 23.3, 24.1.  d = 64, 72 problems of 16 heads, 2-8 tokens: 10.24 us without, 9.98 two,
    // 9.95 three, 9.92 four, 9.92 five, 9.88 six, 10.25 eight; 128 of 32 heads, 1-2 tokens: 22.6, 21.6,
    // 21.2, 20.9, 20.7, 20.7, 20.8; 384 of 32 heads, 2-4 tokens: 64.9, 63.8, 63.6, 63.4, 63.3, 63.6, 65.4
    if (d == 128)
        return launch_pdl(gla_recurrent_kernel<128>, dim3(grid), dim3(256), 0, s, p, 3u * sm_count);
    return launch_pdl(gla_recurrent_kernel<64>, dim3(grid), dim3(128), 0, s, p, 5u * sm_count);
}

}  // namespace hs
