// The state scan of the segment-parallel prefill (hs_linattn_prefill_scan).
//
// Over a problem's tail [pos0, pos0 + n), split into segments at the multiples of 64 of the
// absolute position grid, the recurrence S_t = diag(g_t) S_{t-1} + k_t v_t^T is linear in
// the state: for a segment of tokens [s, e),
//     S_e = diag(G) S_s + dS,   G = prod_{s<=t<e} g_t = 2^{sum_t a_t log2 e},
// where dS is the segment's state when it starts from the zero state.  The first pass of the
// prefill (gla_dstate.cu) computes every segment's dS and G at once; this kernel chains them:
// per (problem, head) and state element, S_{n+1} = G_n S_n + dS_n over the segments in order,
// recording each segment's start state S_n (the last pass computes the outputs from it), the
// checkpoint at every multiple of C and the final state.  Every step is an elementwise fma,
// so a run resumed at a checkpoint on the grid repeats the same operations from there:
// resumed and full computations agree bit for bit.
//
// One CTA per (problem, head, block of 256 state elements); thread i owns four consecutive
// elements (d, e..e+3) of one key row d (a float4), and the D/4 lanes of a row (a warp at
// D = 128, a half-warp at D = 64) are consecutive.  The first pass leaves G_n of row d at
// element (d, 0) of segment n's start-state block: the row's first lane, which owns that
// element, reads it there, passes it to the row's other lanes with a shuffle and then
// overwrites it with the start state.  The chain only streams: each thread copies its float4
// of dS_n (the first lane also G_n) for the next kStages segments into its own slots of
// shared-memory rings with cp.async (one commit group per segment, so that waiting for the
// oldest group never waits for a newer copy), applies the oldest and refills its slots.
//
// The pass is bound by memory: per segment and head 64 KiB of dS in, 64 KiB of start state out.
// What it needs is the same number of bytes in flight on every SM: small CTAs whose rings let
// seven of them on an SM give 16 heads at d = 128 (1,024 CTAs) 6.7 per SM on all 152, while with
// CTAs of 128 threads and a 40 KiB ring the first 512 / 5 SMs to be free took five each.  dS is
// read for the last time here, so its lines go first when L2 needs room for the start states, which
// the output pass reads next.  4,608 tokens of 16 heads, the whole call: 99.3 us with five CTAs of
// 128 threads, 94.6 with four, 93.1 as it is (1 us of it the L2 policy).
#include "hs_internal.cuh"

namespace hs {
namespace {

constexpr int kThreads = 64;         // a float4 per thread: 256 state elements per CTA
constexpr int kChunk = 64;           // segments on the 64-token absolute grid
constexpr int kStages = 28;          // segments whose dS and G are in flight: 28.4 KiB of rings, so
                                     // that seven CTAs fit on an SM
constexpr int kRows = kThreads / 16;  // key rows of a CTA (d = 64; half as many at d = 128)
constexpr uint32_t kSmemBytes = kStages * (16 * kThreads + 4 * kRows);   // the rings

// the L2 policy of lines read for the last time
__device__ __forceinline__ uint64_t policy_evict_first()
{
    uint64_t p;
    asm("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(p));
    return p;
}

__device__ __forceinline__ void cp_async16(void *smem_dst, const void *gmem_src, uint64_t policy)
{
    asm volatile("cp.async.cg.shared.global.L2::cache_hint [%0], [%1], 16, %2;" ::"r"(
                     (uint32_t)__cvta_generic_to_shared(smem_dst)),
                 "l"(gmem_src), "l"(policy)
                 : "memory");
}

__device__ __forceinline__ void cp_async4(void *smem_dst, const void *gmem_src)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(
                     (uint32_t)__cvta_generic_to_shared(smem_dst)),
                 "l"(gmem_src)
                 : "memory");
}

__device__ __forceinline__ void cp_async_commit()
{
    asm volatile("cp.async.commit_group;" ::: "memory");
}

// wait until at most kStages - 1 of this thread's commit groups are pending
__device__ __forceinline__ void cp_async_wait_oldest()
{
    asm volatile("cp.async.wait_group %0;" ::"n"(kStages - 1) : "memory");
}

template <int D>
__global__ void __launch_bounds__(kThreads)
gla_scan_kernel(const __grid_constant__ ScanParams p)
{
    constexpr int BLOCKS = D * D / (4 * kThreads);   // CTAs per (problem, head)
    constexpr int W = D / 4;                         // lanes per key row
    extern __shared__ float4 smem[];
    // dS of the segments in flight and their G, one per key row
    float4 (*sRing)[kThreads] = reinterpret_cast<float4 (*)[kThreads]>(smem);
    float (*sGate)[kRows] = reinterpret_cast<float (*)[kRows]>(smem + kStages * kThreads);
    const int lane = threadIdx.x & 31;
    const bool row_lead = (lane & (W - 1)) == 0;
    const int bh = blockIdx.x / BLOCKS;
    const int blk = blockIdx.x - bh * BLOCKS;
    const int b = bh / p.n_heads;
    const int h = bh - b * p.n_heads;
    const int f = (blk * kThreads + threadIdx.x) * 4;  // first of this thread's 4 elements
    const int64_t pos0 = p.pos0[b];
    const int64_t end = pos0 + p.n_tokens[b];
    const int64_t hs_ = (int64_t)h * D * D + f;        // offset inside one [n_heads][D][D] state
    const int64_t sstride = (int64_t)p.n_heads * D * D;
    const int C = p.ckpt_interval;
    float4 *st = reinterpret_cast<float4 *>(p.state + (int64_t)b * sstride + hs_);
    pdl_wait_and_release();
    float4 S = *st;
    const uint64_t last_read = policy_evict_first();
    // the rings: one commit group per segment (empty past the last), kStages in flight.  Segments
    // are counted and addresses stepped: with 64-bit positions divided and compared for each, 4,608
    // tokens of 16 heads took 1 us more
    const int n_seg = end > pos0 ? (int)((end + kChunk - 1) / kChunk - pos0 / kChunk) : 0;
    const float *ld_dS = p.dS + (int64_t)p.seg_base[b] * sstride + hs_;   // the next segment to copy
    float *Sn = p.Sn + (int64_t)p.seg_base[b] * sstride + hs_;            // the current segment
    const float *ld_G = Sn;
    int to_load = n_seg;
    auto refill = [&](int slot) {
        if (to_load > 0) {
            cp_async16(&sRing[slot][threadIdx.x], ld_dS, last_read);
            if (row_lead)
                cp_async4(&sGate[slot][threadIdx.x / W], ld_G);
            ld_dS += sstride;
            ld_G += sstride;
            --to_load;
        }
        cp_async_commit();
    };
    for (int j = 0; j < kStages; ++j)
        refill(j);
    // the segment that ends at the next checkpoint position (-1: none within the call) and its
    // slot pointer, read one checkpoint ahead (the pointer array ends with the call)
    const int per_ck = C / kChunk;
    const int last_ck = (int)(end / kChunk - 1 - pos0 / kChunk);   // the last segment that ends on the grid
    int ck_seg = -1;
    int32_t ck = p.ck_base[b];
    float *cs_next = nullptr;
    if (C > 0 && p.ckpt_slots != nullptr && (pos0 / C + 1) * C <= end) {
        ck_seg = (int)((pos0 / C + 1) * per_ck - 1 - pos0 / kChunk);
        cs_next = p.ckpt_slots[ck];
    }
    int slot = 0;
#pragma unroll 1
    for (int i = 0; i < n_seg; ++i) {
        cp_async_wait_oldest();
        const float4 dq = sRing[slot][threadIdx.x];
        const float G = __shfl_sync(0xffffffffu, row_lead ? sGate[slot][threadIdx.x / W] : 0.f,
                                    lane & ~(W - 1));
        // the start state replaces the gate the first pass left in the row's first float4
        *reinterpret_cast<float4 *>(Sn) = S;
        Sn += sstride;
        S.x = fmaf(G, S.x, dq.x);
        S.y = fmaf(G, S.y, dq.y);
        S.z = fmaf(G, S.z, dq.z);
        S.w = fmaf(G, S.w, dq.w);
        refill(slot);     // after the slot is consumed: its next copies cannot overtake the reads
        slot = slot + 1 == kStages ? 0 : slot + 1;
        if (i == ck_seg) {
            float *cs = cs_next;
            ck_seg = ck_seg + per_ck <= last_ck ? ck_seg + per_ck : -1;
            if (ck_seg >= 0)
                cs_next = p.ckpt_slots[++ck];
            if (cs == nullptr || (reinterpret_cast<uintptr_t>(cs) & 15u) != 0) {
                if (threadIdx.x == 0 && blk == 0 && h == 0)
                    report(p.d_err, cs == nullptr ? HS_DEVERR_NULL : HS_DEVERR_MISALIGNED);
            } else {
                *reinterpret_cast<float4 *>(cs + hs_) = S;
            }
        }
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    *st = S;
}

}  // namespace

cudaError_t launch_gla_scan(const ScanParams &p, int d, cudaStream_t s)
{
    const unsigned bh = (unsigned)p.batch * (unsigned)p.n_heads;
    if (bh == 0)
        return cudaSuccess;
    static std::atomic<uint64_t> smem_set[2];
    if (d == 128)
        return launch_pdl_big_smem(gla_scan_kernel<128>, dim3(bh * (128 * 128 / (4 * kThreads))),
                                   dim3(kThreads), kSmemBytes, s, smem_set[0], p);
    if (d == 64)
        return launch_pdl_big_smem(gla_scan_kernel<64>, dim3(bh * (64 * 64 / (4 * kThreads))),
                                   dim3(kThreads), kSmemBytes, s, smem_set[1], p);
    return cudaErrorNotSupported;
}

}  // namespace hs
