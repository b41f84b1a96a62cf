// Chunked gated linear attention on tcgen05 tensor cores (sm_103a).
//
// Recurrence (per head):  S_t = diag(g_t) S_{t-1} + k_t v_t^T,  o_t = q_t S_t,
// g_t = exp(a_t).  The paper runs its linear layers on FLA kernels without
// printing their recurrence; this is the form the library implements, in
// the chunked matrix form.  For a segment of L <= 64 tokens inside one
// 64-token chunk of the absolute position grid, with cumulative log2-decay
// Lam_i = log2(e) * sum_{s<=i} a_s (per key dimension):
//
//   Q~_i = q_i * 2^{Lam_i}            K~_j = k_j * 2^{-Lam_j}
//   A_ij = [j <= i] * Q~_i . K~_j     (= sum_d q_id k_jd 2^{Lam_id - Lam_jd})
//   o_i  = Q~_i S + sum_j A_ij v_j
//   S'   = diag(2^{Lam_last}) (S + K~^T V)
//
// One CTA owns one (problem, head) and walks its segments in order; the
// float32 state lives in tensor memory (TMEM) for the whole call, stored
// transposed (lane = value dim e, column = key dim d).  (The RESTART
// instantiation, the output pass of the segment-parallel prefill, instead
// starts every segment from its own start state; see the kernel.)
//
// Fast chunks run kind::f16 MMA groups with fp16 operands and float32
// accumulators:  D_O = S^T Q~^T (A operand: an fp16 copy of S^T in TMEM),
// D_A = Q~ K~^T, then per 16 tokens D_O += V^T A^T (N = 64) and S^T += V^T K~
// (N = D, the K~ tile read MN-major), V^T in TMEM.  fp16 keeps the 10-bit
// mantissa of tf32 but halves the instructions (K = 16 per MMA).  The CTA's
// 16 warps form two groups in a pipeline over three operand sets in turn:
// while the eight state warps finish chunk c (the state pass, which applies
// the pending decay 2^{Lam_last}, writes a due checkpoint and refreshes the
// fp16 copy of S^T; the causal mask with each token's own score summed in
// float32 on the diagonal; the output epilogue) the eight builder warps stage
// chunk c+1 and build its operands (cumulative decay scan, Q~, K~, V^T).  Threads
// of two builder warps issue the TMA copies, one state thread the MMAs.
//
// A chunk is fast only if every fp16 operand provably stays below 2^15 in
// magnitude (|q|, |v|, |K~|, the bound 128 max|q| max|k| on |A|, and a bound
// on |S| carried from the measured state) and its total decay factor
// 2^{Lam_last} stays >= 2^-10 in every key dim (so Q~ never nears fp16's
// subnormals).  Any other chunk (strong decay, huge values) runs the exact
// path: tf32 operands (the state split into two exact tf32 parts), the
// intra-chunk matrix formed as exactly as float32 sums from factors
// 2^{Lam_i - Lam_j} <= 1 before it is rounded to tf32, and the state updated as
// diag(2^{Lam_last}) S + K^^T V with K^_j = k_j 2^{Lam_last - Lam_j}.  The
// choice depends only on the chunk's inputs and on the state it starts from,
// as does every operation order, so a resumed run reproduces a full
// recomputation bit for bit when it starts on the chunk grid.  Segments of at
// most 8 tokens run the per-token recurrence with the recurrent kernel's exact
// operation order.
//
// Every wait on an mbarrier is bounded (1 s) and is followed by a barrier that
// reduces the abort flag, so every thread of a group takes the same branch; on
// timeout the CTA reports HS_DEVERR_TIMEOUT, waits (bounded) for its own copies
// and MMAs in flight, frees its TMEM and returns.
#include "gla_chunk_common.cuh"

namespace hs {
namespace {

using namespace ptx;
using namespace gck;

// RESTART: the output pass of the segment-parallel prefill.  Every segment of a problem
// starts from its own start state (segment k of problem b from state slot ck_base[b] + k of
// p.state) instead of the state the previous segment leaves, and decides its path on that
// state as the first segment of a run does, so that a segment's outputs do not depend on
// which other segments share its CTA; no state or checkpoint is written.
template <int D, bool RESTART>
__global__ void __launch_bounds__(NT, 1)
gla_chunked_tc_kernel(const __grid_constant__ GlaParams p, const __grid_constant__ TmaMaps maps)
{
    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = reinterpret_cast<uint8_t *>(
        (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~static_cast<uintptr_t>(1023));
    const uint32_t sb = smem_u32(smem);
    float *sRed = reinterpret_cast<float *>(smem + OFF_RED);
    // [0] TMEM base, [1] abort flag, [3] run result (1 = the segment at [4] needs the exact path),
    // [4] token index where the run stopped, [5] whether that segment's build is whole (0: its gates
    // alone send it to the exact path, its inputs still staged), [6..7] decisions on the latest
    // segments (1 = fast), by segment, [9] an exact segment's look ahead, [10] its task counter,
    // [11..12] whether the build of the latest segments is whole, by segment parity
    volatile uint32_t *sMisc = reinterpret_cast<volatile uint32_t *>(smem + OFF_MISC);
    const uint32_t bar_tma = sb + OFF_BAR, bar_a = sb + OFF_BAR + 8, bar_o = sb + OFF_BAR + 16,
                   bar_s = sb + OFF_BAR + 24, bar_built = sb + OFF_BAR + 32,
                   bar_go = sb + OFF_BAR + 40;

    const int tid = threadIdx.x, warp = tid >> 5;
    // (signed: the unsigned division left the d = 128 kernel with 56 bytes of spills, which cost
    // 4 to 5 % of every tail: 29.8 us instead of 28.5 for 256 tokens of 9 x 16 heads)
    const int bh = blockIdx.x;
    const int b = bh / p.n_heads;
    const int h = bh - b * p.n_heads;
    const int n = p.n_tokens[b];
    if (n <= 0)
        return;
    // positions are token indexes of this call (32 bits); the chunk grid is `off` tokens ahead
    const int off = p.off[b];
    const int64_t tstride = (int64_t)p.n_heads * D;   // elements between consecutive tokens

    if (tid == 0) {
        mbar_init(bar_tma, 1);
        mbar_init(bar_a, 1);
        mbar_init(bar_o, 1);
        mbar_init(bar_s, 1);
        mbar_init(bar_built, 1);
        mbar_init(bar_go, 1);
        fence_mbar_init();
        sMisc[1] = 0;   // abort flag
    }
    if (warp == NB / 32)   // not the loader's warp: the first copy does not wait for it
        tmem_alloc(sb + OFF_MISC, TMEM_COLS);
    // the v buffer of the segment at token `at`
    auto vbuf = [&](int at) -> int { return (int)((((uint32_t)at + off) / CH) & 1u); };
    // (one thread) the inputs of the segment at token tok_local into the staging buffers
    auto copy_inputs = [&](int tok_local) {
        const int32_t y = p.row0[b] + tok_local;
        const int32_t x = h * D;
        mbar_arrive_expect_tx(bar_tma, Geo<D>::STAGE);
        tma_load_2d(sb + OFF_SG, &maps.g, x, y, bar_tma);
        tma_load_2d(sb + OFF_SQ, &maps.q, x, y, bar_tma);
        tma_load_2d(sb + OFF_SK, &maps.k, x, y, bar_tma);
        tma_load_2d(sb + OFF_SV + vbuf(tok_local) * 16384, &maps.v, x, y, bar_tma);
    };
    if (tid == kLoader) {
        // the first segment's inputs into L2 while the previous kernel finishes: a
        // prefetch moves no data into this SM, and L2 holds the only copy any later write
        // updates, so it is safe even if that kernel writes those inputs
        const int32_t y = (int32_t)p.row0[b];
        tma_prefetch_2d(&maps.q, h * D, y);
        tma_prefetch_2d(&maps.k, h * D, y);
        tma_prefetch_2d(&maps.v, h * D, y);
        tma_prefetch_2d(&maps.g, h * D, y);
    }
    // RESTART: only the start states come from the kernel before (the scan).  The inputs are
    // final already: the scan's CTAs released this launch after their own wait, hence after the
    // segment-state pass, which itself waited for whatever wrote them.  So the builders stage and
    // build at once, and the state warps wait below, before they load a state
    if (!RESTART)
        pdl_wait();
    if (tid == kLoader)
        copy_inputs(0);   // the barriers are this thread's own work so far: no CTA barrier needed
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = (uint32_t)uniform((int)sMisc[0]);
    const int warp_u = uniform(warp);      // for the single-thread issues (elect_one)
    const bool builder = warp < 8;
    const bool worker = !builder;                              // a state warp

    // bookkeeping of the loader (copies issued, one still in flight) and of the issuer,
    // for the waits and the abort path; every mbarrier is waited on by one thread only
    uint32_t n_tma = 1;
    bool tma_pending = true;
    uint32_t ph_tma = 0, ph_o = 0, ph_s = 0, ph_built = 0, ph_go = 0;
    uint32_t ph_a = 0;               // D_A products
    bool aborted = false;

    // L2 prefetch of the 64 tokens `ahead` tokens past token t (if any are this problem's)
    auto prefetch = [&](int t, int ahead) {
        if (n - t <= ahead)
            return;
        const int32_t y = p.row0[b] + t + ahead;
        const int32_t x = h * D;
        tma_prefetch_2d(&maps.q, x, y);
        tma_prefetch_2d(&maps.k, x, y);
        tma_prefetch_2d(&maps.v, x, y);
        tma_prefetch_2d(&maps.g, x, y);
    };
    // (loader) the same with its bookkeeping; segments after the first start on the 64-token grid,
    // so the segment kPrefetch ahead starts at tok_local + 64 * kPrefetch and is requested into L2
    auto issue_tma = [&](int tok_local) {
        copy_inputs(tok_local);
        ++n_tma;
        tma_pending = true;
        prefetch(tok_local, CH * kPrefetch);
    };
    // one thread (`who`) waits on an mbarrier; false (for every thread) if that wait ran
    // out or another thread raised the abort flag.  CTA-wide, or within the builder (id 1)
    // or state (id 2) warps; the barrier's OR reduction makes the answer uniform.
    auto wait_all = [&](int who, uint32_t bar, uint32_t &ph) -> bool {
        bool bad = false;
        if (tid == who)
            bad = !mbar_wait_bounded(bar, ph, kTimeoutNs);
        if (bad)
            sMisc[1] = 1;
        ph ^= 1;
        const bool stop = __syncthreads_or(bad || sMisc[1] != 0) != 0;
        tc_fence_after();
        if (stop)
            aborted = true;
        return !stop;
    };
    auto wait_group = [&](int id, int who, uint32_t bar, uint32_t &ph) -> bool {
        bool bad = false;
        if (tid == who)
            bad = !mbar_wait_bounded(bar, ph, kTimeoutNs);
        if (bad)
            sMisc[1] = 1;
        ph ^= 1;
        const bool stop = bar_or(id, bad || sMisc[1] != 0);
        tc_fence_after();
        if (stop)
            aborted = true;
        return !stop;
    };
    // (state warps) the next segment built and, if `o` as well, the issued products complete,
    // waited for by the issuer with one barrier
    auto wait_group_o = [&](bool o) -> bool {
        bool bad = false;
        if (tid == kIssuer)
            bad = (o && !mbar_wait_bounded(bar_o, ph_o, kTimeoutNs)) ||
                  !mbar_wait_bounded(bar_built, ph_built, kTimeoutNs);
        if (bad)
            sMisc[1] = 1;
        if (o)
            ph_o ^= 1;
        ph_built ^= 1;
        const bool stop = bar_or(2, bad || sMisc[1] != 0);
        tc_fence_after();
        if (stop)
            aborted = true;
        return !stop;
    };
    // a group barrier that also reports the abort flag, uniformly
    auto sync_group = [&](int id) -> bool {
        const bool stop = bar_or(id, sMisc[1] != 0);
        if (stop)
            aborted = true;
        return !stop;
    };
    // (builder warps) the next decision.  In the output pass it waits for the state warps, and they
    // for the kernel before: the loader waits for that kernel itself first, so that the time limit
    // covers this kernel's own work alone
    auto wait_go = [&]() -> bool {
        if (RESTART && tid == kLoader)
            pdl_wait();
        return wait_group(1, kLoader, bar_go, ph_go);
    };
    auto sync_all = [&]() -> bool {
        const bool stop = __syncthreads_or(sMisc[1] != 0) != 0;
        if (stop)
            aborted = true;
        return !stop;
    };
    auto wait_tma = [&]() -> bool {
        tma_pending = false;
        return wait_all(kLoader, bar_tma, ph_tma);
    };
    auto seg_len = [&](int at) -> int { return min(n - at, CH - (int)(((uint32_t)at + off) & (CH - 1))); };
    auto is_long = [&](int at) -> bool { return at < n && seg_len(at) > kShort; };
    // (state warps) the checkpoint due at the end of a segment, segments taken in order: the
    // next one's token index and slot number (a position modulo the interval would be a 64-bit
    // division on the state warps' chain)
    int next_ck = p.first_ck[b], ck_i = p.ck_base[b];
    auto ckpt_slot = [&](int seg_end) -> float * {
        if (RESTART || seg_end != next_ck)
            return nullptr;
        float *slot = p.ckpt_slots[ck_i++];
        next_ck = next_ck <= n - p.ckpt_interval ? next_ck + p.ckpt_interval : 0;
        if (slot == nullptr || (reinterpret_cast<uintptr_t>(slot) & 15u) != 0) {
            if (tid == kIssuer)
                report(p.d_err, slot == nullptr ? HS_DEVERR_NULL : HS_DEVERR_MISALIGNED);
            return nullptr;
        }
        return slot + (int64_t)h * D * D;
    };
    int smax = 0;   // maxima set of the last state pass (state warps)
    // largest |S| recorded by the last state pass (valid after the barrier that follows it)
    auto state_max = [&]() -> float {
        float m = 0.f;
#pragma unroll
        for (int w = 0; w < 8; ++w)
            m = fmaxf(m, sRed[smax * 64 + w * 8 + 4]);
        return m;
    };
    // the set the next pass records its maximum in: the other one, since a warp may still be
    // reading the last
    auto next_max = [&]() -> int { return smax ^= 1; };

    bool prefetched = false;   // (loader) the segments after the first requested into L2

    // incoming state -> TMEM (state warps), transposed: S^T[e][d] = state[d][e]; its
    // largest magnitude.  The builders meanwhile stage and build the first segment.
    float *st_g = p.state + ((int64_t)(RESTART ? p.ck_base[b] : b) * p.n_heads + h) * D * D;
    if (worker) {
        if (RESTART)
            pdl_wait();
        state_load<D>(smem, tmem, st_g, next_max());
        tc_fence_before();
        bar_staters();
        tc_fence_after();
    }

    // the output rows from local token t
    auto outp = [&](int t) { return p.o + (((int64_t)p.row0[b] + t) * p.n_heads + h) * D; };

    // ---- a short segment (<= kShort tokens, staged inputs already waited for, no decay
    // pending): the per-token recurrence with the recurrent kernel's exact operation order
    // (fma chains over groups of 16 key rows, group partials summed left to right)
    auto short_segment = [&](int tok_s, int L) {
        short_state<D>(smem, tmem, L, vbuf(tok_s), worker ? ckpt_slot(tok_s + L) : nullptr, next_max());
        if (tid == kLoader && tok_s + L < n)
            issue_tma(tok_s + L);
        short_outputs<D>(smem, L, outp(tok_s), tstride);
        tc_fence_before();
        __syncthreads();
        tc_fence_after();
    };

    int kseq = 0;   // long segments of the current run so far (slot of 2^{Lam_last}: kseq mod 4)
    // the decision word of the run's segment k
    auto decision = [&](int k) -> volatile uint32_t & { return sMisc[6 + (k & (kDecisions - 1))]; };
    // the guard of a built fast segment (state warps, after the wait for the builders): log-gates
    // <= 0, and every fp16 operand (Q~, K~, V, A, the fp16 copy of the state it starts from)
    // below 2^15 in magnitude.  Returns whether the segment's own inputs pass; `state_ok` says
    // whether the state (its measured magnitude, or a bound on it) passes too.
    float mk_new = 0.f, mv_new = 0.f;
    auto guard = [&](float s_mag, int kset, bool &state_ok) -> bool {
        const float *red = sRed + kset * 64;
        float mq = 0.f, mk = 0.f, mv = 0.f;
        bool ok = true;
#pragma unroll
        for (int w = 0; w < 8; ++w) {
            mq = fmaxf(mq, red[w * 8 + 0]);
            ok = ok && red[w * 8 + 1] != 0.f;
            mk = fmaxf(mk, red[w * 8 + 2]);
            mv = fmaxf(mv, red[w * 8 + 3]);
        }
        mk_new = mk;
        mv_new = mv;
        state_ok = s_mag < kF16Lim;
        return ok && (float)D * mq * mk < kF16Lim;
    };

    // ---- one exact segment, from staged inputs, no decay pending and no MMA in flight; stages
    // the next segment once its own inputs are read; leaves the final state in TMEM, writes
    // its outputs and checkpoint.  Meanwhile the builders look ahead: the next segment's inputs
    // waited for and its gates judged, into `ready` (see the main loop).
    int ready = 0;
    auto exact_segment = [&](int tok_s, int L) -> bool {
        const int seg_end = tok_s + L;
        exact_operands<D>(smem, tmem, L, vbuf(tok_s),
                          const_cast<int *>(reinterpret_cast<volatile int *>(sMisc + 10)));
        if (warp_u == kIssuer / 32) {
            tc_fence_after();
            if (elect_one()) {
                exact_issue_update<D>(tmem, sb);
                tc_commit(bar_o);
            }
            __syncwarp();
        }
        const bool ahead = is_long(seg_end);
        if (builder) {
            if (tid == kLoader && seg_end < n)
                issue_tma(seg_end);
            if (ahead && wait_group(1, kLoader, bar_tma, ph_tma)) {
                tma_pending = false;
                const bool exact = gates_exact<D>(smem, seg_len(seg_end), vbuf(seg_end));
                if (tid == kLoader)
                    sMisc[9] = exact ? 1u : 2u;
            }
        } else if (wait_group(2, kIssuer, bar_o, ph_o)) {
            // checkpoint and |S| of the final state
            state_pass<D>(smem, tmem, -1, ckpt_slot(seg_end), false, next_max());
            out_epilogue<D>(tmem, outp(tok_s), tstride, L, 0);
        }
        tc_fence_before();
        if (!sync_all())
            return false;
        tc_fence_after();
        ready = ahead ? (int)sMisc[9] : 0;
        return true;
    };

    // ---- a run of long segments on the fast path, the two groups of warps in a pipeline:
    // the builders stage and build segment k+1 while the state warps finish segment k.
    // Handoffs (each mbarrier has one waiting thread and one arriving party):
    //   bar_built: builders -> state warps, segment k built (operands, V^T, guard maxima)
    //   bar_go:    state warps -> builders, the decision on segment k is made (see kDecisions);
    //              when it is fast, it also means the products of segment k-1 are complete, so
    //              that segment k+2 may take their operand set and V^T buffer
    // A run ends after the last long segment, before a segment whose own inputs the guard
    // sends to the exact path, or before a segment whose state bound fails: a decision inside a
    // run only has a bound on the state it starts from (that state is still being computed), so
    // such a segment starts a new run, whose first decision reads the measured state exactly as
    // a run resumed from a checkpoint at that segment does.  The groups then meet CTA-wide.
    // No MMA is in flight at either end.
    // The builders run up to one segment ahead of the decisions: segment k+1 goes into a third
    // operand set and V^T buffer while segment k is judged and segment k-1 finishes, and only its
    // hand-over waits for "go" on segment k.  Its staged rows are overwritten by the copy of segment
    // k+2 as soon as q, k and the gates are consumed (v has two staging buffers).  With two sets and
    // one copy at the hand-over, the builders' chain (build, hand over, issue, wait for the
    // decision, wait for the copy) set the pace at ~9 k cycles a segment; the D_A and copy issues
    // (~1 k cycles of single-thread work) and two barriers a segment are off it, and the state
    // warps' passes run in rolled halves (less code, fewer registers): 4 x 32 heads of 16,384
    // tokens 1,088 -> 977 us, 256-token tails of 9 x 16 heads 28.5 -> 26.7 us, 81 packed tails 248 ->
    // 234 us.
    auto builder_run = [&](int rtok, bool waited) {
        int iset = 0;
        while (true) {
            const int L = seg_len(rtok);
            if (!waited && !wait_group(1, kLoader, bar_tma, ph_tma))
                return;
            waited = false;
            tma_pending = false;
            if (tid == kLoader && !prefetched) {
                // once the first segment has landed (the state and the first segment are
                // not queued behind these): the next kPrefetch segments into L2
                prefetched = true;
                for (int j = 1; j <= kPrefetch; ++j)
                    prefetch(rtok + L, CH * (j - 1));
            }
            float mq, mk;
            bool ok;
            const bool built = build_fast<D>(smem, L, vbuf(rtok), iset, kseq & 3, mq, mk, ok);
            fence_proxy_async_smem();
            if (built && rtok + L < n) {
                // q, k and the gates are consumed: stage the next segment (long or short); an exact
                // decision on this one reloads it
                if (!sync_group(1))
                    return;
                if (tid == kLoader) {
                    ++n_tma;
                    tma_pending = true;
                }
                if (warp_u == 1 && elect_one())
                    copy_inputs(rtok + L);
                __syncwarp();
            }
            build_values<D>(smem, tmem, vbuf(rtok), iset, built, mq, mk, ok);
            tc_fence_before();
            // every warp's part done, and the decision on the segment before
            if (kseq > 0 ? !wait_go() || decision(kseq - 1) == 0 : !sync_group(1))
                return;
            if (tid == kLoader) {
                sMisc[11 + (kseq & 1)] = built ? 1u : 0u;
                mbar_arrive(bar_built);
            }
            if (!built || !is_long(rtok + L)) {
                wait_go();   // the run ends with this segment
                return;
            }
            rtok += L;
            iset = iset == 2 ? 0 : iset + 1;
            ++kseq;
        }
    };
    // The issuing thread's product groups (state warps; each call ends converged)
    auto issue_sq = [&](int par, int iset) {       // D_O = S^T Q~^T
        if (warp_u == kIssuer / 32) {
            const int pu = uniform(par), iu = uniform(iset);
            if (elect_one())
                fast_issue_sq<D>(tmem, sb, pu, iu);
        }
        __syncwarp();
    };
    auto issue_update = [&](int par, int iset) {   // (RESTART: D_O only, the state is discarded)
        if (warp_u == kIssuer / 32) {
            const int pu = uniform(par), iu = uniform(iset);
            tc_fence_after();
            if (elect_one()) {
                fast_issue_update<D, !RESTART>(tmem, sb, pu, iu);
                tc_commit(bar_o);
            }
        }
        __syncwarp();
    };
    auto issue_scores = [&](int iset) {            // D_A = Q~ K~^T
        if (warp_u == kIssuer / 32) {
            const int iu = uniform(iset);
            if (elect_one()) {
                fast_issue_scores<D>(tmem, sb, iu);
                tc_commit(bar_a);
            }
        }
        __syncwarp();
    };
    // (another state warp) the L2 requests of the segment kPrefetch past the next one
    auto request = [&](int next) {
        if (warp_u == NB / 32 + 7 && elect_one())
            prefetch(next, CH * kPrefetch);
        __syncwarp();
    };
    // Per segment the state warps' chain is: built (with the products of the segment before),
    // decision, state pass, D_A, the mask of A beside the issue of D_O, the issue of the update;
    // the outputs of the segment before are written behind that, while the update runs.
    auto state_run = [&](int rtok) {
        int iset = 0;
        bool drained = true;   // no products outstanding
        uint32_t stop = 0;   // why the run ended: 0 done or short segment, 1 exact, 2 new run
        int pend_L = 0;        // the previous segment's tokens
        float mk_cur = 0.f, mv_cur = 0.f;
        while (true) {
            // the segment at rtok built, and the products of the previous one complete
            tc_fence_before();
            if (!wait_group_o(kseq > 0))
                return;
            drained = true;
            // first segment of a run: the measured state (float32 maximum of the last state pass
            // or of the loaded state).  Else the state it starts from is bounded by the fp16
            // copy's largest |S| at the previous segment's start plus that segment's largest
            // update, 64 max|k| max|v| (the decay factors are <= 1)
            bool state_ok;
            const bool inputs_ok =
                guard(kseq > 0 ? (state_max() + 64.0f * mk_cur * mv_cur) * kBoundMargin : state_max(), iset,
                      state_ok);
            const bool fast = inputs_ok && state_ok;
            if (tid == kIssuer) {
                decision(kseq) = fast ? 1u : 0u;
                mbar_arrive(bar_go);
            }
            const int L = seg_len(rtok);
            request(rtok + L);
            if (!fast) {
                stop = kseq > 0 && inputs_ok ? 2u : 1u;   // the exact path or a new run takes this segment
                break;
            }
            issue_scores(iset);
            mk_cur = mk_new;
            mv_cur = mv_new;
            state_pass<D>(smem, tmem, kseq > 0 ? (kseq - 1) & 3 : -1,
                          kseq > 0 ? ckpt_slot(rtok) : nullptr, true,
                          next_max());
            tc_fence_before();
            // the state in place, and D_A of this segment
            if (!wait_group(2, kIssuer, bar_a, ph_a))
                return;
            issue_sq(kseq & 1, iset);
            a_build<D>(smem, tmem, iset);
            fence_proxy_async_smem();
            tc_fence_before();
            if (!sync_group(2))
                return;
            issue_update(kseq & 1, iset);
            if (kseq > 0)
                out_epilogue<D>(tmem, outp(rtok - pend_L), tstride, pend_L, (kseq - 1) & 1);
            drained = false;
            pend_L = L;
            rtok += L;
            iset = iset == 2 ? 0 : iset + 1;
            ++kseq;
            if (!is_long(rtok))
                break;
        }
        if (kseq > 0) {
            if (!drained && !wait_group(2, kIssuer, bar_o, ph_o))
                return;
            state_pass<D>(smem, tmem, (kseq - 1) & 3, ckpt_slot(rtok), false, next_max());
            out_epilogue<D>(tmem, outp(rtok - pend_L), tstride, pend_L, (kseq - 1) & 1);
            tc_fence_before();
            if (!sync_group(2))
                return;
        }
        if (tid == kIssuer) {
            sMisc[3] = stop;
            sMisc[4] = (uint32_t)rtok;
            sMisc[5] = sMisc[11 + (kseq & 1)];
        }
    };

    // RESTART: the state warps' side of a run in which every segment decides on, and is
    // computed from, its own start state, loaded before its decision (the first segment's is
    // loaded before the run); the builders' side is builder_run, unchanged.  No product reads
    // the float32 state in TMEM here (the state update is skipped and D_O reads the fp16 copy),
    // so the next segment's state is loaded while the previous segment's products run.
    int loaded = 0;   // index of the segment whose start state is in TMEM (state warps)
    auto seg_idx = [&](int at) -> int { return (int)(((uint32_t)at + off) / CH); };
    // (issuing thread) the start state of the segment at `at` into L2, one bulk request
    auto prefetch_state = [&](int at) {
        const float *src = st_g + (int64_t)seg_idx(at) * p.n_heads * D * D;
        asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(src),
                     "r"((uint32_t)(D * D * 4))
                     : "memory");
    };
    auto state_run_restart = [&](int rtok) {
        int iset = 0;
        bool drained = true;
        uint32_t stop = 0;   // 0 done or short segment, 1 exact
        int pend_L = 0;
        while (true) {
            const int L = seg_len(rtok);
            if (loaded != seg_idx(rtok)) {
                state_load<D>(smem, tmem, st_g + (int64_t)seg_idx(rtok) * p.n_heads * D * D, next_max());
                loaded = seg_idx(rtok);
            }
            // the loaded state (its TMEM columns and its largest |S|) visible to the group, the
            // segment built, the products of the previous one complete
            tc_fence_before();
            if (!wait_group_o(kseq > 0))
                return;
            drained = true;
            bool state_ok;
            const bool fast = guard(state_max(), iset, state_ok) && state_ok;
            if (tid == kIssuer) {
                decision(kseq) = fast ? 1u : 0u;
                mbar_arrive(bar_go);
            }
            request(rtok + L);
            if (!fast) {
                stop = 1;   // the exact path takes this segment
                break;
            }
            issue_scores(iset);
            if (tid == kIssuer && is_long(rtok + L))
                prefetch_state(rtok + L);   // read by the load at the end of this segment
            __syncwarp();
            state_pass<D>(smem, tmem, -1, nullptr, true, next_max());   // the fp16 copy of S for D_O
            tc_fence_before();
            if (!wait_group(2, kIssuer, bar_a, ph_a))
                return;
            issue_sq(kseq & 1, iset);
            a_build<D>(smem, tmem, iset);
            fence_proxy_async_smem();
            tc_fence_before();
            if (!sync_group(2))
                return;
            issue_update(kseq & 1, iset);
            if (kseq > 0)
                out_epilogue<D>(tmem, outp(rtok - pend_L), tstride, pend_L, (kseq - 1) & 1);
            drained = false;
            pend_L = L;
            rtok += L;
            iset = iset == 2 ? 0 : iset + 1;
            ++kseq;
            if (!is_long(rtok))
                break;
            // the next segment's start state, while this segment's products run and the
            // builders build it (this segment's fp16 copy is made: TMEM S is free)
            state_load<D>(smem, tmem, st_g + (int64_t)seg_idx(rtok) * p.n_heads * D * D, next_max());
            loaded = seg_idx(rtok);
        }
        if (kseq > 0) {
            if (!drained && !wait_group(2, kIssuer, bar_o, ph_o))
                return;
            out_epilogue<D>(tmem, outp(rtok - pend_L), tstride, pend_L, (kseq - 1) & 1);
            tc_fence_before();
            if (!sync_group(2))
                return;
        }
        if (tid == kIssuer) {
            sMisc[3] = stop;
            sMisc[4] = (uint32_t)rtok;
            sMisc[5] = sMisc[11 + (kseq & 1)];
        }
    };

    // failure-detection hook (tests only): every thread joins one CTA-wide wait on an
    // mbarrier that nothing completes before the first decision (bar_go, phase 0); the
    // loader's bounded wait runs out and raises the abort flag, and the CTA leaves through
    // the abort path below
    if (p.stall_for_test) {
        uint32_t ph_stall = 0;
        wait_all(kLoader, bar_go, ph_stall);
    }

    // `ready`, the long segment at tok after an exact one: its inputs are staged and waited for,
    // and its gates alone send it to the exact path (1) or do not (2); 0: not looked at
    int tok = 0;
    while (!aborted && tok < n) {
        if (RESTART && worker && loaded != seg_idx(tok)) {
            // this segment's own start state (the previous segment's state is not used)
            state_load<D>(smem, tmem, st_g + (int64_t)seg_idx(tok) * p.n_heads * D * D, next_max());
            tc_fence_before();
            bar_staters();
            tc_fence_after();
            loaded = seg_idx(tok);
        }
        const int L = seg_len(tok);
        if (L <= kShort) {
            // a leading or trailing short segment (its inputs are staged or in flight)
            if (!wait_tma())
                break;
            short_segment(tok, L);
            tok += L;
            continue;
        }
        if (ready != 1) {
            if (builder)
                builder_run(tok, ready == 2);
            else if constexpr (RESTART)
                state_run_restart(tok);
            else
                state_run(tok);
            ready = 0;
            if (!sync_all())
                break;
            tc_fence_after();
            const uint32_t stop = sMisc[3];
            tok = (int)sMisc[4];
            kseq = 0;
            if (stop == 0)
                continue;
            // the segment at tok takes the exact path (1) or starts a new run (2).  Its inputs
            // are still staged if its build stopped early (sMisc[5] == 0); else restage them (the
            // copy of a later segment may be in flight)
            if (sMisc[5] != 0) {
                if (tid == kLoader) {
                    if (tma_pending && !mbar_wait_bounded(bar_tma, ph_tma, kTimeoutNs))
                        sMisc[1] = 1;
                    if (tma_pending)
                        ph_tma ^= 1;
                    issue_tma(tok);
                }
                if (stop == 2)
                    continue;   // the new run waits for the copy
                if (!wait_tma())
                    break;
            }
        }
        // every thread runs the exact segment
        const int Lx = seg_len(tok);
        if (!exact_segment(tok, Lx))
            break;
        tok += Lx;
    }

    if (!aborted) {
        if (!RESTART)
            state_store<D>(tmem, st_g);   // final state back to global memory, row = key dim
    } else {
        // let this CTA's own copies and MMAs drain (bounded) before its memory goes away
        if (tid == kLoader) {
            report(p.d_err, HS_DEVERR_TIMEOUT);
            if (n_tma > 0)
                mbar_wait_bounded(bar_tma, (n_tma - 1) & 1, kTimeoutNs);
        }
        __syncwarp();
        if (warp_u == kIssuer / 32 && elect_one()) {
            tc_commit(bar_s);
            mbar_wait_bounded(bar_s, ph_s, kTimeoutNs);
        }
        __syncwarp();
    }
    tc_fence_before();
    __syncthreads();
    if (warp == NB / 32) {
        tc_fence_after();
        tmem_dealloc(tmem, TMEM_COLS);
    }
}


}  // namespace

bool gla_chunked_tc_supported(int d)
{
    return d == 64 || d == 128;
}

namespace {

template <int D, bool RESTART>
cudaError_t launch_tc(const GlaParams &p, cudaStream_t s)
{
    TmaMaps maps;
    const uint64_t inner = (uint64_t)p.n_heads * D;
    // rows up to the last token any problem has: copies never read beyond the tokens the
    // caller passed (boxes reaching further are zero-filled), so q/k/v/log_g may be
    // offset views whose last rows run past the end of the allocation
    uint64_t rows = 0;
    for (int32_t b = 0; b < p.batch; ++b) {
        const uint64_t r = (uint64_t)p.row0[b] + (uint64_t)p.n_tokens[b];
        rows = r > rows ? r : rows;
    }
    if (rows == 0)
        return cudaSuccess;
    if (!encode_rows<D>(&maps.q, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, p.q, inner, rows, 2) ||
        !encode_rows<D>(&maps.k, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, p.k, inner, rows, 2) ||
        !encode_rows<D>(&maps.v, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, p.v, inner, rows, 2) ||
        !encode_rows<D>(&maps.g, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, p.log_g, inner, rows, 4))
        return cudaErrorInvalidValue;
    static std::atomic<uint64_t> smem_set{0};
    const unsigned grid = (unsigned)p.batch * (unsigned)p.n_heads;
    return launch_pdl_big_smem(gla_chunked_tc_kernel<D, RESTART>, dim3(grid), dim3(NT), SMEM_BYTES, s,
                               smem_set, p, maps);
}

}  // namespace

cudaError_t launch_gla_chunked_tc(const GlaParams &p, int d, cudaStream_t s)
{
    if (d == 128)
        return launch_tc<128, false>(p, s);
    if (d == 64)
        return launch_tc<64, false>(p, s);
    return cudaErrorNotSupported;
}

cudaError_t launch_gla_chunked_tc_restart(const GlaParams &p, int d, cudaStream_t s)
{
    if (d == 128)
        return launch_tc<128, true>(p, s);
    if (d == 64)
        return launch_tc<64, true>(p, s);
    return cudaErrorNotSupported;
}

}  // namespace hs
