// The tails of the forward kernels: they take the loop's decisions (Eq. 6 / Eq. 7 /
// Algorithm 1) on the device, in the launch that computed what they decide on.
#pragma once
#include "fwd_phases.cuh"
#include "sampling.cuh"

namespace fwd {

// ------------------------------------------------------------------ tails (one block per sequence)

__device__ __forceinline__ float hidden_at(const Args &a, const Ctx &c, int r, int i) {
    return __ldcg(a.d.xres + (size_t)r * a.m.cfg.d_model + i) * c.inv_rms[r] * __bfloat162float(a.m.normf[i]);
}

// 1/rms of the final residual rows of sequence s, for the final RMSNorm the tails apply (MMA warps of one block, a row
// per warp).
__device__ __forceinline__ void tail_inv_rms(Ctx &c, const Args &a, int s) {
    const int dm = a.m.cfg.d_model;
    for (int j = c.warp; j < c.n_rows[s]; j += MMA_WARPS) {
        const int r = s * a.g.rps + j;
        const float4 *x = reinterpret_cast<const float4 *>(a.d.xres + (size_t)r * dm);
        float ss = 0.f;
        for (int i = c.lane; i < dm / 4; i += 32) { const float4 v = __ldcg(x + i); ss += v.x * v.x + v.y * v.y + v.z * v.z + v.w * v.w; }
        ss = warp_sum(ss);
        if (c.lane == 0) c.inv_rms[r] = rsqrtf(ss / (float)dm + a.m.cfg.rms_eps);
    }
    bsync();
}

// End of one draft forward (Eq. 6): y_i, h_i queued for the pre-verification model, cache length.
__device__ __forceinline__ void tail_draft(Ctx &c, const Args &a, int s) {
    const DevPtrs &d = a.d;
    SeqState &st = d.st[s];
    const int n_in = c.n_rows[s], dm = a.m.cfg.d_model;
    if (n_in == 0) return;
    const int gamma = st.gamma, n_pend = st.n_pend, r_last = s * a.g.rps + n_in - 1;
    int y_new = 0;
    if (st.mode == PACER_SAMPLE)                          // y_i ~ q_i by the Gumbel-max rule at the token's position
        y_new = gumbel_argmax(d.draft_logits + ((size_t)s * d.gamma_cap + gamma) * a.m.cfg.vocab, a.m.cfg.vocab, st.seed,
                              st.P + gamma, s, TAG_DRAFT, MMA_THREADS, reinterpret_cast<BestD *>(c.scratch), true);
    const bool queue = !st.sched;                        // with prescribed windows nothing is pre-verified
    for (int jj = 0; queue && jj < n_in; ++jj) {
        float *dst = d.hpend + ((size_t)s * (d.block_b + 1) + n_pend + jj) * dm;
        for (int i = threadIdx.x; i < dm; i += MMA_THREADS) dst[i] = hidden_at(a, c, s * a.g.rps + jj, i);
    }
    bsync();
    if (threadIdx.x == 0) {
        for (int jj = 0; queue && jj < n_in; ++jj)
            d.hpend_e[s * (d.block_b + 1) + n_pend + jj] = (jj == n_in - 1) ? gamma + 1 : 0;
        d.y[(size_t)s * d.gamma_cap + gamma] = st.mode == PACER_SAMPLE ? y_new : d.row_arg[r_last];
        if (queue) st.n_pend = n_pend + n_in;
        st.gamma = gamma + 1;
        st.len_D += n_in;
        st.n_draft_fwd += 1;
    }
}

// End of a pre-verification call (Eq. 7 + the block test of Algorithm 1).
__device__ __forceinline__ void tail_mb(Ctx &c, const Args &a, int s) {
    const DevPtrs &d = a.d;
    SeqState &st = d.st[s];
    const int n = c.n_rows[s], dm = a.m.cfg.d_model;
    if (n == 0) return;
    for (int j = c.warp; j < n; j += MMA_WARPS) {         // a row per warp: its 1/rms and the two scores in one pass
        const int r = s * a.g.rps + j, e = c.row_tok[r];
        if (e == 0) continue;
        const float2 *x = reinterpret_cast<const float2 *>(d.xres + (size_t)r * dm);
        const __nv_bfloat162 *gn = reinterpret_cast<const __nv_bfloat162 *>(a.m.normf);
        const __nv_bfloat162 *h0 = reinterpret_cast<const __nv_bfloat162 *>(a.m.head_b), *h1 = h0 + dm / 2;
        float ss = 0.f, z0 = 0.f, z1 = 0.f;
        for (int i = c.lane; i < dm / 2; i += 32) {
            const float2 v = __ldcg(x + i), g = __bfloat1622float2(gn[i]), p = __bfloat1622float2(h0[i]), q = __bfloat1622float2(h1[i]);
            ss += v.x * v.x + v.y * v.y;
            z0 += v.x * g.x * p.x + v.y * g.y * p.y;
            z1 += v.x * g.x * q.x + v.y * g.y * q.y;
        }
        ss = warp_sum(ss); z0 = warp_sum(z0); z1 = warp_sum(z1);
        const float inv = rsqrtf(ss / (float)dm + a.m.cfg.rms_eps);
        if (c.lane == 0) d.alpha[(size_t)s * d.gamma_cap + e - 1] = 1.f / (1.f + expf((z0 - z1) * inv));
    }
    bsync();
    if (threadIdx.x == 0) {
        const int b = d.block_b, gamma = st.gamma;
        const float *ab = d.alpha + (size_t)s * d.gamma_cap + (gamma - b);
        float stat;
        if (d.criterion == 1) { stat = ab[0]; for (int i = 1; i < b; ++i) stat = fminf(stat, ab[i]); }
        else if (d.criterion == 2) stat = ab[b - 1];
        else { stat = 0.f; for (int i = 0; i < b; ++i) stat += ab[i]; stat /= (float)b; }
        int stop = 0;
        if (st.t0 >= 0.f && stat <= st.t_k) stop = 1;
        if (gamma + b > st.gamma_max) stop = 1;
        if (stop) st.drafting = 0;
        else { st.t_k = st.t_k * d.rho; st.k_round += 1; }
        if (gamma == b) {                     // first call of the step: where its drafts begin in the cache
            int n_hist = 0;
            while (n_hist < n && c.row_tok[s * a.g.rps + n_hist] == 0) ++n_hist;
            st.mb_start = st.len_B + n_hist;
        }
        st.len_B += n;
        st.n_pend = 0;
        st.n_mb_calls += 1;
    }
}

// End of a prefill chunk: the caches grew; the draft's hidden rows are the
// history rows the pre-verification model is prefilled with.
__device__ __forceinline__ void tail_prefill(Ctx &c, const Args &a, int s, int which) {
    const DevPtrs &d = a.d;
    const int n = c.n_rows[s], dm = a.m.cfg.d_model;
    if (n == 0) return;
    if (which == PACER_DRAFT)
        for (int j = 0; j < n; ++j) {
            const int r = s * a.g.rps + j;
            for (int i = threadIdx.x; i < dm; i += MMA_THREADS) d.hidden[(size_t)r * dm + i] = hidden_at(a, c, r, i);
        }
    if (threadIdx.x == 0) {
        SeqState &st = d.st[s];
        if (which == PACER_TARGET) st.len_T += n;
        else if (which == PACER_DRAFT) st.len_D += n;
        else st.len_B += n;
    }
}

// End of one autoregressive target step (Eq. 1).  pick: the sampled token when the forward has drawn it already, else -1.
__device__ __forceinline__ void tail_ar(Ctx &c, const Args &a, int s, int pick) {
    if (c.n_rows[s] == 0) return;
    const DevPtrs &d = a.d;
    SeqState &st = d.st[s];
    int tok = d.row_arg[s * a.g.rps];
    if (st.mode == PACER_SAMPLE && pick >= 0) tok = pick;
    else if (st.mode == PACER_SAMPLE)
        tok = gumbel_argmax(d.verify_logits + (size_t)s * (d.gamma_cap + 1) * a.m.cfg.vocab, a.m.cfg.vocab, st.seed, st.P, s,
                            TAG_NEXT, MMA_THREADS, reinterpret_cast<BestD *>(c.scratch), true);
    if (threadIdx.x != 0) return;
    d.x[(size_t)s * d.max_ctx + st.P] = tok;
    st.P += 1;
    st.len_T += 1;
    st.n_target_fwd += 1;
    st.n_steps += 1;
    if (st.P - st.n_prompt >= st.max_new) st.finished = 1;
}

}  // namespace fwd
