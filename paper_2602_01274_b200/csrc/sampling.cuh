// Seeded sampling at temperature 1: counter-based uniforms (Philox4x32-10, Salmon
// et al., "Parallel random numbers: as easy as 1, 2, 3"), Gumbel-max draws from
// logits, and the acceptance rule of speculative sampling (Eq. 5; Algorithm 1's
// accept / resample part) with commit and cache rollback.
//
// One uniform belongs to (vocabulary index v, absolute position, sequence, tag):
// counter = (v / 4, position, sequence, tag), key = the seed's two halves, word
// v % 4 of the output block, u = ((word >> 8) + 0.5) * 2^-24 in (0, 1).
// Gumbel noise -log(-log u) is evaluated in fp64 (u can be within 2^-25 of 1).
#pragma once
#include "common.cuh"
#include "control.cuh"

enum { TAG_DRAFT = 1, TAG_ACCEPT = 2, TAG_NEXT = 3 };

__device__ __forceinline__ void philox4x32_10(uint32_t c0, uint32_t c1, uint32_t c2, uint32_t c3, uint32_t k0, uint32_t k1,
                                              uint32_t (&out)[4]) {
#pragma unroll
    for (int r = 0; r < 10; ++r) {
        const uint32_t h0 = __umulhi(0xD2511F53u, c0), l0 = 0xD2511F53u * c0;
        const uint32_t h1 = __umulhi(0xCD9E8D57u, c2), l1 = 0xCD9E8D57u * c2;
        const uint32_t n0 = h1 ^ c1 ^ k0, n2 = h0 ^ c3 ^ k1;
        c0 = n0; c1 = l1; c2 = n2; c3 = l0;
        k0 += 0x9E3779B9u; k1 += 0xBB67AE85u;
    }
    out[0] = c0; out[1] = c1; out[2] = c2; out[3] = c3;
}

__device__ __forceinline__ double uniform01(uint64_t seed, uint32_t v, uint32_t pos, uint32_t seq, uint32_t tag) {
    uint32_t o[4];
    philox4x32_10(v >> 2, pos, seq, tag, (uint32_t)seed, (uint32_t)(seed >> 32), o);
    const uint32_t w = (v & 3) == 0 ? o[0] : (v & 3) == 1 ? o[1] : (v & 3) == 2 ? o[2] : o[3];
    return ((double)(w >> 8) + 0.5) * (1.0 / 16777216.0);
}

__device__ __forceinline__ double gumbel_noise(uint64_t seed, uint32_t v, uint32_t pos, uint32_t seq, uint32_t tag) {
    return -log(-log(uniform01(seed, v, pos, seq, tag)));
}

struct BestD {
    double v; int i;
};
__device__ __forceinline__ BestD best_merge(BestD a, BestD b) {       // larger value; equal values keep the lower index
    return (a.v > b.v || (a.v == b.v && a.i <= b.i)) ? a : b;
}

// The token of a finished draw.  No column wins where every score is NaN or -inf: token 0 then.
__device__ __forceinline__ int drawn_token(BestD t, int V) { return in_vocab(t.i, V); }

// Block-wide arg-max of a per-thread candidate; every thread gets the result.
// sm: at least blockDim.x / 32 entries.  All threads of the block must call it.
__device__ __forceinline__ BestD block_best(BestD t, BestD *sm, bool named_barrier) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        BestD u;
        u.v = __shfl_xor_sync(0xffffffffu, t.v, o);
        u.i = __shfl_xor_sync(0xffffffffu, t.i, o);
        t = best_merge(t, u);
    }
    const int nw = named_barrier ? 8 : (blockDim.x >> 5);
    if (named_barrier) asm volatile("bar.sync 1, 256;" ::: "memory"); else __syncthreads();
    if (lane == 0) sm[w] = t;
    if (named_barrier) asm volatile("bar.sync 1, 256;" ::: "memory"); else __syncthreads();
    BestD r = sm[0];
    for (int i = 1; i < nw; ++i) r = best_merge(r, sm[i]);
    if (named_barrier) asm volatile("bar.sync 1, 256;" ::: "memory"); else __syncthreads();
    return r;
}

// A draw from softmax(logits) by the Gumbel-max rule: argmax_v(logit_v + G_v).
// nthreads threads (threadIdx.x < nthreads) walk the row; result in every thread.
__device__ __forceinline__ int gumbel_argmax(const float *logits, int V, uint64_t seed, int pos, int seq, int tag, int nthreads,
                                             BestD *sm, bool named_barrier) {
    BestD t{-INFINITY, 0x7fffffff};
    for (int v = threadIdx.x; v < V; v += nthreads) {
        const double s = (double)__ldcg(logits + v) + gumbel_noise(seed, (uint32_t)v, (uint32_t)pos, (uint32_t)seq, (uint32_t)tag);
        if (s > t.v) { t.v = s; t.i = v; }
    }
    return drawn_token(block_best(t, sm, named_barrier), V);
}

// Block-wide sum of doubles (plain __syncthreads version, for the acceptance kernels).
__device__ __forceinline__ double block_sum_d(double v, double *sm) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    __syncthreads();
    if ((threadIdx.x & 31) == 0) sm[threadIdx.x >> 5] = v;
    __syncthreads();
    double s = 0.0;
    for (int i = 0; i < (int)(blockDim.x >> 5); ++i) s += sm[i];
    __syncthreads();
    return s;
}
__device__ __forceinline__ float block_max_f(float v, double *sm) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
    __syncthreads();
    if ((threadIdx.x & 31) == 0) sm[threadIdx.x >> 5] = (double)v;
    __syncthreads();
    float s = -INFINITY;
    for (int i = 0; i < (int)(blockDim.x >> 5); ++i) s = fmaxf(s, (float)sm[i]);
    __syncthreads();
    return s;
}

// Acceptance by rejection sampling (Eq. 5).  The transcendentals are fp64 (a step at vocabulary 32 000 and window 8 has
// 17 rows of exponentials and one of logarithms), so they are spread over the device: k_lse_parts takes every row that the
// acceptance may need in LSE_PARTS pieces, k_accept_sample the vocabulary of the resampling in PICK_PARTS pieces.  One
// block per sequence for all of it took 0.3 to 0.6 ms a step, these two 0.03 ms.
constexpr int LSE_PARTS = 4, LSE_THREADS = 512, PICK_PARTS = 32, PICK_THREADS = 256;

struct AcceptBufs {
    double2 *lse;              // [batch][2 * gamma_cap + 1 rows][LSE_PARTS] (max, sum of exponentials): p rows, then q rows
    BestD *pick;               // [batch][PICK_PARTS]
    int32_t *arrived;          // [batch], zero between launches
};

// Row blockIdx.x of sequence blockIdx.z (target rows 0 .. gamma, then draft rows), piece blockIdx.y of its vocabulary.
static __global__ void __launch_bounds__(LSE_THREADS) k_lse_parts(DevPtrs d, AcceptBufs ab, int V) {
    __shared__ double smd[32];
    const int row = blockIdx.x, part = blockIdx.y, s = blockIdx.z, gc = d.gamma_cap;
    const SeqState &st = d.st[s];
    if (!st.active || st.finished || d.n_rows[s] == 0) return;
    const bool q = row > gc;
    const int j = q ? row - gc - 1 : row;
    if (j > st.gamma - (q ? 1 : 0)) return;
    const float *x = q ? d.draft_logits + ((size_t)s * gc + j) * V : d.verify_logits + ((size_t)s * (gc + 1) + j) * V;
    const int v0 = (int)((long long)V * part / LSE_PARTS), v1 = (int)((long long)V * (part + 1) / LSE_PARTS);
    float m = -INFINITY;
    for (int v = v0 + threadIdx.x; v < v1; v += LSE_THREADS) m = fmaxf(m, __ldcg(x + v));
    m = block_max_f(m, smd);
    double e = 0.0;
    const double base = m == -INFINITY ? 0.0 : (double)m;      // (a piece of -inf only: a sum of 0, as in the whole row's sum)
    for (int v = v0 + threadIdx.x; v < v1; v += LSE_THREADS) e += exp((double)__ldcg(x + v) - base);
    e = block_sum_d(e, smd);
    if (threadIdx.x == 0) ab.lse[((size_t)s * (2 * gc + 1) + row) * LSE_PARTS + part] = make_double2((double)m, e);
}
__device__ __forceinline__ double row_lse(const double2 *p) {          // (an empty piece: -inf, 0; a NaN logit: its piece's sum)
    double M = -INFINITY, e = 0.0;
    for (int i = 0; i < LSE_PARTS; ++i) M = fmax(M, __ldcg(&p[i].x));
    for (int i = 0; i < LSE_PARTS; ++i)
        if (__ldcg(&p[i].y) != 0.0) e += __ldcg(&p[i].y) * exp(__ldcg(&p[i].x) - M);
    return M + log(e);
}

// Draft y_i is kept while r_i <= p_i(y_i) / q_i(y_i) (tested as log r <= log p - log q); on the first rejection the next
// token is drawn from norm(max(0, p - q)) of that position, when all are kept from p_{gamma+1}; the last block of a
// sequence to arrive merges the draws of the pieces, commits and rolls the caches back.
static __global__ void __launch_bounds__(PICK_THREADS) k_accept_sample(DevPtrs d, AcceptBufs ab, int V) {
    __shared__ BestD smb[32];
    __shared__ double ratio[160];                    // log r - (log p - log q) of every draft (at most 143)
    __shared__ int last;
    const int part = blockIdx.x, s = blockIdx.y, gc = d.gamma_cap;
    SeqState &st = d.st[s];
    if (!st.active || st.finished || d.n_rows[s] == 0) return;
    const int gamma = st.gamma, P = st.P;
    const uint64_t seed = st.seed;
    const int32_t *y = d.y + (size_t)s * gc;
    const float *plog = d.verify_logits + (size_t)s * (gc + 1) * V;
    const float *qlog = d.draft_logits + (size_t)s * gc * V;
    const double2 *lse = ab.lse + (size_t)s * (2 * gc + 1) * LSE_PARTS;
    for (int i = threadIdx.x; i < gamma; i += PICK_THREADS) {
        const double lp = (double)__ldcg(plog + (size_t)i * V + y[i]) - row_lse(lse + i * LSE_PARTS);
        const double lq = (double)__ldcg(qlog + (size_t)i * V + y[i]) - row_lse(lse + (gc + 1 + i) * LSE_PARTS);
        ratio[i] = log(uniform01(seed, 0u, (uint32_t)(P + i), (uint32_t)s, TAG_ACCEPT)) - (lp - lq);
    }
    __syncthreads();
    int n = 0;
    while (n < gamma && !(ratio[n] > 0.0)) ++n;      // r > p / q: reject
    const int v0 = (int)((long long)V * part / PICK_PARTS), v1 = (int)((long long)V * (part + 1) / PICK_PARTS);
    const float *p = plog + (size_t)n * V, *q = qlog + (size_t)n * V;
    BestD t{-INFINITY, 0x7fffffff};
    if (n == gamma) {
        for (int v = v0 + threadIdx.x; v < v1; v += PICK_THREADS) {
            const double sc = (double)__ldcg(p + v) + gumbel_noise(seed, (uint32_t)v, (uint32_t)(P + gamma), (uint32_t)s, TAG_NEXT);
            if (sc > t.v) { t.v = sc; t.i = v; }
        }
    } else {
        const double lsp = row_lse(lse + n * LSE_PARTS), lsq = row_lse(lse + (gc + 1 + n) * LSE_PARTS);
        for (int v = v0 + threadIdx.x; v < v1; v += PICK_THREADS) {
            const double res = exp((double)__ldcg(p + v) - lsp) - exp((double)__ldcg(q + v) - lsq);
            if (!(res > 0.0)) continue;
            const double sc = log(res) + gumbel_noise(seed, (uint32_t)v, (uint32_t)(P + n), (uint32_t)s, TAG_NEXT);
            if (sc > t.v) { t.v = sc; t.i = v; }
        }
    }
    t = block_best(t, smb, false);
    BestD *pick = ab.pick + (size_t)s * PICK_PARTS;
    if (threadIdx.x == 0) {
        pick[part] = t;
        __threadfence();
        last = atomicAdd(ab.arrived + s, 1) == PICK_PARTS - 1;
        __threadfence();
    }
    __syncthreads();
    if (!last) return;
    t = BestD{-INFINITY, 0x7fffffff};
    for (int i = 0; i < PICK_PARTS; ++i) t = best_merge(t, BestD{__ldcg(&pick[i].v), __ldcg(&pick[i].i)});
    int next = t.i;
    if (next == 0x7fffffff) {                        // p == q exactly: cannot be rejected in exact arithmetic
        BestD a{-INFINITY, 0x7fffffff};
        for (int v = threadIdx.x; v < V; v += PICK_THREADS) {
            const double pv = (double)__ldcg(p + v);
            if (pv > a.v) { a.v = pv; a.i = v; }
        }
        next = drawn_token(block_best(a, smb, false), V);
    }
    if (threadIdx.x == 0) {
        ab.arrived[s] = 0;
        commit_step(d, st, s, n, next);
    }
}
