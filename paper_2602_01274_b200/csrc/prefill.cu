// Prompt prefill.  The rows of a prompt are known on the host and there are many of them, so unlike the decoding forwards
// this path is bound by the tensor cores: per layer three kinds of GEMM launches and one of flash attention over chunks of
// up to 2048 rows (a chunk reads the weights once; the forward kernel took 128 rows at a time and re-read them, its 8
// phase warps and 9 grid barriers per layer idle the tensor cores most of the time).
//
// GEMM: 128 token rows x up to 256 weight rows per tile on tcgen05, operands by one bulk copy each per 64 columns (both
// are stored in the 128-byte-swizzle order the tensor cores read), three stages of 64 KB, two accumulators so that a
// tile's epilogue runs under the next tile's products.  The token rows come as split bf16 (value + remainder: 16 mantissa
// bits, as in the forward kernels): two products accumulate into the same tile.  Epilogues do the decoder's row-wise step:
// rotary embedding + cache append, residual add + next operand, SwiGLU; 1/rms is applied to the output of the projection
// that follows a norm, from shares of sum(x^2) left by the epilogue before.  A stage is 64 KB for 0.52 us of tensor time at 1965
// MHz.  The widest projections are bound by the tensor cores at the clock that the power cap leaves them (2047 rows x 38400 x
// 7168, two planes: 1.47 ms = 1.54 PFLOP/s, tensor pipe 95 % active at 1.43 GHz, L2 50 % busy); narrower ones keep the pipe 70
// to 84 % active, with L2 no busier.
// The tensor cores truncate when they add to an accumulator, so a tile's products over 512 columns are taken out and added
// in ordinary fp32 (registers of the epilogue warps) while the next 512 run into the other accumulator: with one
// accumulator over all of K the logits behind a 300-token prompt were 1.7 times as far from an fp64 forward (1.4e-4 against
// 8e-5 at 14 layers of width 7168).
//
// Attention: pf_attention.cuh.
#include "prefill.h"

#include <cuda.h>

#include <algorithm>

#include "fwd_stream.cuh"

namespace pf {

using namespace fwd;

constexpr int SEG = 8;                     // k blocks of 64 columns accumulated inside the tensor cores
constexpr int TM = 128, STAGES = 3, A_BYTES = 32 * 1024, B_BYTES = 32 * 1024;
constexpr int EPI_WARPS = 8, THREADS_G = 32 * (EPI_WARPS + 2);
constexpr int SMEM_G = STAGES * (A_BYTES + B_BYTES) + 1024;

// Operand of a projection: per tile of 128 rows, per 64 columns, the 8-row atoms of values and then those of the rounding
// remainders (only as many atoms as the last tile has rows), an atom being 1 KB in the 128-byte-swizzle layout.
__device__ __forceinline__ size_t operand_index(int r, int k, int K, int rows) {
    const int m = r >> 7, left = rows - (m << 7), na = left >= TM ? 16 : (left + 7) >> 3;
    return (size_t)m * K * 256 + ((size_t)(k >> 6) * (2 * na) + ((r & 127) >> 3)) * 512 + (r & 7) * 64 + ((((k >> 3) & 7) ^ (r & 7)) << 3) + (k & 7);
}
__device__ __forceinline__ int operand_plane(int r, int rows) {          // elements from a value to its remainder
    const int left = rows - (r & ~127);
    return (left >= TM ? 16 : (left + 7) >> 3) * 512;
}
__device__ __forceinline__ void split2(float a, float b, uint32_t &hi, uint32_t &lo) {
    const __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
    hi = *reinterpret_cast<const uint32_t *>(&h);
    lo = pack_bf16x2(a - __low2float(h), b - __high2float(h));
}
// eight consecutive columns (k a multiple of 8): one 16-byte chunk of each plane
__device__ __forceinline__ void store8(bf16 *base, int r, int k, int K, int rows, const float (&v)[8]) {
    uint4 hi, lo;
    split2(v[0], v[1], hi.x, lo.x); split2(v[2], v[3], hi.y, lo.y); split2(v[4], v[5], hi.z, lo.z); split2(v[6], v[7], hi.w, lo.w);
    bf16 *p = base + operand_index(r, k, K, rows);
    *reinterpret_cast<uint4 *>(p) = hi;
    *reinterpret_cast<uint4 *>(p + operand_plane(r, rows)) = lo;
}

// ------------------------------------------------------------------ input rows

struct InArgs {
    const int32_t *tok;                    // [batch][max_ctx]
    const bf16 *embed, *gain, *normf;
    float *x;
    bf16 *xg;
    float *ssq;
    int32_t max_ctx, d, nj, c0, rows, input;
    float eps;
};
// One block per row: x, x * gain as the first operand, sum(x^2).
__global__ void __launch_bounds__(256) k_pf_input(const InArgs a) {
    __shared__ float red[33];
    const int r = blockIdx.x, s = r / a.nj, j = r - s * a.nj;
    float *x = a.x + (size_t)r * a.d;
    float scale = 1.f, ss = 0.f;
    if (a.input == HIDDEN) {
        for (int k = threadIdx.x; k < a.d; k += 256) { const float v = x[k]; ss += v * v; }
        scale = rsqrtf(block_sum(ss, red) / (float)a.d + a.eps);
        ss = 0.f;
    }
    const bf16 *e = a.input == EMBED ? a.embed + (size_t)a.tok[(size_t)s * a.max_ctx + a.c0 + j] * a.d : nullptr;
    for (int k = threadIdx.x * 8; k < a.d; k += 256 * 8) {
        float v[8], w[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            v[i] = a.input == EMBED ? __bfloat162float(e[k + i]) : x[k + i] * scale * __bfloat162float(a.normf[k + i]);
            ss += v[i] * v[i];
            w[i] = v[i] * __bfloat162float(a.gain[k + i]);
        }
#pragma unroll
        for (int i = 0; i < 8; ++i) x[k + i] = v[i];
        store8(a.xg, r, k, a.d, a.rows, w);
    }
    ss = block_sum(ss, red);
    if (threadIdx.x == 0) a.ssq[r] = ss;
}

// ------------------------------------------------------------------ projections

enum Epi { E_QKV = 0, E_RES = 1, E_GU = 2 };

struct GArgs {
    const bf16 *A, *W;                     // operand; weights of the layer, [K/64][2 * MT atoms]
    int32_t K, MT, N;                      // columns; 16-row weight tiles; weight rows
    int32_t rows, mt, w, nt;               // token rows, tiles of 128 of them; 16-row weight tiles of a tile; such tiles
    int32_t rpad;                          // rows padded to 128: stride of ssq
    const float *ssq_in;                   // parts [nss][rpad] of the norm before (QKV, GU)
    int32_t nss;
    float eps;
    // QKV
    float *q;
    bf16 *kc, *vc;                         // caches of the layer: [seq][Hkv][max_ctx][hd] for the values, kv_lo further the remainders
    size_t kv_lo;
    const float2 *rope;
    int32_t H, Hkv, hd, max_ctx, nj, c0;
    // RES
    float *x, *ssq_out;
    const bf16 *gain;
    // next operand: xg (RES), act (GU)
    bf16 *out;
    int32_t out_k;                         // its columns
    int32_t *abort_flag;
};

__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t (&v)[16]) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
                 : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]), "=r"(v[8]), "=r"(v[9]),
                   "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15]) : "r"(taddr));
}
__device__ __forceinline__ void tmem_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

// The row-wise step on 16 accumulator columns (weight rows n0 ..) of token row r.
template <int EPI>
__device__ __forceinline__ void tile_epilogue(const GArgs &a, int r, int seq, int pos, int n0, float inv, const float (&v)[16], const float4 (&xr)[4], float &ss) {
    if (EPI == E_GU) {                     // eight gate rows, then the eight up rows of the same columns
        float o[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) { const float g = v[i] * inv; o[i] = g / (1.f + expf(-g)) * (v[8 + i] * inv); }
        store8(a.out, r, n0 >> 1, a.out_k, a.rows, o);
    } else if (EPI == E_RES) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            float y[8], w[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                y[i] = v[h * 8 + i] + reinterpret_cast<const float *>(xr)[h * 8 + i];
                ss += y[i] * y[i];
            }
            float4 *dst = reinterpret_cast<float4 *>(a.x + (size_t)r * a.N + n0 + h * 8);
            dst[0] = make_float4(y[0], y[1], y[2], y[3]); dst[1] = make_float4(y[4], y[5], y[6], y[7]);
            const uint4 gw = *reinterpret_cast<const uint4 *>(a.gain + n0 + h * 8);
            const __nv_bfloat162 *gp = reinterpret_cast<const __nv_bfloat162 *>(&gw);
#pragma unroll
            for (int i = 0; i < 4; ++i) { w[2 * i] = y[2 * i] * __low2float(gp[i]); w[2 * i + 1] = y[2 * i + 1] * __high2float(gp[i]); }
            store8(a.out, r, n0 + h * 8, a.out_k, a.rows, w);
        }
    } else {
        const int hd = a.hd, half = hd >> 1, h = n0 / hd, w = n0 - h * hd;
        if (h < a.H + a.Hkv) {             // eight rotary pairs (channels ii, ii + hd/2) of a q or k head
            const int ii = w >> 1;
            const float4 *cs4 = reinterpret_cast<const float4 *>(a.rope + (size_t)pos * half + ii);
            float y0[8], y1[8];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const float4 c = cs4[i];
                const float p0 = v[4 * i] * inv, p1 = v[4 * i + 1] * inv, p2 = v[4 * i + 2] * inv, p3 = v[4 * i + 3] * inv;
                y0[2 * i] = p0 * c.x - p1 * c.y; y1[2 * i] = p1 * c.x + p0 * c.y;
                y0[2 * i + 1] = p2 * c.z - p3 * c.w; y1[2 * i + 1] = p3 * c.z + p2 * c.w;
            }
            if (h < a.H) {
                const float sc = rsqrtf((float)hd);
                float *q = a.q + (size_t)r * (a.H * hd) + h * hd + ii;
#pragma unroll
                for (int i = 0; i < 2; ++i) {
                    reinterpret_cast<float4 *>(q)[i] = make_float4(y0[4 * i] * sc, y0[4 * i + 1] * sc, y0[4 * i + 2] * sc, y0[4 * i + 3] * sc);
                    reinterpret_cast<float4 *>(q + half)[i] = make_float4(y1[4 * i] * sc, y1[4 * i + 1] * sc, y1[4 * i + 2] * sc, y1[4 * i + 3] * sc);
                }
            } else {
                bf16 *k = a.kc + (((size_t)seq * a.Hkv + (h - a.H)) * a.max_ctx + pos) * hd + ii;
                uint4 hi, lo;
                split2(y0[0], y0[1], hi.x, lo.x); split2(y0[2], y0[3], hi.y, lo.y); split2(y0[4], y0[5], hi.z, lo.z); split2(y0[6], y0[7], hi.w, lo.w);
                *reinterpret_cast<uint4 *>(k) = hi; *reinterpret_cast<uint4 *>(k + a.kv_lo) = lo;
                split2(y1[0], y1[1], hi.x, lo.x); split2(y1[2], y1[3], hi.y, lo.y); split2(y1[4], y1[5], hi.z, lo.z); split2(y1[6], y1[7], hi.w, lo.w);
                *reinterpret_cast<uint4 *>(k + half) = hi; *reinterpret_cast<uint4 *>(k + a.kv_lo + half) = lo;
            }
        } else {
            bf16 *p = a.vc + (((size_t)seq * a.Hkv + (h - a.H - a.Hkv)) * a.max_ctx + pos) * hd + w;
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                uint4 hi, lo;
                split2(v[8 * i] * inv, v[8 * i + 1] * inv, hi.x, lo.x); split2(v[8 * i + 2] * inv, v[8 * i + 3] * inv, hi.y, lo.y);
                split2(v[8 * i + 4] * inv, v[8 * i + 5] * inv, hi.z, lo.z); split2(v[8 * i + 6] * inv, v[8 * i + 7] * inv, hi.w, lo.w);
                *reinterpret_cast<uint4 *>(p + 8 * i) = hi; *reinterpret_cast<uint4 *>(p + a.kv_lo + 8 * i) = lo;
            }
        }
    }
}

// Persistent: block b computes the tiles b, b + grid, ...; row tiles vary fastest, so that the blocks that run together
// share their weights in L2.  Warps 0..7 epilogues (warp w reads accumulator lanes 32 (w % 4) .., the first or second half
// of the tile's columns), warp 8 copies, warp 9 tensor cores.
template <int EPI>
__global__ void __launch_bounds__(THREADS_G, 1) k_pf_gemm(const __grid_constant__ GArgs a) {
    extern __shared__ __align__(1024) unsigned char smem[];
    __shared__ uint64_t full[STAGES], empty[STAGES], acc_full[2], acc_empty[2];
    __shared__ uint32_t tmem_slot;
    const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
    if (smem_u32(smem) & 1023u) {                        // (the same in every block)
        if (threadIdx.x == 0) atomicCAS(a.abort_flag, 0, 13);
        return;
    }
    FwdBufs fb;
    fb.abort_flag = a.abort_flag;
    if (threadIdx.x == 0) {
        for (int i = 0; i < STAGES; ++i) { mbar_init(full + i, 1); mbar_init(empty + i, 1); }
        for (int i = 0; i < 2; ++i) { mbar_init(acc_full + i, 1); mbar_init(acc_empty + i, EPI_WARPS); }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        fence_proxy_async();
    }
    if (warp == 9) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_slot)), "r"(512) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_slot;
    const int tiles = a.mt * a.nt, nkb = a.K >> 6;
    const int na_last = (a.rows - ((a.mt - 1) << 7) + 7) >> 3;

    if (warp == 8) {
        if (lane == 0) {
            asm volatile("fence.proxy.async;" ::: "memory");          // the operand was written by ordinary stores of earlier kernels
            uint64_t pol_a, pol_w;
            asm volatile("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(pol_a));
            asm volatile("createpolicy.fractional.L2::evict_normal.b64 %0, 1.0;" : "=l"(pol_w));
            int n = 0;
            bool ok = true;
            for (int t = blockIdx.x; t < tiles && ok; t += gridDim.x) {
                const int m = t % a.mt, u0 = (t / a.mt) * a.w, wu = min(a.w, a.MT - u0), na = m == a.mt - 1 ? na_last : 16;
                const bf16 *A = a.A + (size_t)m * a.K * 256, *W = a.W + (size_t)u0 * 1024;
                for (int kb = 0; kb < nkb; ++kb, ++n) {
                    const int slot = n % STAGES;
                    ok = wait_bar(fb, empty + slot, (((uint32_t)(n / STAGES)) & 1u) ^ 1u, 20, n);
                    if (!ok) break;
                    unsigned char *st = smem + slot * (A_BYTES + B_BYTES);
                    mbar_expect_tx(full + slot, (uint32_t)(na * 2048 + wu * 2048));
                    bulk_g2s(st, A + (size_t)kb * (2 * na) * 512, (uint32_t)(na * 2048), full + slot, pol_a);
                    bulk_g2s(st + A_BYTES, W + (size_t)kb * (2 * a.MT) * 512, (uint32_t)(wu * 2048), full + slot, pol_w);
                }
            }
            for (int j = max(0, n - STAGES); j < n; ++j)              // no copy may be in flight when the block ends
                for (unsigned it = 0; it < MBAR_SPIN_LIMIT && !mbar_try_wait(full + j % STAGES, ((uint32_t)(j / STAGES)) & 1u); ++it) {}
        }
    } else if (warp == 9) {
        const uint32_t on = elect_lane();                // (all lanes wait, one issues)
        int n = 0, i = 0;
        bool ok = true;
        for (int t = blockIdx.x; t < tiles && ok; t += gridDim.x, ++i) {
            const int m = t % a.mt, u0 = (t / a.mt) * a.w, wu = min(a.w, a.MT - u0), na = m == a.mt - 1 ? na_last : 16;
            const uint32_t idesc = umma_idesc(wu * 16);
            for (int kb = 0; kb < nkb && ok; ++kb, ++n) {
                if (kb % SEG == 0) {
                    if (kb) { umma_commit_if(on, acc_full + (i & 1)); ++i; }
                    ok = __all_sync(0xffffffffu, wait_bar(fb, acc_empty + (i & 1), (((uint32_t)(i >> 1)) & 1u) ^ 1u, 21, i));
                    if (!ok) break;
                }
                const uint32_t acc = tmem + (uint32_t)(i & 1) * 256u;
                const int slot = n % STAGES;
                ok = __all_sync(0xffffffffu, wait_bar(fb, full + slot, ((uint32_t)(n / STAGES)) & 1u, 22, n));
                if (!ok) break;
                tc_fence_after();
                const uint32_t a0 = smem_u32(smem + slot * (A_BYTES + B_BYTES)), b0 = a0 + A_BYTES, a1 = a0 + (uint32_t)na * 1024u;
#pragma unroll
                for (int k16 = 0; k16 < 4; ++k16) {
                    umma_if(on, acc, umma_desc(a0 + k16 * 32), umma_desc(b0 + k16 * 32), idesc, (kb % SEG > 0 || k16 > 0) ? 1u : 0u);
                    umma_if(on, acc, umma_desc(a1 + k16 * 32), umma_desc(b0 + k16 * 32), idesc, 1u);
                }
                umma_commit_if(on, empty + slot);
            }
            umma_commit_if(on, acc_full + (i & 1));
        }
    } else {
        const int quad = warp & 3, half = warp >> 2;
        int i = 0;                                       // segments so far
        for (int t = blockIdx.x; t < tiles; t += gridDim.x) {
            const int m = t % a.mt, nti = t / a.mt, u0 = nti * a.w, wu = min(a.w, a.MT - u0);
            const int r = m * TM + quad * 32 + lane;
            const bool live = r < a.rows;
            int seq = 0, pos = 0;
            float inv = 0.f;
            if (EPI != E_RES) {                          // 1/rms of the row, while the tensor cores work
                float s0 = 0.f, s1 = 0.f, s2 = 0.f, s3 = 0.f;
                int p = 0;
                const float *sp = a.ssq_in + r;
                for (; p + 4 <= a.nss; p += 4) {
                    s0 += __ldg(sp + (size_t)p * a.rpad); s1 += __ldg(sp + (size_t)(p + 1) * a.rpad);
                    s2 += __ldg(sp + (size_t)(p + 2) * a.rpad); s3 += __ldg(sp + (size_t)(p + 3) * a.rpad);
                }
                for (; p < a.nss; ++p) s0 += __ldg(sp + (size_t)p * a.rpad);
                inv = rsqrtf(((s0 + s1) + (s2 + s3)) / (float)a.K + a.eps);
            }
            if (EPI == E_QKV) { seq = r / a.nj; pos = a.c0 + r - seq * a.nj; }
            const int ub = half ? (wu + 1) >> 1 : 0, un = (half ? wu : (wu + 1) >> 1) - ub;      // this warp's 16-column units
            float sum[8][16];
            bool ok = true;
            for (int kb = 0; kb < nkb && ok; kb += SEG, ++i) {
                ok = wait_bar(fb, acc_full + (i & 1), ((uint32_t)(i >> 1)) & 1u, 23, i);
                ok = __all_sync(0xffffffffu, ok);
                tc_fence_after();
                const uint32_t acc = tmem + (uint32_t)(i & 1) * 256u + ((uint32_t)(quad * 32) << 16) + (uint32_t)ub * 16u;
#pragma unroll
                for (int u = 0; u < 8; ++u)
                    if (u < un) {
                        uint32_t raw[16];
                        tmem_ld16(acc + u * 16u, raw);
                        tmem_wait_ld();
#pragma unroll
                        for (int e = 0; e < 16; ++e) sum[u][e] = kb ? sum[u][e] + __uint_as_float(raw[e]) : __uint_as_float(raw[e]);
                    }
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(acc_empty + (i & 1));     // the next products may overwrite the accumulator
            }
            float ss = 0.f;
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                const int n0 = (u0 + ub + u) * 16;
                if (u < un && live && n0 < a.N) {
                    float4 xr[4];
                    if (EPI == E_RES) {
                        const float4 *px = reinterpret_cast<const float4 *>(a.x + (size_t)r * a.N + n0);
#pragma unroll
                        for (int e = 0; e < 4; ++e) xr[e] = px[e];
                    }
                    tile_epilogue<EPI>(a, r, seq, pos, n0, inv, sum[u], xr, ss);
                }
            }
            if (EPI == E_RES) a.ssq_out[(size_t)(nti * 2 + half) * a.rpad + r] = live ? ss : 0.f;
            if (!ok) break;
        }
    }
    __syncwarp();
    tc_fence_before();
    __syncthreads();
    if (warp == 9) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512) : "memory");
}

// ------------------------------------------------------------------ attention

#include "pf_attention.cuh"

__global__ void k_pf_lengths(SeqState *st, int batch, int n, int target, int draft, int mb) {
    const int s = threadIdx.x;
    if (s >= batch) return;
    if (target) st[s].len_T = n;
    if (draft) st[s].len_D = n;
    if (mb) st[s].len_B = n;
}

// ------------------------------------------------------------------ host

Sizes sizes(int d_max, int hh_max, int f_max, int rows) {
    const size_t R = (size_t)((rows + TM - 1) / TM) * TM;
    Sizes s;
    s.x = R * d_max * sizeof(float);
    s.xg = R * d_max * 2 * sizeof(bf16);
    s.att = R * hh_max * 2 * sizeof(bf16);
    s.act = std::max(R * f_max * 2 * sizeof(bf16), R * hh_max * sizeof(float));
    s.ssq = R * sizeof(float) * 2 * ((size_t)d_max / 16 + 1);
    return s;
}

// 16-row weight tiles of a GEMM tile: the width with the least waves x time of a tile.  A stage takes the longer of its
// tensor time (0.49 us at full width) and its copies (32 KB of token rows, 2 KB per weight tile, at about 95 GB/s per SM).
static int tile_width(int mt, int na, int MT, int n_sm) {
    int best = 16;
    double best_cost = 1e30;
    for (int w = 16; w >= 2; --w) {
        const int nt = (MT + w - 1) / w, waves = (mt * nt + n_sm - 1) / n_sm;
        const double tensor = 0.49 * std::max(w, 8) / 16, copy = ((mt > 1 ? 32 : 2 * na) + 2 * w) / 95.0;
        const double cost = waves * std::max(tensor, copy);
        if (cost < best_cost * 0.99) { best_cost = cost; best = w; }
    }
    return best;
}

template <int EPI>
static cudaError_t launch_gemm(GArgs &a, int n_sm, cudaStream_t st) {
    static bool attr_set[64] = {};           // the opt-in is per device
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= 64 || !attr_set[dev]) {
        e = cudaFuncSetAttribute(k_pf_gemm<EPI>, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM_G);
        if (e != cudaSuccess) return e;
        if (dev >= 0 && dev < 64) attr_set[dev] = true;
    }
    a.mt = (a.rows + TM - 1) / TM; a.rpad = a.mt * TM;
    a.w = tile_width(a.mt, (a.rows + 7) / 8, a.MT, n_sm);
    a.nt = (a.MT + a.w - 1) / a.w;
    k_pf_gemm<EPI><<<std::min(n_sm, a.mt * a.nt), THREADS_G, SMEM_G, st>>>(a);
    return cudaGetLastError();
}

#define PF(call)                                     \
    do {                                             \
        cudaError_t e_ = (call);                     \
        if (e_ != cudaSuccess) return e_;            \
        ++*launches;                                 \
    } while (0)

cudaError_t run(const ModelDev &m, const DevPtrs &d, const Bufs &b, int32_t *abort_flag, int batch, int nj, int c0, Input input,
                const bf16 *normf, bool need_x, int n_sm, cudaStream_t st, int64_t *launches) {
    const pacer_model_cfg &k = m.cfg;
    const int rows = batch * nj, dm = k.d_model, hh = k.n_heads * m.hd, F = k.d_ffn, L = k.n_layers;
    InArgs in{d.x, m.embed, m.norm1, normf, b.x, b.xg, b.ssq, d.max_ctx, dm, nj, c0, rows, (int32_t)input, k.rms_eps};
    k_pf_input<<<rows, 256, 0, st>>>(in);
    PF(cudaGetLastError());
    CUtensorMap mk, mv;
    cudaError_t e = attn_map(&mk, m, m.kcache, d.max_batch, d.max_ctx);
    if (e == cudaSuccess) e = attn_map(&mv, m, m.vcache, d.max_batch, d.max_ctx);
    if (e != cudaSuccess) return e;
    int nss = 1;
    for (int l = 0; l < L; ++l) {
        const size_t kv = (size_t)l * d.max_batch * k.n_kv_heads * (size_t)d.max_ctx * m.hd;
        GArgs g{};
        g.rows = rows; g.eps = k.rms_eps; g.abort_flag = abort_flag; g.nj = nj; g.c0 = c0;
        auto op = [&](OpKind i, const bf16 *A, int N, int K, int MT) {
            g.A = A; g.K = K; g.N = N; g.MT = MT;
            g.W = m.wt[i] + (size_t)l * (K / KB) * (2 * MT) * 512;
        };
        op(OP_QKV, b.xg, m.qrows, dm, (m.qrows + 15) / 16);
        g.ssq_in = b.ssq; g.nss = nss;
        g.q = b.q; g.kc = m.kcache + kv; g.vc = m.vcache + kv; g.kv_lo = m.kv_lo; g.rope = m.rope;
        g.H = k.n_heads; g.Hkv = k.n_kv_heads; g.hd = m.hd; g.max_ctx = d.max_ctx;
        PF(launch_gemm<E_QKV>(g, n_sm, st));
        if (l == L - 1 && !need_x) break;                // nothing reads the rest of the last layer
        const AArgs at{b.q, b.att, k.n_heads, k.n_kv_heads, nj, c0, rows, l * d.max_batch * k.n_kv_heads, abort_flag};
        PF(m.hd == 64 ? launch_attn<64>(mk, mv, at, batch, st) : launch_attn<128>(mk, mv, at, batch, st));
        op(OP_O, b.att, dm, hh, (dm + 15) / 16);
        g.x = b.x; g.ssq_out = b.ssq; g.gain = m.norm2 + (size_t)l * dm; g.out = b.xg; g.out_k = dm;
        PF(launch_gemm<E_RES>(g, n_sm, st));
        g.nss = 2 * g.nt;
        op(OP_GU, b.xg, 2 * F, dm, (F + 7) / 8);
        g.out = b.act; g.out_k = F;
        PF(launch_gemm<E_GU>(g, n_sm, st));
        op(OP_DOWN, b.act, dm, F, (dm + 15) / 16);
        g.gain = l + 1 < L ? m.norm1 + (size_t)(l + 1) * dm : m.normf; g.out = b.xg; g.out_k = dm;
        PF(launch_gemm<E_RES>(g, n_sm, st));
        nss = 2 * g.nt;
    }
    return cudaSuccess;
}

cudaError_t set_lengths(const DevPtrs &d, int batch, int n, bool target, bool draft, bool mb, cudaStream_t st) {
    k_pf_lengths<<<1, 64, 0, st>>>(d.st, batch, n, target, draft, mb);
    return cudaGetLastError();
}

}  // namespace pf
