// Causal attention of a prompt chunk: 128 query rows of one head per block over the keys 0 .. c0 + j, from the cache (the
// chunk's own keys are there already), in tiles of 128 keys, FlashAttention style on tcgen05.  Part of prefill.cu.
//
// Queries, probabilities, keys and values are split bf16 (value + remainder); a product of two split operands is three MMA
// passes (remainder x value, value x remainder, value x value: small terms first, the tensor cores truncate when they add;
// products of two remainders, 2^-18, are left out), so a 128 x 128 tile at head dimension 128 is 48 MMAs = 3072 cycles, and
// the exponentials and splits of a tile run under the MMAs of its neighbours:
//   warps 0..3, 4..7   softmax of the even and of the odd key tiles, a thread per query row, the scores in registers.  The
//                      probabilities (relative to the maximum of the TILE, so that the two warpgroups do not depend on one
//                      another) go back over the scores' columns, values and remainders of 16 keys side by side, and are
//                      read from there as the A operand;
//   warps 8..11        the output rows in registers: sum <- sum * f + tile * f', in ordinary fp32;
//   warp 12            tiles by TMA in the 128-byte swizzle: keys are a K-major operand, values an MN-major one;
//   warp 13            issues the MMAs: scores of tile i + 1 before the values of tile i, so the tensor cores run while
//                      the softmax of tile i does.
// One tile's planes of K, then of V, pass through a ring of NSLOT slots; scores and tile sums have two buffers each.
// 56 heads (8 of keys), 2047 rows, launches in a row: 653 us on mma.sync with 64-row blocks, 264 here (0.67 PFLOP/s, the three passes
// counted); between the projections of a layer of width 7168, under the power cap, 780 and 330.  A block takes 10 us and 3.7 us a
// tile (148 heads of 256 to 2048 rows, the same work on every SM, within 10 %).  The tile: the chain softmax - values - next scores of
// a warpgroup; its MMAs are 1.6 us at 1965 MHz.  The 10 us overlap nothing, one block being all that an SM holds: barriers and tensor
// memory, the conversion of the queries, the first keys, the last sums and the stores.  Up to some 200 rows they outweigh the rest
// (128 rows, 56 heads: 12.8 us on mma.sync, 14.4 here; head dimension 64 8.5, 12.0).  The softmax warps hold 128 scores in 152
// registers (104 bytes spilled at head dimension 128, 28 at 64).
// Error against fp64: 0.96 to 1.006 of what mma.sync with 32 keys a tile had, 33 to 2047 rows, flat, ordinary and peaked softmax,
// values with and without a mean (ordinary: 4.9e-6).
constexpr int AQ = 128, AK = 128;          // query rows of a block, keys of a tile
constexpr int A_SM_WARPS = 8, A_TMA = 12, A_MMA = 13, A_THREADS = 512;
// Registers a thread of a softmax, the output and the last warpgroup: 128 at launch, 2 * 152 + 168 + 40 = 4 * 128.
template <int HD>
struct AttnCfg {
    static constexpr int NP = HD / 64, PANEL = AK * 128, SLOT = NP * PANEL;      // 64-column panels; bytes of one, of a tile's plane
    static constexpr int NSLOT = HD == 128 ? 5 : 8;
    static constexpr int Q_BYTES = 2 * NP * AQ * 128, BAR_OFF = Q_BYTES + NSLOT * SLOT, STAT_OFF = BAR_OFF + 256;
    static constexpr int SMEM = STAT_OFF + 2 * AQ * 8 + 16;
    static_assert(SMEM <= 227 * 1024 && SMEM > 114 * 1024, "one block per SM: it takes all of the tensor memory");
};

struct AArgs {
    const float *q;
    bf16 *out;
    int32_t H, Hkv, nj, c0, rows;
    int32_t head0;                         // (layer, sequence 0, kv head 0) in the caches' third dimension
    int32_t *abort_flag;
};

__device__ __forceinline__ void tma_tile(void *dst, const CUtensorMap *m, int x, int key, int head, int plane, uint64_t *bar) {
    asm volatile("cp.async.bulk.tensor.4d.shared::cta.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5}], [%6];"
                 ::"r"(smem_u32(dst)), "l"(m), "r"(x), "r"(key), "r"(head), "r"(plane), "r"(smem_u32(bar)) : "memory");
}
// An MN-major operand in the 128-byte swizzle: rows (k) of 64 channels, eight of them 1 KB, the next 64 channels a panel further.
__device__ __forceinline__ uint64_t umma_desc_mn(uint32_t saddr, uint32_t panel) {
    return (uint64_t)((saddr >> 4) & 0x3FFF) | ((uint64_t)(panel >> 4) << 16) | (64ull << 32) | (1ull << 46) | (2ull << 61);
}
// (A operand in tensor memory)
__device__ __forceinline__ void umma_ts_if(uint32_t on, uint32_t d_tmem, uint32_t a_tmem, uint64_t b, uint32_t idesc, uint32_t accumulate) {
    asm volatile("{\n\t.reg .pred p, q;\n\tsetp.ne.b32 p, %4, 0;\n\tsetp.ne.b32 q, %6, 0;\n\t"
                 "@q tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, {%5, %5, %5, %5}, p;\n\t}\n"
                 ::"r"(d_tmem), "r"(a_tmem), "l"(b), "r"(idesc), "r"(accumulate), "r"(0u), "r"(on) : "memory");
}
__device__ __forceinline__ void tmem_st16(uint32_t taddr, const uint32_t (&v)[16]) {
    asm volatile("tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};"
                 ::"r"(taddr), "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7]), "r"(v[8]), "r"(v[9]),
                   "r"(v[10]), "r"(v[11]), "r"(v[12]), "r"(v[13]), "r"(v[14]), "r"(v[15]) : "memory");
}
// (the loaded registers pass through the wait, so that nothing that uses them can move in front of it)
__device__ __forceinline__ void tmem_wait16(uint32_t *v) {
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+r"(v[0]), "+r"(v[1]), "+r"(v[2]), "+r"(v[3]), "+r"(v[4]), "+r"(v[5]), "+r"(v[6]), "+r"(v[7]), "+r"(v[8]), "+r"(v[9]),
                   "+r"(v[10]), "+r"(v[11]), "+r"(v[12]), "+r"(v[13]), "+r"(v[14]), "+r"(v[15]) :: "memory");
}
__device__ __forceinline__ void tmem_ld32_async(uint32_t taddr, uint32_t *v) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
                 : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]), "=r"(v[8]), "=r"(v[9]),
                   "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15]), "=r"(v[16]), "=r"(v[17]), "=r"(v[18]),
                   "=r"(v[19]), "=r"(v[20]), "=r"(v[21]), "=r"(v[22]), "=r"(v[23]), "=r"(v[24]), "=r"(v[25]), "=r"(v[26]), "=r"(v[27]),
                   "=r"(v[28]), "=r"(v[29]), "=r"(v[30]), "=r"(v[31]) : "r"(taddr));
}
__device__ __forceinline__ float ex2(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

template <int HD>
__global__ void __launch_bounds__(A_THREADS, 1) k_pf_attn(const __grid_constant__ CUtensorMap mk, const __grid_constant__ CUtensorMap mv,
                                                          const __grid_constant__ AArgs a) {
    using C = AttnCfg<HD>;
    constexpr int NP = C::NP, K16 = HD / 16;
    constexpr uint32_t ACC_O = 256;                      // tensor-memory columns: two tiles of scores, then two of sums
    constexpr float L2E = 1.4426950408889634f;
    extern __shared__ __align__(1024) unsigned char smem[];
    const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
    if (smem_u32(smem) & 1023u) {                        // (the same in every block)
        if (threadIdx.x == 0) atomicCAS(a.abort_flag, 0, 13);
        return;
    }
    uint64_t *full = reinterpret_cast<uint64_t *>(smem + C::BAR_OFF), *empty = full + C::NSLOT, *s_full = empty + C::NSLOT;
    uint64_t *p_full = s_full + 2, *o_full = p_full + 2, *o_empty = o_full + 2, *q_full = o_empty + 2;
    static_assert((2 * C::NSLOT + 9) * 8 <= 256, "barriers");
    float2 *stat = reinterpret_cast<float2 *>(smem + C::STAT_OFF);                // [2][AQ] (maximum * log2 e, sum) of a tile's row
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(stat + 2 * AQ);
    unsigned char *ring = smem + C::Q_BYTES;
    FwdBufs fb;
    fb.abort_flag = a.abort_flag;
    if (threadIdx.x == 0) {
        for (int i = 0; i < C::NSLOT; ++i) { mbar_init(full + i, 1); mbar_init(empty + i, 1); }
        for (int i = 0; i < 2; ++i) { mbar_init(s_full + i, 1); mbar_init(p_full + i, 4); mbar_init(o_full + i, 1); mbar_init(o_empty + i, 4); }
        mbar_init(q_full, 12);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        fence_proxy_async();
    }
    if (warp == A_TMA && lane == 0) {
        asm volatile("prefetch.tensormap [%0];" ::"l"(&mk) : "memory");
        asm volatile("prefetch.tensormap [%0];" ::"l"(&mv) : "memory");
    }
    if (warp == A_MMA) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)), "r"(512) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;
    const int qt = gridDim.z - 1 - blockIdx.z, h = blockIdx.x, seq = blockIdx.y, kh = h / (a.H / a.Hkv);   // longest rows first
    const int j0 = qt * AQ, n_keys = a.c0 + min(j0 + AQ, a.nj), n_tiles = (n_keys + AK - 1) / AK;

    if (warp < 12) {
        // the query rows as the A operand, values and remainders (rows past the end: zeros)
        for (int i = threadIdx.x; i < AQ * (HD / 8); i += 384) {
            const int r = i / (HD / 8), ch = i - r * (HD / 8), j = j0 + r;
            uint4 hi = make_uint4(0u, 0u, 0u, 0u), lo = hi;
            if (j < a.nj) {
                const float4 *p = reinterpret_cast<const float4 *>(a.q + (size_t)(seq * a.nj + j) * (a.H * HD) + h * HD) + ch * 2;
                const float4 u = p[0], w = p[1];
                split2(u.x, u.y, hi.x, lo.x); split2(u.z, u.w, hi.y, lo.y); split2(w.x, w.y, hi.z, lo.z); split2(w.z, w.w, hi.w, lo.w);
            }
            unsigned char *dst = smem + (ch >> 3) * (AQ * 128) + r * 128 + (((ch & 7) ^ (r & 7)) << 4);
            *reinterpret_cast<uint4 *>(dst) = hi;
            *reinterpret_cast<uint4 *>(dst + NP * AQ * 128) = lo;
        }
        fence_proxy_async();
        __syncwarp();
        if (lane == 0) mbar_arrive(q_full);
    }

    if (warp < A_SM_WARPS) {
        asm volatile("setmaxnreg.inc.sync.aligned.u32 152;");
        const int b = warp >> 2, row = (warp & 3) * 32 + lane, pos = a.c0 + j0 + row;
        const uint32_t sc = tmem + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)b * AK;
        for (int i = b, n = 0; i < n_tiles; i += 2, ++n) {
            if (!__all_sync(0xffffffffu, wait_bar(fb, s_full + b, (uint32_t)n & 1u, 30, i))) break;
            tc_fence_after();
            const int vis = pos - i * AK;                // columns 0 .. vis are visible to this row
            const bool diag = i * AK + AK - 1 > a.c0 + j0 + (warp & 3) * 32;      // (the same in the whole warp)
            const int k16 = min((n_keys - i * AK + 15) >> 4, AK / 16);            // 16-key steps of this tile
            uint32_t v[AK];
#pragma unroll
            for (int c = 0; c < AK; c += 32) tmem_ld32_async(sc + c, v + c);
#pragma unroll
            for (int c = 0; c < AK; c += 16) tmem_wait16(v + c);
            if (diag)                                    // (it also covers the columns behind the last key)
#pragma unroll
                for (int e = 0; e < AK; ++e) if (e > vis) v[e] = 0xff800000u;             // -inf
            float m0 = -INFINITY, m1 = -INFINITY;
#pragma unroll
            for (int e = 0; e < AK; e += 2) { m0 = fmaxf(m0, __uint_as_float(v[e])); m1 = fmaxf(m1, __uint_as_float(v[e + 1])); }
            const float m = fmaxf(m0, m1), ms = m == -INFINITY ? 0.f : m * L2E;
            float l0 = 0.f, l1 = 0.f;
#pragma unroll
            for (int c = 0; c < AK / 16; ++c) {          // 16 keys: eight columns of values, eight of remainders
                if (c >= k16) continue;
                uint32_t w[16];
#pragma unroll
                for (int e = 0; e < 8; ++e) {
                    const float p0 = ex2(fmaf(__uint_as_float(v[c * 16 + 2 * e]), L2E, -ms)), p1 = ex2(fmaf(__uint_as_float(v[c * 16 + 2 * e + 1]), L2E, -ms));
                    l0 += p0; l1 += p1;
                    split2(p0, p1, w[e], w[8 + e]);
                }
                tmem_st16(sc + c * 16, w);
            }
            asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
            // the statistics of two tiles before have been read
            if (!__all_sync(0xffffffffu, wait_bar(fb, o_empty + b, ((uint32_t)n & 1u) ^ 1u, 31, i))) break;
            stat[b * AQ + row] = make_float2(m == -INFINITY ? -INFINITY : ms, l0 + l1);
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(p_full + b);
        }
    } else if (warp < A_TMA) {
        asm volatile("setmaxnreg.inc.sync.aligned.u32 168;");
        const int row = (warp & 3) * 32 + lane;
        const uint32_t base = tmem + ((uint32_t)((warp & 3) * 32) << 16) + ACC_O;
        float o[HD], M = -INFINITY, L = 0.f;
#pragma unroll
        for (int e = 0; e < HD; ++e) o[e] = 0.f;
        bool ok = true;
        for (int i = 0; i < n_tiles; ++i) {
            const int b = i & 1;
            const uint32_t par = (uint32_t)(i >> 1) & 1u;
            ok = wait_bar(fb, p_full + b, par, 32, i) && wait_bar(fb, o_full + b, par, 33, i);
            if (!__all_sync(0xffffffffu, ok)) { ok = false; break; }
            tc_fence_after();
            const float2 st = stat[b * AQ + row];
            const float Mn = fmaxf(M, st.x), f0 = M == -INFINITY ? 0.f : ex2(M - Mn), f1 = st.x == -INFINITY ? 0.f : ex2(st.x - Mn);
            M = Mn;
            L = L * f0 + st.y * f1;
#pragma unroll
            for (int c = 0; c < HD; c += 16) {
                uint32_t v[16];
                tmem_ld16(base + (uint32_t)b * HD + c, v);
                tmem_wait16(v);
#pragma unroll
                for (int e = 0; e < 16; ++e) o[c + e] = o[c + e] * f0 + __uint_as_float(v[e]) * f1;
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(o_empty + b);
        }
        const int j = j0 + row;
        if (ok && j < a.nj) {
            const float inv = 1.f / L;
            const int r = seq * a.nj + j;
#pragma unroll
            for (int c = 0; c < HD; c += 8) {
                float v[8];
#pragma unroll
                for (int e = 0; e < 8; ++e) v[e] = o[c + e] * inv;
                store8(a.out, r, h * HD + c, a.H * HD, a.rows, v);
            }
        }
    } else {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 40;");
        if (warp == A_TMA && lane == 0) {
            const int head = a.head0 + seq * a.Hkv + kh;
            int n = 0;
            bool ok = true;
            auto plane = [&](const CUtensorMap *m, int key, int pl) {
                if (!ok) return;
                const int slot = n % C::NSLOT;
                ok = wait_bar(fb, empty + slot, (((uint32_t)(n / C::NSLOT)) & 1u) ^ 1u, 34, n);
                if (!ok) return;
                mbar_expect_tx(full + slot, C::SLOT);
#pragma unroll
                for (int p = 0; p < NP; ++p) tma_tile(ring + slot * C::SLOT + p * C::PANEL, m, p * 64, key, head, pl, full + slot);
                ++n;
            };
            asm volatile("fence.proxy.async;" ::: "memory");          // the keys were written by ordinary stores of earlier kernels
            for (int i = 0; i <= n_tiles; ++i) {
                if (i < n_tiles) { plane(&mk, i * AK, 0); plane(&mk, i * AK, 1); }
                if (i > 0) { plane(&mv, (i - 1) * AK, 0); plane(&mv, (i - 1) * AK, 1); }
            }
            for (int j = max(0, n - C::NSLOT); j < n; ++j)            // no copy may be in flight when the block ends
                for (unsigned it = 0; it < MBAR_SPIN_LIMIT && !mbar_try_wait(full + j % C::NSLOT, ((uint32_t)(j / C::NSLOT)) & 1u); ++it) {}
        } else if (warp == A_MMA) {
            const uint32_t id_o = umma_idesc(HD) | (1u << 16), q_hi = smem_u32(smem), q_lo = q_hi + NP * AQ * 128, on = elect_lane();
            int n = 0;
            bool ok = wait_bar(fb, q_full, 0, 35, 0);
            // (all lanes wait, one issues)
            auto slot_ready = [&](int k) {
                if (ok) ok = wait_bar(fb, full + k % C::NSLOT, ((uint32_t)(k / C::NSLOT)) & 1u, 36, k);
                return smem_u32(ring + (k % C::NSLOT) * C::SLOT);
            };
            for (int i = 0; i <= n_tiles; ++i) {
                if (i < n_tiles) {                       // scores of tile i (its buffer's probabilities were read by the MMAs before)
                    const uint32_t k_hi = slot_ready(n), k_lo = slot_ready(n + 1), acc = tmem + (uint32_t)(i & 1) * AK;
                    ok = __all_sync(0xffffffffu, ok);
                    if (!ok) break;
                    tc_fence_after();
                    const uint32_t id_s = umma_idesc(16 * min((n_keys - i * AK + 15) >> 4, AK / 16));
#pragma unroll
                    for (int t = 0; t < 3; ++t)
#pragma unroll
                        for (int k = 0; k < K16; ++k) {
                            const uint32_t at = (uint32_t)(k >> 2) * (AQ * 128) + (uint32_t)(k & 3) * 32;
                            umma_if(on, acc, umma_desc((t == 0 ? q_lo : q_hi) + at), umma_desc((t == 1 ? k_lo : k_hi) + at), id_s, t > 0 || k > 0 ? 1u : 0u);
                        }
                    umma_commit_if(on, s_full + (i & 1));
                    umma_commit_if(on, empty + n % C::NSLOT); umma_commit_if(on, empty + (n + 1) % C::NSLOT);
                    n += 2;
                }
                if (i > 0) {                             // values of tile i - 1
                    const int t0 = i - 1, b = t0 & 1;
                    const uint32_t par = (uint32_t)(t0 >> 1) & 1u, v_hi = slot_ready(n), v_lo = slot_ready(n + 1);
                    if (ok) ok = wait_bar(fb, p_full + b, par, 37, t0) && wait_bar(fb, o_empty + b, par ^ 1u, 38, t0);
                    ok = __all_sync(0xffffffffu, ok);
                    if (!ok) break;
                    const int live = n_keys - t0 * AK;   // what lies behind the last key is not read, not even times zero
                    if (live < AK) {                     // (up to the end of its 16-key step)
                        for (int e = lane; e < (-live & 15) * 8 * NP * 2; e += 32) {
                            const int ch = e & 7, p = (e >> 3) & (2 * NP - 1), key = live + (e >> 3) / (2 * NP), slot = (n + p / NP) % C::NSLOT;
                            *reinterpret_cast<uint4 *>(ring + slot * C::SLOT + (p % NP) * C::PANEL + key * 128 + ch * 16) = make_uint4(0u, 0u, 0u, 0u);
                        }
                        fence_proxy_async();
                        __syncwarp();
                    }
                    tc_fence_after();
                    const uint32_t acc = tmem + ACC_O + (uint32_t)b * HD, pr = tmem + (uint32_t)b * AK;
#pragma unroll
                    for (int t = 0; t < 3; ++t)
#pragma unroll
                        for (int k = 0; k < AK / 16; ++k)
                            if (k * 16 < live) umma_ts_if(on, acc, pr + (uint32_t)k * 16 + (t == 0 ? 8 : 0), umma_desc_mn((t == 1 ? v_lo : v_hi) + (uint32_t)k * 2048, C::PANEL), id_o, t > 0 || k > 0 ? 1u : 0u);
                    umma_commit_if(on, o_full + b);
                    umma_commit_if(on, empty + n % C::NSLOT); umma_commit_if(on, empty + (n + 1) % C::NSLOT);
                    n += 2;
                }
            }
        }
    }
    __syncwarp();
    tc_fence_before();
    __syncthreads();
    if (warp == A_MMA) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512) : "memory");
}

// A cache as [plane][layer, sequence, kv head][position][channel]; a box is 64 channels of AK positions.
static cudaError_t attn_map(CUtensorMap *map, const ModelDev &m, const bf16 *cache, int max_batch, int max_ctx) {
    typedef CUresult (*Encode)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *, const cuuint64_t *, const cuuint32_t *,
                               const cuuint32_t *, CUtensorMapInterleave, CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
    static const Encode encode = [] {
        void *p = nullptr;
        cudaDriverEntryPointQueryResult res;
        const cudaError_t e = cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &res);
        return e == cudaSuccess && res == cudaDriverEntryPointSuccess ? (Encode)p : nullptr;
    }();
    if (!encode) return cudaErrorNotSupported;
    const cuuint64_t hd = m.hd, heads = (cuuint64_t)m.cfg.n_layers * max_batch * m.cfg.n_kv_heads;
    const cuuint64_t dim[4] = {hd, (cuuint64_t)max_ctx, heads, 2}, stride[3] = {hd * 2, hd * 2 * max_ctx, m.kv_lo * 2};
    const cuuint32_t box[4] = {64, AK, 1, 1}, step[4] = {1, 1, 1, 1};
    const CUresult r = encode(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<bf16 *>(cache), dim, stride, box, step, CU_TENSOR_MAP_INTERLEAVE_NONE,
                              CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidValue;
}

template <int HD>
static cudaError_t launch_attn(const CUtensorMap &mk, const CUtensorMap &mv, const AArgs &a, int batch, cudaStream_t st) {
    static bool attr_set[64] = {};           // the opt-in is per device
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= 64 || !attr_set[dev]) {
        e = cudaFuncSetAttribute(k_pf_attn<HD>, cudaFuncAttributeMaxDynamicSharedMemorySize, AttnCfg<HD>::SMEM);
        if (e != cudaSuccess) return e;
        if (dev >= 0 && dev < 64) attr_set[dev] = true;
    }
    k_pf_attn<HD><<<dim3(a.H, batch, (a.nj + AQ - 1) / AQ), A_THREADS, AttnCfg<HD>::SMEM, st>>>(mk, mv, a);
    return cudaGetLastError();
}
