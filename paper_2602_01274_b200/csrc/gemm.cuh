// Skinny weight-streaming product: Y[r][n] = sum_k X[r][k] * W[n][k], rows <= 32, bf16 in, fp32 sums, ONE launch.  Two
// kernels: k_linear_wide where every SM has its share of whole weight rows, k_linear else (the rule: lin_plan.h).
//
// k_linear.  Bound by reading W once from HBM.  Every lane reads its share of W with 128-bit loads straight into registers
// (each weight is used exactly once, so staging it in shared memory would only add traffic), 8 to 32 loads in flight
// per lane.  The activations come out of L2 through shared memory, eight chunks ahead: a lane copies exactly the 16-byte
// pieces that it reads, so nothing is synchronised.  mma.m16n8k16 with
// the token rows as the 16-row operand and eight weight rows as the other: a lane (g = lane / 4, t = lane % 4) loads the
// 8 consecutive k of its row at 32c + 8t and uses them as the k slots {2t, 2t+1, 2t+8, 2t+9} of two MMAs; both operands
// follow the rule, so the products pair up and the sum over k is the same.
//
// Split: a block owns up to 64 tiles of eight weight rows; its eight warps are NW tile groups x KW shares of k (summed
// through shared memory).  When the tiles do not fill the 148 SMs evenly, S blocks of a cluster share a tile range and
// take one k slice each; their sums meet through distributed shared memory, in rank order.  No partial sum goes to
// global memory.
#pragma once
#include "common.cuh"
#include "lin_plan.h"

__device__ __forceinline__ uint4 ldg_stream(const void *p) {
    uint4 v;
    asm volatile("ld.global.nc.L1::no_allocate.v4.u32 {%0,%1,%2,%3}, [%4];"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p));
    return v;
}

__device__ __forceinline__ void mma_bf16_16816(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3,
                                               uint32_t b0, uint32_t b1) {
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
                 : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
                 : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

struct LinArgs {
    const bf16 *x, *w;
    float *y;
    int32_t rows, N, K;
    int32_t S;               // blocks of a cluster: k slices
    int32_t groups;          // clusters: tile ranges
    int32_t NW;              // tile groups of a block (8 / NW warps share a group's k)
    int32_t x_aligned;       // x is 16-byte aligned (a view into a larger tensor need not be)
};

constexpr int LIN_THREADS = 256;

// Weight loads in flight per lane: D chunks of TT tiles (about 100 KB per SM where registers allow); activations: LIN_XD
// chunks.  (With the activations in registers, two chunks ahead, 17 x 4096 x 11008 took 30 us: every chunk waited for L2.)
__host__ __device__ constexpr int lin_depth(int TT) { return TT >= 7 ? 4 : TT == 6 ? 5 : TT >= 4 ? 6 : 8; }
constexpr int LIN_XD = 8;

__device__ __forceinline__ uint32_t lin_peer(uint32_t smem_addr, int rank) {
    uint32_t r;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(smem_addr), "r"(rank));
    return r;
}

template <int RM, int TT>
__global__ void __launch_bounds__(LIN_THREADS, 1) k_linear(const LinArgs a) {
    constexpr int D = lin_depth(TT), R = RM * 16;
    extern __shared__ __align__(1024) unsigned char smem[];
    float *lin_red = reinterpret_cast<float *>(smem);              // [8 warps][R rows][TT * 8 columns], after the products
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
    const int slice = blockIdx.x % a.S, grp = blockIdx.x / a.S;
    const int KW = 8 / a.NW, nw = warp / KW, kw = warp % KW;
    const int MT = (a.N + 7) >> 3;
    // this block's tiles, as even as they come; this warp's among them
    const int tb = MT / a.groups, tr = MT % a.groups, t0 = grp * tb + min(grp, tr), T = tb + (grp < tr ? 1 : 0);
    const int w0 = T * nw / a.NW, w1 = T * (nw + 1) / a.NW;
    const int nch = a.K >> 5, c_lo = nch * slice / a.S, c_hi = nch * (slice + 1) / a.S;   // 32-column chunks
    const int mine = max(0, (c_hi - c_lo - kw + KW - 1) / KW);
    const bf16 *wp[TT];
#pragma unroll
    for (int i = 0; i < TT; ++i)                                    // tiles past the end repeat a valid row
        wp[i] = a.w + (size_t)min((t0 + min(w0 + i, max(w1 - 1, 0))) * 8 + g, a.N - 1) * a.K + (size_t)(c_lo + kw) * 32 + 8 * t;
    const bf16 *xp = a.x + (size_t)min(g, a.rows - 1) * a.K + (size_t)(c_lo + kw) * 32 + 8 * t;
    const size_t step = (size_t)KW * 32;
    uint4 w[D][TT];
    unsigned char *xs = smem + warp * (LIN_XD * R * 64) + lane * 16;   // [chunk][8-row half][lane] x 16 bytes
    float acc[TT][RM][4];
#pragma unroll
    for (int i = 0; i < TT; ++i)
#pragma unroll
        for (int m = 0; m < RM; ++m) acc[i][m][0] = acc[i][m][1] = acc[i][m][2] = acc[i][m][3] = 0.f;
    auto load_w = [&](int slot, int c) {
#pragma unroll
        for (int i = 0; i < TT; ++i) w[slot][i] = ldg_stream(wp[i] + (size_t)c * step);
    };
    auto load_x = [&](int c) {                                      // a group per chunk, also when there is nothing to copy
        if (c < mine) {
#pragma unroll
            for (int i = 0; i < 2 * RM; ++i) {
                const bool in = i * 8 + g < a.rows;
                const bf16 *p = xp + (in ? (size_t)(i * 8) * a.K : 0) + (size_t)c * step;    // (an idle row reads nothing)
                unsigned char *dst = xs + ((c % LIN_XD) * 2 * RM + i) * 512;
                if (a.x_aligned)
                    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(p), "r"(in ? 16 : 0) : "memory");
                else {
                    const unsigned short *q = reinterpret_cast<const unsigned short *>(p);
                    *reinterpret_cast<uint4 *>(dst) = in ? make_uint4(q[0] | (uint32_t)q[1] << 16, q[2] | (uint32_t)q[3] << 16, q[4] | (uint32_t)q[5] << 16, q[6] | (uint32_t)q[7] << 16)
                                                         : make_uint4(0u, 0u, 0u, 0u);
                }
            }
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
#pragma unroll
    for (int j = 0; j < D; ++j)
        if (j < mine) load_w(j, j);
#pragma unroll
    for (int j = 0; j < LIN_XD - 1; ++j) load_x(j);
    for (int c0 = 0; c0 < mine; c0 += D) {
#pragma unroll
        for (int j = 0; j < D; ++j) {
            const int c = c0 + j;
            if (c >= mine) break;
            load_x(c + LIN_XD - 1);
            asm volatile("cp.async.wait_group %0;" ::"n"(LIN_XD - 1) : "memory");
            uint4 xv[RM][2];
#pragma unroll
            for (int i = 0; i < 2 * RM; ++i) xv[i >> 1][i & 1] = *reinterpret_cast<const uint4 *>(xs + ((c % LIN_XD) * 2 * RM + i) * 512);
#pragma unroll
            for (int i = 0; i < TT; ++i) {
                const uint4 b = w[j][i];
#pragma unroll
                for (int m = 0; m < RM; ++m) {
                    const uint4 p = xv[m][0], q = xv[m][1];
                    mma_bf16_16816(acc[i][m], p.x, q.x, p.y, q.y, b.x, b.y);
                    mma_bf16_16816(acc[i][m], p.z, q.z, p.w, q.w, b.z, b.w);
                }
            }
            if (c + D < mine) load_w(j, c + D);
        }
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    __syncthreads();                                                // the activations' bytes become the sums'
    // accumulator (g, 2t..): token row m*16 + g (+8), weight row 8i + 2t (+1)
    constexpr int P = TT * 8;
    float *my = lin_red + (size_t)warp * R * P;
#pragma unroll
    for (int i = 0; i < TT; ++i)
#pragma unroll
        for (int m = 0; m < RM; ++m)
#pragma unroll
            for (int h = 0; h < 2; ++h)
                *reinterpret_cast<float2 *>(my + (m * 16 + h * 8 + g) * P + i * 8 + 2 * t) = make_float2(acc[i][m][2 * h], acc[i][m][2 * h + 1]);
    __syncthreads();
    // The sums: a tile group's KW warps share its rows, CL lanes a row's columns; the KW shares are added in warp order.  (An
    // element at a time over the whole block, with the divisions that find its group, this took up to 18 us: 32 x 12210 x 512 in
    // all 27.0 us, now 16.2; 32 x 32000 x 256 22.5, now 12.1; 5 x 2304 x 768 4.1, now 4.0.)
    constexpr int CL = TT == 1 ? 8 : TT == 2 ? 16 : 32, RL = 32 / CL, CH = (P + CL - 1) / CL;
    const int qc = (w1 - w0) * 8, n0 = (t0 + w0) * 8, lc = lane & (CL - 1);
    float *sums = lin_red + (size_t)(nw * KW) * R * P + lc;
#pragma unroll 4
    for (int r = kw * RL + lane / CL; r < a.rows; r += KW * RL)
#pragma unroll
        for (int h = 0; h < CH; ++h) {
            const int col = lc + CL * h;
            if (col >= qc) continue;
            float *p = sums + r * P + CL * h;
            float v = p[0];
            for (int k = 1; k < KW; ++k) v += p[(size_t)k * R * P];
            if (a.S > 1) p[0] = v;                                  // the block's sum, for the cluster
            else if (n0 + col < a.N) a.y[(size_t)r * a.N + n0 + col] = v;
        }
    if (a.S > 1) {
        __syncwarp();
        asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
        // the blocks share the rows; all slices' loads in flight
        for (int r = (slice * KW + kw) * RL + lane / CL; r < a.rows; r += a.S * KW * RL) {
            float u[CH][8];
#pragma unroll
            for (int h = 0; h < CH; ++h) {
                const uint32_t at = (uint32_t)__cvta_generic_to_shared(sums + r * P + CL * h);
#pragma unroll
                for (int s = 0; s < 8; ++s)
                    if (s < a.S && lc + CL * h < qc)
                        asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(u[h][s]) : "r"(lin_peer(at, s)) : "memory");
            }
#pragma unroll
            for (int h = 0; h < CH; ++h) {
                const int col = lc + CL * h;
                float v = 0.f;
#pragma unroll
                for (int s = 0; s < 8; ++s)
                    if (s < a.S) v += u[h][s];
                if (col < qc && n0 + col < a.N) a.y[(size_t)r * a.N + n0 + col] = v;
            }
        }
        __syncwarp();
        asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
    }
}

struct LinWideArgs {
    const bf16 *x, *w;
    float *y;
    int32_t rows, N, K;
    int32_t per;             // weight rows of a pass at most (a multiple of 2, at most LW_ROWS)
    int32_t xr;              // token rows of a stage (rows, up to a multiple of 8)
};

__device__ __forceinline__ void lin_ldsm4(uint32_t (&r)[4], uint32_t a) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];" : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(a));
}

// Everything through shared memory.  A block owns a run of weight rows (units of two, as even as they come: 4096 rows on 148 SMs
// are 28 each, tiles of eight rows would be 32) and takes it in passes of up to 32; warp w owns the 64-column chunks w, w + 8, ...
// of k, token and weight rows alike, and copies them for itself, D chunks deep: whole 128-byte lines, nothing but the sums at
// the end of a pass is shared between warps, and the next pass's first chunks travel while a pass is summed up.  Two sets of
// accumulators: the tensor cores truncate, and K / 16 products a set are what k_linear has with two slices (with one set the
// error against fp64 was twice as large, 1.3e-6 at K = 11 008).  17 x 4096 x 11008: 23.2 us with k_linear (its loads of 64
// bytes a row straight into registers), 19.2 here (4.7 TB/s); 17 x 4096 x 4096 13.1, 9.6; 5 x 2304 x 768 3.6, 3.1.
template <int RM, int NA, int D>
__global__ void __launch_bounds__(LIN_THREADS, 1) k_linear_wide(const LinWideArgs a) {
    extern __shared__ __align__(1024) unsigned char smem[];
    constexpr int R = RM * 16, P = NA * 8;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
    const int units = (a.N + 1) >> 1, ub = units / (int)gridDim.x, ur = units - ub * (int)gridDim.x, b = blockIdx.x;
    const int r0 = 2 * (b * ub + min(b, ur)), r1 = min(a.N, r0 + 2 * (ub + (b < ur ? 1 : 0)));
    const int np = (r1 - r0 + a.per - 1) / a.per, chunks = (a.K + 63) >> 6, mine = (chunks - warp + 7) >> 3;
    const int stage_bytes = (a.xr + a.per) * 128;
    unsigned char *ring = smem + warp * D * stage_bytes;
    float *red = reinterpret_cast<float *>(smem + (np > 1 ? 8 * D * stage_bytes : 0));      // [8 warps][R][P]; a single pass is done with the ring
    auto pass_rows = [&](int p, int &lo, int &n) {                              // as even as they come
        const int u = (r1 - r0 + 1) >> 1, q = u / np, m = u - q * np;
        lo = r0 + 2 * (p * q + min(p, m)); n = min(r1 - lo, 2 * (q + (p < m ? 1 : 0)));
    };
    int lp = 0, lc = 0, lslot = 0, llo = 0, ln = 0;                              // what is copied next: pass, chunk, slot
    if (np > 0) pass_rows(0, llo, ln);
    auto load = [&]() {                                                          // a group per chunk, also when there is none left
        if (lp < np && mine > 0) {
            const int col = (warp + 8 * lc) * 64 + (lane & 7) * 8, sz = col < a.K ? 16 : 0;
            unsigned char *st = ring + lslot * stage_bytes;
            const bf16 *src = a.x + (sz ? col : 0);
            for (int r = lane >> 3; r < a.rows; r += 4)
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"((uint32_t)__cvta_generic_to_shared(st + r * 128 + (((lane & 7) ^ (r & 7)) << 4))), "l"(src + (size_t)r * a.K), "r"(sz) : "memory");
            st += a.xr * 128;
            src = a.w + (size_t)llo * a.K + (sz ? col : 0);
#pragma unroll 4
            for (int r = lane >> 3; r < ln; r += 4)
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"((uint32_t)__cvta_generic_to_shared(st + r * 128 + (((lane & 7) ^ (r & 7)) << 4))), "l"(src + (size_t)r * a.K), "r"(sz) : "memory");
            lslot = lslot + 1 == D ? 0 : lslot + 1;
            if (++lc == mine) { lc = 0; if (++lp < np) pass_rows(lp, llo, ln); }
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
#pragma unroll
    for (int i = 0; i < D - 1; ++i) load();
    int slot = 0;
    for (int p = 0; p < np; ++p) {
        int lo, n;
        pass_rows(p, lo, n);
        float acc[2][NA][RM][4];
#pragma unroll
        for (int i = 0; i < NA; ++i)
#pragma unroll
            for (int m = 0; m < RM; ++m)
#pragma unroll
                for (int e = 0; e < 4; ++e) acc[0][i][m][e] = acc[1][i][m][e] = 0.f;
        for (int c = 0; c < mine; ++c) {
            asm volatile("cp.async.wait_group %0;" ::"n"(D - 2) : "memory");
            __syncwarp();                                                        // every lane's copies; and the slot before is read
            load();
            const uint32_t xa = (uint32_t)__cvta_generic_to_shared(ring + slot * stage_bytes), wa = xa + (uint32_t)a.xr * 128u;
            slot = slot + 1 == D ? 0 : slot + 1;
#pragma unroll
            for (int k = 0; k < 4; ++k) {                                        // 16 columns
                uint32_t x[RM][4], w[NA][2];
#pragma unroll
                for (int m = 0; m < RM; ++m)                                     // matrices: rows 0..7, 8..15 of columns 0..7, then of 8..15
                    lin_ldsm4(x[m], xa + (uint32_t)(m * 16 + (lane & 15)) * 128u + (uint32_t)(((2 * k + (lane >> 4)) ^ (lane & 7)) << 4));
#pragma unroll
                for (int i = 0; i < NA; i += 2) {                                // two atoms: columns 0..7, 8..15 of each
                    uint32_t v[4];
                    lin_ldsm4(v, wa + (uint32_t)(i * 8 + (lane & 7) + ((lane >> 4) << 3)) * 128u + (uint32_t)(((2 * k + ((lane >> 3) & 1)) ^ (lane & 7)) << 4));
                    w[i][0] = v[0]; w[i][1] = v[1]; w[i + 1][0] = v[2]; w[i + 1][1] = v[3];
                }
#pragma unroll
                for (int i = 0; i < NA; ++i)
#pragma unroll
                    for (int m = 0; m < RM; ++m) mma_bf16_16816(acc[k & 1][i][m], x[m][0], x[m][1], x[m][2], x[m][3], w[i][0], w[i][1]);
            }
        }
        if (np == 1) __syncthreads();
        float *my = red + (size_t)warp * R * P;
#pragma unroll
        for (int i = 0; i < NA; ++i)
#pragma unroll
            for (int m = 0; m < RM; ++m)
#pragma unroll
                for (int h = 0; h < 2; ++h)
                    *reinterpret_cast<float2 *>(my + (m * 16 + h * 8 + g) * P + i * 8 + 2 * t) = make_float2(acc[0][i][m][2 * h] + acc[1][i][m][2 * h], acc[0][i][m][2 * h + 1] + acc[1][i][m][2 * h + 1]);
        __syncthreads();
        constexpr int RT = LIN_THREADS / P;                                      // rows at a time
        const int col = threadIdx.x & (P - 1);
        if (col < n)
            for (int r = threadIdx.x / P; r < a.rows; r += RT) {
                const float *q = red + r * P + col;
                float v = q[0];
#pragma unroll
                for (int k = 1; k < 8; ++k) v += q[k * R * P];
                a.y[(size_t)r * a.N + lo + col] = v;
            }
        if (p + 1 < np) __syncthreads();
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");
}

template <int RM, int TT>
static cudaError_t lin_launch(const LinArgs &a, cudaStream_t st) {
    constexpr size_t sums = (size_t)8 * RM * 16 * TT * 8 * sizeof(float), ring = (size_t)8 * LIN_XD * RM * 16 * 64;
    constexpr size_t smem = sums > ring ? sums : ring;
    static bool attr_set[64] = {};           // the opt-in is per device
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (smem > 48 * 1024 && (dev < 0 || dev >= 64 || !attr_set[dev])) {
        e = cudaFuncSetAttribute(k_linear<RM, TT>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        if (dev >= 0 && dev < 64) attr_set[dev] = true;
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(a.groups * a.S); cfg.blockDim = dim3(LIN_THREADS); cfg.dynamicSmemBytes = smem; cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = a.S; at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.attrs = at; cfg.numAttrs = a.S > 1 ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, k_linear<RM, TT>, a);
}

template <int RM>
static cudaError_t lin_dispatch(int TT, const LinArgs &a, cudaStream_t st) {
    switch (TT) {
        case 1: return lin_launch<RM, 1>(a, st);
        case 2: return lin_launch<RM, 2>(a, st);
        case 3: return lin_launch<RM, 3>(a, st);
        case 4: return lin_launch<RM, 4>(a, st);
        case 5: return lin_launch<RM, 5>(a, st);
        case 6: return lin_launch<RM, 6>(a, st);
        case 7: return lin_launch<RM, 7>(a, st);
        default: return lin_launch<RM, 8>(a, st);
    }
}

template <int RM, int NA, int D>
static cudaError_t lin_wide_launch(const LinWideArgs &a, int smem, cudaStream_t st) {
    static bool attr_set[64] = {};           // the opt-in is per device
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= 64 || !attr_set[dev]) {
        e = cudaFuncSetAttribute(k_linear_wide<RM, NA, D>, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
        if (e != cudaSuccess) return e;
        if (dev >= 0 && dev < 64) attr_set[dev] = true;
    }
    const int units = (a.N + 1) / 2;
    k_linear_wide<RM, NA, D><<<units < LIN_SMS ? units : LIN_SMS, LIN_THREADS, smem, st>>>(a);
    return cudaGetLastError();
}

template <int RM, int NA>
static cudaError_t lin_wide_depth(const LinWideArgs &a, int np, cudaStream_t st) {
    // room behind the ring: the sums of a pass, or (one pass) what the last atoms read past their rows
    const int stage = 8 * (a.xr + a.per) * 128, sums = 8 * RM * 16 * NA * 8 * 4;
    auto bytes = [&](int d) { return np > 1 ? d * stage + sums : d * stage + 4096 > sums ? d * stage + 4096 : sums; };
    return bytes(4) <= 227 * 1024 ? lin_wide_launch<RM, NA, 4>(a, bytes(4), st) : lin_wide_launch<RM, NA, 3>(a, bytes(3), st);
}

static inline cudaError_t lin_wide_run(const bf16 *x, const bf16 *w, float *y, int rows, int N, int K, cudaStream_t st) {
    LinWideArgs a;
    a.x = x; a.w = w; a.y = y; a.rows = rows; a.N = N; a.K = K; a.xr = (rows + 7) & ~7;
    const LinPasses q = lin_wide_passes(N);
    const int np = q.np;
    a.per = q.per;
    if (rows <= 16) return a.per <= 16 ? lin_wide_depth<1, 2>(a, np, st) : lin_wide_depth<1, 4>(a, np, st);
    return a.per <= 16 ? lin_wide_depth<2, 2>(a, np, st) : lin_wide_depth<2, 4>(a, np, st);
}

static inline cudaError_t lin_run(const bf16 *x, const bf16 *w, float *y, int rows, int N, int K, cudaStream_t st) {
    const LinPlan p = lin_plan(N, K);
    if (((uintptr_t)x & 15) == 0 && lin_wide_takes(rows, N, K, p.S)) return lin_wide_run(x, w, y, rows, N, K, st);
    LinArgs a;
    a.x = x; a.w = w; a.y = y; a.rows = rows; a.N = N; a.K = K; a.S = p.S; a.groups = p.groups; a.NW = p.NW;
    a.x_aligned = ((uintptr_t)x & 15) == 0;
    return rows <= 16 ? lin_dispatch<1>(p.TT, a, st) : lin_dispatch<2>(p.TT, a, st);
}

// Scratch bytes the interface asks callers for (the limit of the allocation-free entry point is stated in them):
// fragment-ordered activations and the partial sums of k slices of at most 1024 or 2048 columns.
static inline size_t lin_scratch_bytes(int rows, int N, int K) {
    const int nt = (rows + 7) / 8, MT = (N + 15) / 16;
    int ks = MT >= 1024 ? 2048 : 1024;
    while ((size_t)nt * 8 * ks * 2 > 96 * 1024) ks /= 2;
    int S = (K + ks - 1) / ks;
    const int KS = (((K + S - 1) / S) + 31) / 32 * 32;
    S = (K + KS - 1) / KS;
    return ((size_t)nt * 8 * K * sizeof(bf16) + 255) / 256 * 256 + (size_t)S * nt * 8 * N * sizeof(float);
}
