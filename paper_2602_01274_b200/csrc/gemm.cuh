// Skinny weight-streaming product: Y[r][n] = sum_k X[r][k] * W[n][k], rows <= 32, bf16 in, fp32 sums, ONE launch.
//
// Bound by reading W once from HBM.  Every lane reads its share of W with 128-bit loads straight into registers
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

constexpr int LIN_THREADS = 256, LIN_SMS = 148;

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

struct LinPlan {
    int S, groups, NW, TT;
};

// The split with the least weight bytes per block: S = 1 or 2 slices over all SMs (every pair of SMs can hold a
// cluster of two); 4 or 8 only while few clusters are needed (an odd number of SMs per GPC strands some otherwise).  A
// block keeps at least eight chunks of k, and the smaller S wins ties: 17 x 4096 x 11008 runs as 74 clusters of two,
// 7 tiles each (full 98.9 %), where one slice would leave 4 tiles on some SMs against a mean of 3.46.  More than eight tiles a
// block without slices: slices could even out 5 % at most, and the sums of twice the tiles through the cluster cost 1 to 7 us
// (32 x 12210 x 512 16.2 us with two slices, 9.5 without; 32 x 11008 x 4096 33.3, 26.9).
static inline LinPlan lin_plan(int N, int K) {
    const int MT = (N + 7) / 8, nch = K / 32;
    LinPlan best{};
    double best_cost = 1e30;
    const int cap[4] = {LIN_SMS, LIN_SMS / 2, 32, 16};
    for (int i = 0; i < 4; ++i) {
        const int S = 1 << i;
        if (S > 1 && (nch / S < 8 || best.NW > 1)) break;           // (NW > 1: more than eight tiles a block without slices)
        const int waves = (MT + cap[i] * 64 - 1) / (cap[i] * 64);   // at most 64 tiles per block
        if (S > 1 && waves > 1) break;
        const int groups = MT < cap[i] * waves ? MT : cap[i] * waves, tiles = (MT + groups - 1) / groups;
        const double cost = (double)waves * tiles / S;
        if (cost < best_cost * 0.97) {
            best_cost = cost;
            best.S = S; best.groups = groups;
            best.NW = 1;
            while ((tiles + best.NW - 1) / best.NW > 8) best.NW *= 2;
            best.TT = (tiles + best.NW - 1) / best.NW;
        }
    }
    return best;
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

static inline cudaError_t lin_run(const bf16 *x, const bf16 *w, float *y, int rows, int N, int K, cudaStream_t st) {
    const LinPlan p = lin_plan(N, K);
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
