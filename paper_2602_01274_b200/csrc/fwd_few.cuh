// The forward of at most 16 live token rows (draft steps, pre-verification calls, autoregressive steps, verify forwards
// of the windows that pre-verification stopped early): one persistent cooperative kernel, one block per SM, like
// k_forward, but with everything laid out for LATENCY.  Such a forward is a chain of phases of a few microseconds; the
// weights of a phase (0.1 to 30 us at the HBM rate) arrive through the ring while the phases before it run.  What differs
// from k_forward:
//   - the live rows are counted on the device and packed: the cost follows the drafts that exist, not the window;
//   - the projections run on mma.sync straight out of the weight ring: with the token rows as the 16-row operand (8
//     rows of bf16 values over their 8 rows of rounding remainders, so ONE m16n8k16 covers 8 split rows) they need 1
//     MMA per 128 weights, 7 % to 20 % of what the SM can issue while HBM delivers them, and no tensor-memory round
//     trip, commit or accumulator copy stands between the last weight and the epilogue;
//   - ten warps share k (five or ten groups) and the block's rows; their sums meet in shared memory.  A stage costs
//     a warp 0.5 us of waits and dependent instructions however little it computes, so the groups work on different ones
//     (all ten warps on every stage, without groups: 37 us for a 7B gate/up projection against 26);
//   - no projection is cut along k across blocks, so the two residual projections need no reduction pass; a block owns
//     the same columns of the residual stream in both and keeps them in shared memory;
//   - weight rows are dealt out in units of two instead of sixteen (a run of rows of a k block is contiguous at any
//     row), so that the largest share is within 1 to 4 % of the mean;
//   - the q/k/v epilogue applies the rotary embedding (the rows of a pair are adjacent in the re-laid weights) and
//     appends k, v to the cache, so attention reads every key from the cache;
//   - the key splits of an attention head are merged by whichever block finishes last, without a grid barrier.
// A launch may run several draft forwards, each on the token that the one before chose (see the end of the kernel): a forward
// in a launch of its own costs about 4 us more in a captured step.
// Five grid barriers per layer instead of nine.  The whole forward is ONE loop over the projections with one inlined
// copy of the projection code: as a function of its own it read the kernel's parameters through L1, which every grid
// barrier empties (a chain of L2 reads at the start of each phase), and several copies thrash the instruction cache.
// Activations read from global memory by the consumer warps themselves cost 1 to 2 us per 64 columns (L2 latency under
// the weight stream, however far ahead); a few large bulk copies hide it.  One thread's decisions cost 100 to 200 cycles
// each (a barrier wait that is already over takes 120), so stages are as large as the rings allow and the producers run
// as whole warps, the ring's bookkeeping in registers.
#pragma once
#include "fwd_few.h"
#include "few_plan.h"

#include "fwd_attention.cuh"
#include "fwd_tails.cuh"

namespace fwd {

constexpr int FW = 10;                          // consumer warps = k groups x weight row groups (with the two producers
constexpr int FC_THREADS = 32 * FW;             // three warps per scheduler: 168 registers a thread)
constexpr int FEW_THREADS = FC_THREADS + 64;
constexpr int FNB = 32;                         // weight stages in flight (barrier pairs; one lane each in the producer)
constexpr int F_STAGE = 28 * 1024;              // bytes of weights a stage aims at: a stage costs the producer about 0.35 us
constexpr int F_XROWS = 52;                     // 256-byte (row, k block) pieces of an activation stage
// Activation stages, and the bytes they share with the sums of a pass and with attention; the weight ring has the rest.  Up to
// eight rows three stages; the target's forwards of more rows five (few_many): a stage is then four or five k blocks, the k groups
// work on 40 of them at a time, and with three stages they wait for each other's (13 rows, 4 layers of width 4096: 490 us with
// three, 471 with five; head dimension 64: width 2048 262, 251, width 256 129, 130).  The smaller weight ring costs more than that
// with five rows (step of 8 layers of width 4096, 12 drafts in front: 738 us with three, 750 with five), and with nine and ten rows
// of wider models (9 rows, 4 layers of width 7168 844 with three, 869 with five; 3 of width 8192 955, 978; 4 of width 4096 450, 449).
constexpr int FXS = 3, FXS_MANY = 5;
__host__ __device__ constexpr int few_scratch(bool many) { return (many ? 71 : 47) * 1024; }
__device__ __forceinline__ bool few_many(int nlive, int d_model) { return nlive > (d_model > 4096 ? 10 : 8); }
constexpr int F_MISC = 10 * 1024;
constexpr int F_GUARD = 1024;                   // before the ring: the rows of an atom ahead of the first one are read, not used
constexpr int F_SHARED = (227 * 1024 - F_MISC - F_GUARD) / 1024 * 1024;      // weight ring and activations
__host__ __device__ constexpr int few_ring(bool many) { return F_SHARED - few_scratch(many); }
static_assert(FNB == 32 && FXS * F_XROWS * 256 <= few_scratch(false) && FXS_MANY * F_XROWS * 256 <= few_scratch(true) &&
              few_ring(true) >= 5 * FEW_LONGER * 1024, "layout");
constexpr int F_XBYTES = FEW_XBYTES;                  // of F_MISC: this block's columns of the residual stream
// Weight rows [r0, r1) of a block in a projection: units of two rows (gate/up: 16, a gate atom and its up atom), as even
// as they come; kept in shared memory for the whole forward.
struct FewOp {
    int r0, r1, atom0, span;       // rows; first 8-row atom and atoms touched
    int nkb, kbs, nst, npass;      // 64-column k blocks, of a weight stage, weight stages; passes over the atoms
    int kgs, pad;                  // k groups: 10 (a warp takes all atoms of a stage) or 5 (two warps share them)
};

struct FewAtt {
    int chunks, nsplit, items;         // query-row chunks of a kv head (FQ rows each), key splits
};
struct FewItem {
    int split, vc, kh, seq, n_r, pos0, lo, hi;
};

struct FewCtx {
    unsigned char *scratch, *ring;
    uint64_t *wfull, *wempty;      // [FNB] a stage's weights are there / have been read
    uint64_t *xfull, *xempty;      // [FXS_MANY] the same for the activations
    volatile int32_t *ready;       // passes begun by the consumers: a later pass of a projection may overwrite the scratch
    int32_t *slot_at;              // [FNB] ring offset of a stage, written by the producer before the stage's barrier
    const FewOp *ops;              // [N_OPS] of this forward; the first forward's are followed by those of the later ones
    float *xs;                     // [live row][columns of this block] residual stream
    float *inv;                    // [FEW_ROWS] per live row
    int32_t *row_of;               // [FEW_ROWS] token row of live row i
    int32_t *idx_of;               // [MAX_ROWS] live row of a token row
    int32_t *row_pos, *row_tok, *n_rows, *key_start, *flag;
    int32_t *pick, *gamma0;        // [FEW_ROWS] per sequence: the token this forward chose; drafts made before this launch
    int nlater;                    // live rows of the second and later forwards of the launch: one per sequence
    int warp, lane, cta, ncta;
    bool ok;                       // false once a wait gave up
    int nlive;
    int stage, xstage;             // weight and activation stages of the passes done so far
    int pass;                      // passes begun (thread 0)
    int xk;                        // k blocks of an activation stage
    bool many;                     // five activation stages, the same for the whole launch
    unsigned long long bar_target;
    // epilogues
    float **row_dst;               // [FEW_ROWS] where an LM-head row goes, or NULL
    int32_t *bias_at;              // [FEW_ROWS] column of the planted bias, or -1
    Top2 *top;                     // [FEW_ROWS] best two logits of this block's columns so far
    int32_t *draw_pos;             // [FEW_ROWS] position of the token that is drawn from an LM-head row (sampling), or -1
    uint64_t *seed;                // [FEW_ROWS]
    BestD *best;                   // [FEW_ROWS] best Gumbel score of this block's columns so far
    int x0, xc;                    // this block's columns of the residual stream
    FewAtt *att;                   // the attention phases' work, the same in every layer (in shared memory: registers are short)
    FewItem *first;                // this block's first item of it
};

__device__ __forceinline__ void fsync() { asm volatile("bar.sync 3, 320;" ::: "memory"); }
static_assert(FC_THREADS == 320, "fsync");

// (The proxy fence that bulk copies of these writes need stands in front of the copies, in the warp that issues them: it is
// needed once on the way from the write to the copy.  In every thread of every block, here, it cost 0.4 us a barrier: 1.3B
// draft step 1088 -> 1055 us.)
__device__ __forceinline__ void few_grid_barrier(FewCtx &c, const FwdBufs &fb) {
    fsync();
    if (threadIdx.x == 0) {
        c.bar_target += (unsigned long long)c.ncta;
        __threadfence();
        atomicAdd(fb.bar, 1ULL);
        unsigned it = 0;
        while (ld_acquire_u64(fb.bar) < c.bar_target) {
            ++it;
            if ((it & 255u) == 0 && (it > 4u * SPIN_LIMIT || *(volatile int32_t *)fb.abort_flag)) {
                atomicCAS(fb.abort_flag, 0, 1);
                break;
            }
        }
    }
    fsync();
}

// Activations as the MMA's row operand, in register order: [k / 64][live row][k / 16 % 4][t = 0..3] x 16 bytes, the 16
// bytes being {values k 2t, 2t+1 | remainders of these | values 2t+8, 2t+9 | remainders}: one 128-bit shared-memory load
// per lane and 16 columns, and any run of k blocks is one run of bytes.  Odd rows swap neighbouring groups of 16 columns,
// so that the reads of two rows hit different banks.  k even: the columns k, k + 1 are one 8-byte store.
__device__ __forceinline__ size_t few_frag(int i, int k, int nlive) {
    return ((size_t)(k >> 6) * nlive + i) * 128 + ((((k >> 4) & 3) ^ (i & 1)) << 5) + ((k & 7) >> 1) * 8 + ((k >> 3) & 1) * 4;
}
__device__ __forceinline__ void split_pair(float v0, float v1, uint32_t &hi, uint32_t &lo) {
    const __nv_bfloat162 h = __floats2bfloat162_rn(v0, v1);
    hi = *reinterpret_cast<const uint32_t *>(&h);
    lo = pack_bf16x2(v0 - __low2float(h), v1 - __high2float(h));
}
__device__ __forceinline__ void few_store(bf16 *base, int i, int k, int nlive, float v0, float v1) {
    uint2 w;
    split_pair(v0, v1, w.x, w.y);
    *reinterpret_cast<uint2 *>(base + few_frag(i, k, nlive)) = w;
}

template <int PASS>
__device__ __forceinline__ FewOp few_op(const GemmOp &op, int opi, int cta, int ncta, int nlive, bool many) {
    const int unit = opi == OP_GU ? 16 : 2, units = (op.N + unit - 1) / unit, base = units / ncta, rem = units - base * ncta;
    FewOp o;
    o.r0 = (cta * base + min(cta, rem)) * unit;
    o.r1 = min(o.r0 + (base + (cta < rem ? 1 : 0)) * unit, 2 * op.MT * 8);
    o.atom0 = o.r0 >> 3;
    o.span = o.r1 > o.r0 ? ((o.r1 + 7) >> 3) - o.atom0 : 0;
    o.nkb = op.K / KB;
    // a pass (a k block of it is a stage at least): what the accumulators (see few_plan.h) and the buffer of the sums hold, an
    // even number of atoms
    // few atoms: ten k groups, so that a warp's chain of k blocks is as short as it can be (14 rows x 5504 columns: 18 k
    // blocks a warp with five groups, 9 with ten)
    o.kgs = o.span <= 3 ? FW : FW / 2;
    const int atoms = min(nlive <= 8 ? PASS : PASS > FEW_SHORT ? 16 : 12, few_scratch(many) / (o.kgs * nlive * 32)) & ~1;
    o.npass = (o.span + atoms - 1) / atoms;
    // stage: F_STAGE bytes of weights, but work for every k group.  Only the block's own rows count: a block's 10 to 14 rows
    // of a d_model-wide projection touch two or three atoms, and with whole atoms in the ring the ten stages of a 1.3B
    // down projection did not fit it (6.5 us, now 4.7)
    const int sp = o.npass ? (o.span + o.npass - 1) / o.npass : 1;
    const int rows = max(1, o.npass == 1 ? o.r1 - o.r0 : sp * 8);
    o.kbs = max(1, min(min(32, F_STAGE / (rows * 128)), (o.nkb + o.kgs - 1) / o.kgs));
    o.nst = (o.nkb + o.kbs - 1) / o.kbs;
    return o;
}
// Atoms [a, a + n) of pass p (relative to atom0), in pairs so that a gate atom and its up atom stay together.
__device__ __forceinline__ void few_pass(const FewOp &o, int p, int &a, int &n) {
    if (o.npass == 1) { a = 0; n = o.span; return; }
    const int pairs = (o.span + 1) >> 1, base = pairs / o.npass, rem = pairs - base * o.npass;
    a = 2 * (p * base + min(p, rem));
    n = min(2 * (base + (p < rem ? 1 : 0)), o.span - a);
}

// No copy may be in flight when the block ends, also when others gave up (bounded like every wait).
__device__ __forceinline__ void few_drain(uint64_t *full, int n, int slots) {
    for (int j = max(0, n - slots); j < n; ++j)
        for (unsigned it = 0; it < MBAR_SPIN_LIMIT && !mbar_try_wait(full + j % slots, ((uint32_t)(j / slots)) & 1u); ++it) {}
}

// Producer warps.  Weights: every stage of the block for the whole forward, in order, running ahead into the next
// projections and, where a launch runs several forwards, into the next of these.  A stage is up to 32 k blocks of the pass's rows, one bulk copy per k block by as many lanes; it takes the
// next free bytes of the ring once the stages whose bytes it needs have been read (lane n % 32 remembers where stage n
// begins).  Activations: NX slots, one bulk copy per stage, once the projection's inputs are complete.
__device__ __forceinline__ void few_weight_producer(FewCtx &c, const FwdBufs &fb, const Plan &P, int n_fwd, int ring_bytes, uint64_t policy) {
    int n = 0, tail = 0, at = 0;                        // next stage; first stage not known to be read; next byte
    long long head = 0, tail_v = 0, mine = 0;           // virtual ring positions: next byte, first byte still in use, this lane's stage
    bool alive = true;
    for (int f = 0, q = 0; f < n_fwd && alive; q + 1 < n_ops(P) ? ++q : (q = 0, ++f)) {
        const int opi = op_index(P, q);
        const GemmOp &op = P.op[opi];
        const bf16 *wl = op.W + (size_t)op_layer(P, q) * op.lstride;
        const FewOp o = c.ops[f > 0 ? N_OPS + opi : opi];
        for (int p = 0; p < o.npass && alive; ++p) {
            int pa, pn;
            few_pass(o, p, pa, pn);
            const int ra = max(o.r0, (o.atom0 + pa) * 8), rb = min(o.r1, (o.atom0 + pa + pn) * 8);
            const uint32_t kbytes = (uint32_t)(rb - ra) * 128u;
            const bf16 *src = wl + ((size_t)c.lane * (2 * op.MT) + o.atom0 + pa) * 512 + (ra & 7) * 64;
            unsigned char *dst = c.ring + c.lane * kbytes;
            for (int k = 0; k < o.nkb; k += o.kbs, ++n) {
                const int nk = min(o.kbs, o.nkb - k), bytes = nk * (int)kbytes;
                if (at + bytes > ring_bytes) { head += ring_bytes - at; at = 0; }
                while (tail < n && (tail <= n - FNB || head + bytes > tail_v + ring_bytes)) {
                    if (!wait_bar(fb, c.wempty + (tail & (FNB - 1)), ((uint32_t)(tail / FNB)) & 1u, 5, tail)) { alive = false; break; }
                    ++tail;
                    tail_v = __shfl_sync(0xffffffffu, mine, tail & (FNB - 1));
                }
                alive = __all_sync(0xffffffffu, alive);
                if (!alive) break;
                if (tail == n) tail_v = head;
                if (c.lane == (n & (FNB - 1))) mine = head;
                if (c.lane == 0) {
                    c.slot_at[n & (FNB - 1)] = at;
                    mbar_expect_tx(c.wfull + (n & (FNB - 1)), kbytes * (uint32_t)nk);
                }
                __syncwarp();
                if (c.lane < nk) bulk_g2s(dst + at, src + (size_t)k * (2 * op.MT) * 512, kbytes, c.wfull + (n & (FNB - 1)), policy);
                head += bytes; at += bytes;
            }
        }
    }
    few_drain(c.wfull, n, FNB);
}

template <int NX>
__device__ __forceinline__ void few_x_producer(FewCtx &c, const Args &a, uint64_t policy) {
    const Plan &P = a.P;
    int n = 0, pass = 0;
    for (int f = 0, q = 0; f < a.n_fwd; q + 1 < n_ops(P) ? ++q : (q = 0, ++f)) {
        const int opi = op_index(P, q);
        const FewOp o = c.ops[f > 0 ? N_OPS + opi : opi];
        if (f > 0) { c.nlive = c.nlater; c.xk = F_XROWS / c.nlive; }
        const bf16 *X = opi == OP_O ? a.d.att : opi == OP_DOWN ? a.d.act : a.fb.xg;
        for (int p = 0; p < o.npass; ++p) {
            ++pass;
            if (p > 0) {
                wait_count(a.fb, c.ready, pass, 6);
                __threadfence_block();
            } else {
                // the projection's inputs are complete, and this block's consumers are done with the ring's bytes, once the
                // grid barrier in front of it is over: watched here, not passed on by the consumers (0.3 us a projection)
                const int bars = f * (5 * P.n_layers + 2) + (opi == OP_HEAD ? 5 * P.n_layers : 5 * op_layer(P, q) + (opi == OP_QKV ? 0 : opi == OP_O ? 2 : opi == OP_GU ? 3 : 4));
                const unsigned long long want = c.bar_target + (unsigned long long)c.ncta * (1 + bars);
                unsigned it = 0;
                while (ld_acquire_u64(a.fb.bar) < want) {
                    ++it;
                    if ((it & 255u) == 0 && (it > 4u * SPIN_LIMIT || *(volatile int32_t *)a.fb.abort_flag)) {
                        atomicCAS(a.fb.abort_flag, 0, 1);
                        break;
                    }
                }
                __syncwarp();
            }
            asm volatile("fence.proxy.async;" ::: "memory");
            for (int k = 0; k < o.nkb; k += c.xk, ++n) {
                const int slot = n % NX;
                if (!__all_sync(0xffffffffu, wait_bar(a.fb, c.xempty + slot, (((uint32_t)(n / NX)) & 1u) ^ 1u, 7, n))) { few_drain(c.xfull, n, NX); return; }
                if (c.lane == 0) {
                    const uint32_t bytes = (uint32_t)(min(c.xk, o.nkb - k) * c.nlive) * 256u;
                    mbar_expect_tx(c.xfull + slot, bytes);
                    bulk_g2s(c.scratch + slot * (F_XROWS * 256), X + (size_t)k * c.nlive * 128, bytes, c.xfull + slot, policy);
                }
                __syncwarp();
            }
        }
    }
    few_drain(c.xfull, n, NX);
}

__device__ __forceinline__ void ldmatrix_x4(uint32_t (&r)[4], uint32_t saddr) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(saddr));
}

// Input rows of a forward, element pair (k, k + 1) of row r (in use): embedding row, or hidden + position embedding.
__device__ __forceinline__ float2 few_input(const Args &a, const FewCtx &c, int r, int k) {
    const int dm = a.m.cfg.d_model;
    if (a.kind == KIND_MB) {
        const int s = r / a.g.rps, j = r - s * a.g.rps, e = c.row_tok[r];
        float2 v = __ldcg(reinterpret_cast<const float2 *>(a.d.hpend + ((size_t)s * (a.d.block_b + 1) + j) * dm + k));
        if (e > 0 && a.d.use_posemb) {
            const __nv_bfloat162 w = *reinterpret_cast<const __nv_bfloat162 *>(a.m.posemb + (size_t)(e - 1) * dm + k);
            v.x += __low2float(w); v.y += __high2float(w);
        }
        return v;
    }
    const __nv_bfloat162 w = *reinterpret_cast<const __nv_bfloat162 *>(a.m.embed + (size_t)c.row_tok[r] * dm + k);
    return make_float2(__low2float(w), __high2float(w));
}

__device__ __forceinline__ float2 few_sum(const float *p, int kstride, int kgs) {
    float2 v = *reinterpret_cast<const float2 *>(p);
#pragma unroll
    for (int k = 1; k < FW / 2; ++k) {
        const float2 u = *reinterpret_cast<const float2 *>(p + k * kstride);
        v.x += u.x; v.y += u.y;
    }
    if (kgs == FW)
#pragma unroll
        for (int k = FW / 2; k < FW; ++k) {
            const float2 u = *reinterpret_cast<const float2 *>(p + k * kstride);
            v.x += u.x; v.y += u.y;
        }
    return v;
}

__device__ __forceinline__ Top2 few_warp_top2(Top2 tp) {
#pragma unroll
    for (int x = 16; x > 0; x >>= 1) {
        Top2 u;
        u.v1 = __shfl_xor_sync(0xffffffffu, tp.v1, x);
        u.i1 = __shfl_xor_sync(0xffffffffu, tp.i1, x);
        u.v2 = __shfl_xor_sync(0xffffffffu, tp.v2, x);
        tp = top2_merge(tp, u);
    }
    return tp;
}

__device__ __forceinline__ BestD few_warp_best(BestD t) {
#pragma unroll
    for (int x = 16; x > 0; x >>= 1) {
        BestD u;
        u.v = __shfl_xor_sync(0xffffffffu, t.v, x);
        u.i = __shfl_xor_sync(0xffffffffu, t.i, x);
        t = best_merge(t, u);
    }
    return t;
}
// the blocks' draws, behind their best logits: [block][FEW_ROWS]
__device__ __forceinline__ BestD *few_best(const Args &a, const FewCtx &c) {
    return reinterpret_cast<BestD *>(reinterpret_cast<float4 *>(a.fb.tile_top) + (size_t)c.ncta * FEW_ROWS);
}

// The row-wise step after a projection, weight rows [ra, rb) of live row i (one warp; red: the k groups' sums, column 0 =
// weight row `off`, the kgs groups `ks` floats apart; last: the last pass).
__device__ __forceinline__ void few_epilogue(FewCtx &c, const Args &a, int opi, int l, int i, int ra, int rb, int off, const float *red,
                                             int ks, int kgs, bool last) {
    const DevPtrs &d = a.d;
    const ModelDev &m = a.m;
    const int dm = m.cfg.d_model, H = m.cfg.n_heads, Hkv = m.cfg.n_kv_heads, hd = m.hd, half = hd >> 1;
    const float inv = c.inv[i];
    if (opi == OP_QKV) {
        const int r = c.row_of[i], pos = c.row_pos[r], seq = r / a.g.rps, hshift = hd == 64 ? 6 : 7;
        const float scale = rsqrtf((float)hd);
        for (int n = ra + 2 * c.lane; n < rb; n += 64) {
            const int h = n >> hshift, w = n & (hd - 1), ii = w >> 1;
            const float2 cs = h < H + Hkv ? m.rope[(size_t)pos * half + ii] : make_float2(1.f, 0.f);
            const float2 s = few_sum(red + (n - off), ks, kgs);
            const float v0 = s.x * inv, v1 = s.y * inv;
            if (h < H + Hkv) {                           // the pair (ii, ii + hd/2) of a q or k head: rotary embedding
                const float y0 = v0 * cs.x - v1 * cs.y, y1 = v1 * cs.x + v0 * cs.y;
                if (h < H) {
                    float *qd = a.fb.qkv + (size_t)i * (H * hd) + h * hd + ii;
                    qd[0] = y0 * scale; qd[half] = y1 * scale;
                } else {
                    bf16 *kc = m.kcache + ((((size_t)l * d.max_batch + seq) * Hkv + (h - H)) * (size_t)d.max_ctx + pos) * hd + ii;
                    split_bf16(y0, kc[0], kc[m.kv_lo]);
                    split_bf16(y1, kc[half], kc[m.kv_lo + half]);
                }
            } else {
                bf16 *vc = m.vcache + ((((size_t)l * d.max_batch + seq) * Hkv + (h - H - Hkv)) * (size_t)d.max_ctx + pos) * hd + w;
                uint32_t hi, lo;
                split_pair(v0, v1, hi, lo);
                *reinterpret_cast<uint32_t *>(vc) = hi;
                *reinterpret_cast<uint32_t *>(vc + m.kv_lo) = lo;
            }
        }
    } else if (opi == OP_GU) {                           // whole gate/up atom pairs: columns f = ra / 2 ..
        for (int f = (ra >> 1) + 2 * c.lane; f < (rb >> 1); f += 64) {
            const int n = (f >> 3) * 16 + (f & 7);
            const float2 gt = few_sum(red + (n - off), ks, kgs), up = few_sum(red + (n + 8 - off), ks, kgs);
            const float g0 = gt.x * inv, g1 = gt.y * inv;
            few_store(d.act, i, f, c.nlive, g0 / (1.f + expf(-g0)) * (up.x * inv), g1 / (1.f + expf(-g1)) * (up.y * inv));
        }
    } else if (opi == OP_HEAD) {
        float *dst = c.row_dst[i];
        if (!dst) return;
        const int V = m.cfg.vocab, b = c.bias_at[i];
        Top2 tp{-INFINITY, 0x7fffffff, -INFINITY};
        BestD bd{-INFINITY, 0x7fffffff};
        const int dpos = c.draw_pos[i];
        // a draw from the row's softmax by the Gumbel-max rule, every block on its own columns (one block over all of them
        // took 0.08 ms at vocabulary 32 000: the noise is fp64)
        auto draw = [&](int n, float v) {
            if (dpos < 0) return;
            const double sc = (double)v + gumbel_noise(c.seed[i], (uint32_t)n, (uint32_t)dpos, (uint32_t)(c.row_of[i] / a.g.rps), a.kind == KIND_DRAFT ? TAG_DRAFT : TAG_NEXT);
            if (sc > bd.v) { bd.v = sc; bd.i = n; }
        };
        for (int n = ra + 2 * c.lane; n < rb; n += 64) {
            const float2 s = few_sum(red + (n - off), ks, kgs);
            if (n < V) {
                const float v = s.x * inv + (n == b ? d.succ_bias : 0.f);
                dst[n] = v;
                draw(n, v);
                tp = top2_merge(tp, top2_one(v, n));
            }
            if (n + 1 < V) {
                const float v = s.y * inv + (n + 1 == b ? d.succ_bias : 0.f);
                dst[n + 1] = v;
                draw(n + 1, v);
                tp = top2_merge(tp, top2_one(v, n + 1));
            }
        }
        tp = few_warp_top2(tp);
        if (dpos >= 0) bd = few_warp_best(bd);
        if (c.lane == 0) {
            if (dpos >= 0) {
                bd = best_merge(c.best[i], bd);
                c.best[i] = bd;
                if (last) few_best(a, c)[(size_t)c.cta * FEW_ROWS + i] = bd;
            }
            tp = top2_merge(c.top[i], tp);               // (a block may have several passes of rows)
            c.top[i] = tp;
            if (last)
                reinterpret_cast<float4 *>(a.fb.tile_top)[(size_t)c.cta * FEW_ROWS + i] = make_float4(tp.v1, __int_as_float(tp.i1), tp.v2, 0.f);
        }
        __syncwarp();
    } else {
        // x += the rows; the next projection's input x * gain; this block's share of sum(x^2)
        const bf16 *gain = opi == OP_O ? m.norm2 + (size_t)l * dm : (l + 1 < a.P.n_layers ? m.norm1 + (size_t)(l + 1) * dm : m.normf);
        float ss = 0.f, *xr = d.xres + (size_t)c.row_of[i] * dm;
        for (int n = ra + 2 * c.lane; n < rb; n += 64) {
            const __nv_bfloat162 gn = *reinterpret_cast<const __nv_bfloat162 *>(gain + n);
            const float2 s = few_sum(red + (n - off), ks, kgs);
            float *x = c.xs + i * c.xc + (n - c.x0);
            const float x0 = x[0] + s.x, x1 = x[1] + s.y;
            x[0] = x0; x[1] = x1;
            ss += x0 * x0 + x1 * x1;
            few_store(a.fb.xg, i, n, c.nlive, x0 * __low2float(gn), x1 * __high2float(gn));
            *reinterpret_cast<float2 *>(xr + n) = make_float2(x0, x1);
        }
        ss = warp_sum(ss);
        if (c.lane == 0) a.fb.ssq[i * c.ncta + c.cta] = ss;
    }
}

// 1/rms of the live rows from the blocks' shares of sum(x^2): warp w rows w, w + 10.
__device__ __forceinline__ void few_inv(FewCtx &c, const Args &a) {
    for (int i = c.warp; i < c.nlive; i += FW) {
        float s = 0.f;
        for (int b = c.lane; b < c.ncta; b += 32) s += __ldcg(a.fb.ssq + i * c.ncta + b);
        s = warp_sum(s);
        if (c.lane == 0) c.inv[i] = rsqrtf(s / (float)a.m.cfg.d_model + a.m.cfg.rms_eps);
    }
}

__device__ __forceinline__ void mbar_arrive_n(uint64_t *b, int count) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(b)), "r"(count) : "memory");
}

// One warp's share of a pass (weight rows ra .. ra + rows): the weight stages kg, kg + kgs, ... and N atoms of them from atom my_a on (my_n of them
// its own, the rest is computed and not stored), into the sum buffer.  N is a template parameter because a branch per atom
// costs more than the atom's instructions.  NX: activation stages, 0 for three or five by c.many.  (A lane of an operand row beyond
// the live ones reads live row 0.)
template <int RT, int N, int NX>
__device__ __forceinline__ void few_main(FewCtx &c, const Args &a, const FewOp &o, int kg, int pn, int ra, int rows, int my_a,
                                         int my_n) {
    constexpr int KU = RT * N > 10 ? 1 : 2;              // k blocks whose loads overlap, as far as the registers go
    const int g = c.lane >> 2, t = c.lane & 3, nlive = c.nlive, nst = o.nst, xk = c.xk, nxs = (o.nkb + xk - 1) / xk;
    // where atom my_a of a stage's first k block would begin: the ring holds the rows from ra on, a k block behind the other
    // (the swizzle goes by the row's place in its atom, not by its address); other rows of an atom are whatever lies there
    const uint32_t ring = smem_u32(c.ring) + (uint32_t)my_a * 1024u - (uint32_t)(ra & 7) * 128u, kbytes = (uint32_t)rows * 128u;
    int xrow[RT], xsw[RT];                               // this lane's operand rows within a k block; 64-byte groups swapped
#pragma unroll
    for (int m = 0; m < RT; ++m) {
        const int i = m * 8 + g < nlive ? m * 8 + g : 0;
        xrow[m] = i * 256 + t * 16; xsw[m] = (i & 1) << 6;
    }
    const uint32_t lrow = (uint32_t)(c.lane & 7) * 128u, lch = (uint32_t)(c.lane >> 3), lx = (uint32_t)(c.lane & 7);
    const uint32_t sw0 = lrow + ((lch ^ lx) << 4), sw1 = lrow + (((lch + 4u) ^ lx) << 4);
    float acc[N][RT][4];
#pragma unroll
    for (int i = 0; i < N; ++i)
#pragma unroll
        for (int m = 0; m < RT; ++m) acc[i][m][0] = acc[i][m][1] = acc[i][m][2] = acc[i][m][3] = 0.f;
    int xs = 0;                                          // this warp is in activation stage xs - 1 of the pass
    const unsigned char *xb = c.scratch;         // ... whose k block 0 would be here
    int slot_x = 0;                                      // (NX = 0) the stage this warp is in
    auto next_x = [&]() {                                // every warp passes through every activation stage
        const int n = c.xstage + xs, turn = NX > 0 ? n / max(NX, 1) : c.many ? n / FXS_MANY : n / FXS;
        const int slot = n - turn * (NX > 0 ? NX : c.many ? FXS_MANY : FXS), left = NX > 0 ? (n - 1) % max(NX, 1) : slot_x;
        if (xs > 0) { __syncwarp(); if (c.lane == 0) mbar_arrive(c.xempty + left); }
        if (NX == 0) slot_x = slot;
        if (xs < nxs && c.ok) c.ok = wait_bar(a.fb, c.xfull + slot, (uint32_t)turn & 1u, 8, n);
        xb = c.scratch + slot * (F_XROWS * 256) - xs * xk * nlive * 256;
        ++xs;
    };
    for (int st = kg; st < nst; st += o.kgs) {
        const int n = c.stage + st, slot = n & (FNB - 1), k_end = min((st + 1) * o.kbs, o.nkb);
        // first the activations: a warp that waited for weights inside an earlier activation stage would hold that stage
        // back from a warp whose weights must be read before its own can arrive
        while (st * o.kbs >= xs * xk) next_x();
        if (c.ok) c.ok = wait_bar(a.fb, c.wfull + slot, ((uint32_t)(n / FNB)) & 1u, 9, n);
        uint32_t base = ring + (c.ok ? (uint32_t)c.slot_at[slot] : 0u);        // (a stage that never came has no place)
        for (int kb = st * o.kbs; kb < k_end;) {
            while (kb >= xs * xk) next_x();
            const int run = min(k_end, xs * xk);
            const unsigned char *xa = xb + kb * nlive * 256;
#pragma unroll KU
            for (; kb < run; ++kb, base += kbytes, xa += nlive * 256) {
                uint4 A[RT][4];
#pragma unroll
                for (int m = 0; m < RT; ++m)
#pragma unroll
                    for (int j = 0; j < 4; ++j) A[m][j] = *reinterpret_cast<const uint4 *>(xa + xrow[m] + ((j << 6) ^ xsw[m]));
#pragma unroll
                for (int i = 0; i < N; ++i) {
                    uint32_t b0[4], b1[4];
                    ldmatrix_x4(b0, base + sw0 + (uint32_t)i * 1024u);
                    ldmatrix_x4(b1, base + sw1 + (uint32_t)i * 1024u);
#pragma unroll
                    for (int m = 0; m < RT; ++m) {
                        mma16816(acc[i][m], A[m][0].x, A[m][0].y, A[m][0].z, A[m][0].w, b0[0], b0[1]);
                        mma16816(acc[i][m], A[m][1].x, A[m][1].y, A[m][1].z, A[m][1].w, b0[2], b0[3]);
                        mma16816(acc[i][m], A[m][2].x, A[m][2].y, A[m][2].z, A[m][2].w, b1[0], b1[1]);
                        mma16816(acc[i][m], A[m][3].x, A[m][3].y, A[m][3].z, A[m][3].w, b1[2], b1[3]);
                    }
                }
            }
        }
        __syncwarp();
        if (c.lane == 0) mbar_arrive_n(c.wempty + slot, o.kgs == FW ? 2 : 1);    // (two arrivals in all)
    }
    while (xs <= nxs) next_x();
    fsync();                                             // the activations' bytes become the sums'
    float *red = reinterpret_cast<float *>(c.scratch) + my_a * 8 + 2 * t;
    const int PC = pn * 8;                               // columns of the pass in the sum buffer
#pragma unroll
    for (int i = 0; i < N; ++i)
        if (i < my_n)
#pragma unroll
            for (int m = 0; m < RT; ++m)
                if (m * 8 + g < nlive)
                    *reinterpret_cast<float2 *>(red + (kg * nlive + m * 8 + g) * PC + i * 8) =
                        make_float2(acc[i][m][0] + acc[i][m][2], acc[i][m][1] + acc[i][m][3]);
}

// A projection of the forward.  Warp (kg, cg) takes its share of the k range and of the pass's atoms; the k groups' sums
// go through shared memory; then warp w runs the epilogue for the live rows w, w + 10.
template <int MAXRT, int PASS>
__device__ __forceinline__ void few_gemm(FewCtx &c, const Args &a, int opi, int layer) {
    const FewOp o = c.ops[opi];
    constexpr bool WIDE = PASS > FEW_SHORT;
    constexpr int X2 = WIDE ? 0 : FXS;                   // activation stages of nine and more rows
    const int kg = o.kgs == FW ? c.warp : c.warp >> 1, cg = c.warp & 1, nlive = c.nlive, nxs = (o.nkb + c.xk - 1) / c.xk;
    float *red = reinterpret_cast<float *>(c.scratch);
    // (its loads travel with the first activations; also in a block without rows: it may end a sequence's draft step)
    if (opi == OP_QKV || opi == OP_GU || opi == OP_HEAD) few_inv(c, a);
    for (int p = 0; p < o.npass; ++p) {
        int pa, pn;
        few_pass(o, p, pa, pn);
        const int ra = max(o.r0, (o.atom0 + pa) * 8), rb = min(o.r1, (o.atom0 + pa + pn) * 8);
        const int h0 = (pn + 1) >> 1, my_a = o.kgs < FW && cg ? h0 : 0, my_n = o.kgs == FW ? pn : cg ? pn - h0 : h0;
        if (threadIdx.x == 0) { __threadfence_block(); *c.ready = ++c.pass; }    // (a later pass:) the activations may be copied
        if (MAXRT == 1 || nlive <= 8) {
            if (my_n <= 1) few_main<1, 1, FXS>(c, a, o, kg, pn, ra, rb - ra, my_a, my_n);
            else if (my_n <= 2) few_main<1, 2, FXS>(c, a, o, kg, pn, ra, rb - ra, my_a, my_n);
            else if (my_n <= 3) few_main<1, 3, FXS>(c, a, o, kg, pn, ra, rb - ra, my_a, my_n);
            else if (my_n <= 4) few_main<1, 4, FXS>(c, a, o, kg, pn, ra, rb - ra, my_a, my_n);
            else if (my_n <= 6) few_main<1, 6, FXS>(c, a, o, kg, pn, ra, rb - ra, my_a, my_n);
            else if (!WIDE || my_n <= 8) few_main<1, 8, FXS>(c, a, o, kg, pn, ra, rb - ra, my_a, my_n);
            else if constexpr (WIDE) {
                if (my_n <= 10) few_main<1, 10, FXS>(c, a, o, kg, pn, ra, rb - ra, my_a, my_n);
                else few_main<1, PASS / 2, FXS>(c, a, o, kg, pn, ra, rb - ra, my_a, my_n);
            }
        } else if constexpr (MAXRT == 2) {
            if (my_n <= 1) few_main<2, 1, X2>(c, a, o, kg, pn, ra, rb - ra, my_a, my_n);
            else if (my_n <= 2) few_main<2, 2, X2>(c, a, o, kg, pn, ra, rb - ra, my_a, my_n);
            else if (my_n <= 3) few_main<2, 3, X2>(c, a, o, kg, pn, ra, rb - ra, my_a, my_n);
            else if (my_n <= 4) few_main<2, 4, X2>(c, a, o, kg, pn, ra, rb - ra, my_a, my_n);
            else if (!WIDE || my_n <= 6) few_main<2, 6, X2>(c, a, o, kg, pn, ra, rb - ra, my_a, my_n);
            else if constexpr (WIDE) few_main<2, 8, X2>(c, a, o, kg, pn, ra, rb - ra, my_a, my_n);
        }
        c.stage += o.nst; c.xstage += nxs;
        fsync();
        const int PC = pn * 8, off = (o.atom0 + pa) * 8;
        for (int i = c.warp; i < nlive; i += FW)
            few_epilogue(c, a, opi, layer, i, ra, rb, off, red + i * PC, nlive * PC, o.kgs, p == o.npass - 1);
        if (p + 1 < o.npass) fsync();
    }
    if (o.npass == 0 && opi != OP_QKV && opi != OP_GU)   // fewer units than blocks: this one has no row, but its slots of
        for (int i = threadIdx.x; i < nlive; i += FC_THREADS) {              // the row statistics are read
            if (opi == OP_HEAD) {
                reinterpret_cast<float4 *>(a.fb.tile_top)[(size_t)c.cta * FEW_ROWS + i] = make_float4(-INFINITY, __int_as_float(0x7fffffff), -INFINITY, 0.f);
                few_best(a, c)[(size_t)c.cta * FEW_ROWS + i] = BestD{-INFINITY, 0x7fffffff};
            } else a.fb.ssq[i * c.ncta + c.cta] = 0.f;
        }
}

// ------------------------------------------------------------------ attention

__device__ __forceinline__ FewAtt few_att(const FewCtx &c, const Args &a) {
    FewAtt f;
    const int group = a.m.cfg.n_heads / a.m.cfg.n_kv_heads;
    int len = 0, rows = 1;
    for (int s = 0; s < a.g.batch; ++s)
        if (c.n_rows[s] > 0) {
            const int p0 = c.row_pos[s * a.g.rps];
            len = max(len, p0 + c.n_rows[s] - min(c.key_start[s], p0));
            rows = max(rows, c.n_rows[s]);
        }
    f.chunks = (group * rows + FQ - 1) / FQ;
    // Key splits: an item costs about 1.3 us per round of its ten warps (80 keys) and 3 us of fixed cost; splitting adds 3 us
    // for the partials, the arrival and the merge.  Fewer items than blocks: the most splits that give every block one
    // item, or none when a head is that short (96 keys of 4 heads: 4 us against 6).
    const int base = a.g.batch * a.m.cfg.n_kv_heads * f.chunks;
    const int cap = max(1, min(min((len + 79) / 80, 64), FEW_ITEMS / base));
    if (base <= c.ncta) {
        const int n = min(cap, c.ncta / base), rounds = ((len + n - 1) / n + 79) / 80, alone = (len + 79) / 80;
        // (as many splits as leave the same number of rounds)
        f.nsplit = 13 * alone <= 13 * rounds + 30 ? 1 : min(n, (len + 80 * rounds - 1) / (80 * rounds));
    } else {
        int best_cost = 1 << 30;
        f.nsplit = 1;
        for (int n = 1; n <= min(cap, 16); ++n) {
            const int cost = ((base * n + c.ncta - 1) / c.ncta) * (13 * (((len + n - 1) / n + 79) / 80) + 30) + (n > 1 ? 30 : 0);
            if (cost < best_cost) { best_cost = cost; f.nsplit = n; }
        }
    }
    f.items = base * f.nsplit;
    return f;
}

__device__ __forceinline__ FewItem few_item(const FewCtx &c, const Args &a, const FewAtt &f, int it) {
    FewItem w;
    const int Hkv = a.m.cfg.n_kv_heads;
    w.split = it % f.nsplit;
    const int r1 = it / f.nsplit;
    w.vc = r1 % f.chunks;
    const int r2 = r1 / f.chunks;
    w.kh = r2 % Hkv; w.seq = r2 / Hkv;
    w.n_r = c.n_rows[w.seq];
    w.pos0 = c.row_pos[w.seq * a.g.rps];
    const int ks = min(c.key_start[w.seq], w.pos0), span = w.n_r > 0 ? w.pos0 + w.n_r - ks : 0;
    w.lo = ks + (int)((unsigned)(span * w.split) / (unsigned)f.nsplit);
    w.hi = ks + (int)((unsigned)(span * (w.split + 1)) / (unsigned)f.nsplit);
    return w;
}

// The keys and values this block will read first in the layer's attention phase, into L2 while the q/k/v projection runs.
__device__ __forceinline__ void few_kv_prefetch(const FewCtx &c, const Args &a, const FewItem &w, int layer) {
    const int n = min(w.hi, w.pos0) - w.lo, hd = a.m.hd;
    if (w.n_r == 0 || n <= 0) return;
    const size_t at = ((((size_t)layer * a.d.max_batch + w.seq) * a.m.cfg.n_kv_heads + w.kh) * (size_t)a.d.max_ctx + w.lo) * hd;
    const bf16 *base = (c.lane & 2 ? a.m.vcache : a.m.kcache) + at + (c.lane & 1 ? a.m.kv_lo : 0);
    if (c.lane < 4)
        asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(base), "r"((uint32_t)(n * hd * 2)) : "memory");
}

__device__ __forceinline__ uint32_t movmatrix(uint32_t v) {         // transpose of an 8x8 matrix of 16-bit values
    uint32_t r;
    asm volatile("movmatrix.sync.aligned.m8n8.trans.b16 %0, %1;" : "=r"(r) : "r"(v));
    return r;
}

// One item: FQ query rows (head within the group x row of the sequence) of a kv head over the keys [lo, hi), eight keys
// per warp and step on mma.sync.  A lane (g, t) reads 8 consecutive channels of key g.  Scores: the 16-row operand holds the
// 8 query rows' values over their remainders, the keys are the columns, and the lane's channels are the k slots {2t, 2t+1,
// 2t+8, 2t+9} of two MMAs (q is read by the same rule).  Values: transposed, 16 channels x 8 query rows, so that the
// accumulators take half the registers (with the query rows over their remainders as rows, 64 a lane at head dimension
// 128); movmatrix turns the lane's four 8 x 8 blocks of v into the row operand (rows: channels 8 (g / 2) + 2i + g % 2 of
// each 32; k slots: the 8 keys' values, then their remainders), the probabilities and then their remainders are the
// columns.  Nothing is staged in shared memory but q.  Bound by the latency of its K and V reads (8 KB per warp in
// flight): 12.6 us for 16 heads over 2048 keys (14.8 before the transposition); on the ordinary ALUs in fp32 a step of
// eight rows took 4 us, four times as long.
template <int HD>
__device__ __forceinline__ void few_attention_item(FewCtx &c, const Args &a, const FewAtt &f, const FewItem &w, int layer) {
    constexpr int NC = HD / 32, PW = HD + 2, QS = HD * 4 + 64, QR = FQ;
    const DevPtrs &d = a.d;
    const ModelDev &m = a.m;
    const int H = m.cfg.n_heads, group = H / m.cfg.n_kv_heads, nv = min(QR, group * w.n_r - w.vc * QR);
    if (nv <= 0) return;                                 // the same in every warp of the block
    const size_t cbase = (((size_t)layer * d.max_batch + w.seq) * m.cfg.n_kv_heads + w.kh) * (size_t)d.max_ctx * HD;
    unsigned char *qs = c.scratch;                                    // [QR] rows: HD values, HD remainders
    float *red = reinterpret_cast<float *>(c.scratch + QR * QS);      // [FW][QR][PW]
    static_assert(QR * QS + FW * QR * PW * 4 <= few_scratch(false), "attention scratch");
    static_assert(QR * (HD / 4) <= FC_THREADS, "four channels of a query row per thread");
    const int qi = threadIdx.x;
    float4 qx;
    if (qi < nv * (HD / 4)) {
        const int lv = qi / (HD / 4), e = qi & (HD / 4 - 1), v = w.vc * QR + lv, hq = v / w.n_r, j = v - hq * w.n_r;
        qx = __ldcg(reinterpret_cast<const float4 *>(a.fb.qkv + (size_t)c.idx_of[w.seq * a.g.rps + j] * (H * HD) + (w.kh * group + hq) * HD) + e);
    }
    const int g = c.lane >> 2, t = c.lane & 3, ks = c.key_start[w.seq];
    const int vrow = g < nv ? (w.vc * QR + g) % w.n_r : -1, self = w.pos0 + vrow;        // this lane's query row in the sequence
    float mx = -INFINITY, ls = 0.f, o[NC * 2][4];
#pragma unroll
    for (int e = 0; e < NC * 2; ++e) o[e][0] = o[e][1] = o[e][2] = o[e][3] = 0.f;
    uint4 kh[NC], kl[NC], vh[NC], vl[NC];
    // (no condition around the loads, only around the row: it would keep a second set of the registers)
    auto load_k = [&](int k0) {
        const bf16 *kp = m.kcache + cbase + (size_t)max(min(k0 + g, w.hi - 1), 0) * HD + t * 8;
#pragma unroll
        for (int n = 0; n < NC; ++n) {
            kh[n] = __ldcg(reinterpret_cast<const uint4 *>(kp + n * 32));
            kl[n] = __ldcg(reinterpret_cast<const uint4 *>(kp + m.kv_lo + n * 32));
        }
    };
    int k0 = w.lo + c.warp * 8;
    auto load_v = [&](int k0) {
        const bf16 *vp = m.vcache + cbase + (size_t)max(min(k0 + g, w.hi - 1), 0) * HD + t * 8;
#pragma unroll
        for (int n = 0; n < NC; ++n) {
            vh[n] = __ldcg(reinterpret_cast<const uint4 *>(vp + n * 32));
            vl[n] = __ldcg(reinterpret_cast<const uint4 *>(vp + m.kv_lo + n * 32));
        }
    };
    load_k(k0);           // in flight with the query rows
    if (qi < nv * (HD / 4)) {                            // (rows past nv: stale, their sums are not read)
        uint2 hi, lo;
        split_pair(qx.x, qx.y, hi.x, lo.x); split_pair(qx.z, qx.w, hi.y, lo.y);
        *reinterpret_cast<uint2 *>(qs + qi / (HD / 4) * QS + (qi & (HD / 4 - 1)) * 8) = hi;
        *reinterpret_cast<uint2 *>(qs + qi / (HD / 4) * QS + HD * 2 + (qi & (HD / 4 - 1)) * 8) = lo;
    }
    fsync();                                             // the query rows are staged
    for (; k0 < w.hi; k0 += FW * 8) {
        load_v(k0);
        float sa[4] = {0.f, 0.f, 0.f, 0.f}, sb[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int n = 0; n < NC; ++n) {
            const uint4 qh = *reinterpret_cast<const uint4 *>(qs + g * QS + n * 64 + t * 16);
            const uint4 ql = *reinterpret_cast<const uint4 *>(qs + g * QS + HD * 2 + n * 64 + t * 16);
            mma16816(sa, qh.x, ql.x, qh.y, ql.y, kh[n].x, kh[n].y);
            mma16816(sb, qh.z, ql.z, qh.w, ql.w, kh[n].z, kh[n].w);
            mma16816(sa, qh.x, ql.x, qh.y, ql.y, kl[n].x, kl[n].y);
            mma16816(sb, qh.z, ql.z, qh.w, ql.w, kl[n].z, kl[n].w);
        }
        load_k(k0 + FW * 8);
        // scores of row g, keys 2t, 2t + 1: a row sees the keys of its context up to its own position; a row before a
        // restricted context sees itself
        float s0 = (sa[0] + sb[0]) + (sa[2] + sb[2]), s1 = (sa[1] + sb[1]) + (sa[3] + sb[3]);
        const int ka = k0 + 2 * t, kb = ka + 1;
        if (!(ka < w.hi && vrow >= 0 && ka <= self && (ka >= ks || ka == self))) s0 = -INFINITY;
        if (!(kb < w.hi && vrow >= 0 && kb <= self && (kb >= ks || kb == self))) s1 = -INFINITY;
        float mn = fmaxf(s0, s1);
        mn = fmaxf(mn, __shfl_xor_sync(0xffffffffu, mn, 1));
        mn = fmaxf(mn, __shfl_xor_sync(0xffffffffu, mn, 2));
        mn = fmaxf(mn, mx);
        const float corr = mn == -INFINITY ? 1.f : __expf(mx - mn);
        mx = mn;
        const float p0 = s0 == -INFINITY ? 0.f : __expf(s0 - mn), p1 = s1 == -INFINITY ? 0.f : __expf(s1 - mn);
        ls = ls * corr + p0 + p1;
        uint32_t ph, pl;
        split_pair(p0, p1, ph, pl);
        const float c0 = __shfl_sync(0xffffffffu, corr, 8 * t), c1 = __shfl_sync(0xffffffffu, corr, 8 * t + 4);
#pragma unroll
        for (int e = 0; e < NC * 2; ++e) { o[e][0] *= c0; o[e][1] *= c1; o[e][2] *= c0; o[e][3] *= c1; }
#pragma unroll
        for (int n = 0; n < NC; ++n) {
            uint32_t a0 = movmatrix(vh[n].x), a1 = movmatrix(vh[n].y), a2 = movmatrix(vl[n].x), a3 = movmatrix(vl[n].y);
            mma16816(o[n * 2], a0, a1, a2, a3, ph, ph);
            mma16816(o[n * 2], a0, a1, a2, a3, pl, pl);
            a0 = movmatrix(vh[n].z); a1 = movmatrix(vh[n].w); a2 = movmatrix(vl[n].z); a3 = movmatrix(vl[n].w);
            mma16816(o[n * 2 + 1], a0, a1, a2, a3, ph, ph);
            mma16816(o[n * 2 + 1], a0, a1, a2, a3, pl, pl);
        }
    }
    ls += __shfl_xor_sync(0xffffffffu, ls, 1);
    ls += __shfl_xor_sync(0xffffffffu, ls, 2);
    {
        // rows 2t, 2t + 1; channel of block i, column g: 8 (g / 2) + 2 i + g % 2
        float *my = red + (c.warp * QR + 2 * t) * PW + 8 * (g >> 1) + (g & 1);
#pragma unroll
        for (int e = 0; e < NC * 2; ++e) {
            float *p = my + (e >> 1) * 32 + (e & 1) * 4;
            p[0] = o[e][0]; p[PW] = o[e][1]; p[2] = o[e][2]; p[PW + 2] = o[e][3];
        }
        if (t == 0) { float *st = red + (c.warp * QR + g) * PW + HD; st[0] = mx; st[1] = ls; }
    }
    fsync();
    // the warps' shares -> the item's, two channels per thread
    const int unit = (w.seq * m.cfg.n_kv_heads + w.kh) * f.chunks + w.vc;
    float *part = a.fb.attf + (size_t)unit * f.nsplit * QR * PW;      // [split][QR][PW]
    for (int i = threadIdx.x; i < nv * (HD / 2); i += FC_THREADS) {
        const int lv = i / (HD / 2), ch = 2 * (i - lv * (HD / 2));
        float M = -INFINITY;
#pragma unroll
        for (int x = 0; x < FW; ++x) M = fmaxf(M, red[(x * QR + lv) * PW + HD]);
        float L = 0.f, v0 = 0.f, v1 = 0.f;
#pragma unroll
        for (int x = 0; x < FW; ++x) {
            const float *rw = red + (x * QR + lv) * PW;
            const float fc = rw[HD] == -INFINITY ? 0.f : __expf(rw[HD] - M);
            L += rw[HD + 1] * fc; v0 += rw[ch] * fc; v1 += rw[ch + 1] * fc;
        }
        const int v = w.vc * QR + lv, hq = v / w.n_r, j = v - hq * w.n_r;
        if (f.nsplit == 1) {
            few_store(d.att, c.idx_of[w.seq * a.g.rps + j], (w.kh * group + hq) * HD + ch, c.nlive, v0 / L, v1 / L);
        } else {
            float *pp = part + ((size_t)w.split * QR + lv) * PW;
            __stcg(reinterpret_cast<float2 *>(pp + ch), make_float2(v0, v1));
            if (ch == 0) __stcg(reinterpret_cast<float2 *>(pp + HD), make_float2(M, L));
        }
    }
    if (f.nsplit > 1) {
        fsync();
        if (threadIdx.x == 0) {
            int n;                                       // releases this split's partial and acquires the others'
            asm volatile("atom.acq_rel.gpu.global.add.s32 %0, [%1], 1;" : "=r"(n) : "l"(a.fb.att_cnt + unit) : "memory");
            const bool last = n == f.nsplit - 1;
            if (last) a.fb.att_cnt[unit] = 0;            // for the next layer (all splits have arrived)
            *c.flag = last;
        }
        fsync();
        if (*c.flag) {                                   // the last split to arrive merges them, in split order
            for (int i = threadIdx.x; i < nv * (HD / 2); i += FC_THREADS) {
                const int lv = i / (HD / 2), ch = 2 * (i - lv * (HD / 2));
                const float *pp = part + (size_t)lv * PW;
                float M = -INFINITY, L = 0.f, v0 = 0.f, v1 = 0.f;
                for (int s0 = 0; s0 < f.nsplit; s0 += 16) {             // sixteen splits' loads in flight
                    float2 ml[16], vv[16];
#pragma unroll
                    for (int x = 0; x < 16; ++x) {
                        const bool in = s0 + x < f.nsplit;
                        const float *sp = pp + (size_t)(in ? s0 + x : 0) * QR * PW;
                        ml[x] = __ldcg(reinterpret_cast<const float2 *>(sp + HD));
                        vv[x] = __ldcg(reinterpret_cast<const float2 *>(sp + ch));
                    }
                    float Mn = M;
#pragma unroll
                    for (int x = 0; x < 16; ++x) {
                        if (s0 + x >= f.nsplit) ml[x] = make_float2(-INFINITY, 0.f);
                        Mn = fmaxf(Mn, ml[x].x);
                    }
                    const float fo = M == -INFINITY ? 0.f : __expf(M - Mn);
                    L *= fo; v0 *= fo; v1 *= fo;
                    M = Mn;
#pragma unroll
                    for (int x = 0; x < 16; ++x) {
                        const float fc = ml[x].x == -INFINITY ? 0.f : __expf(ml[x].x - M);
                        L += ml[x].y * fc; v0 += vv[x].x * fc; v1 += vv[x].y * fc;
                    }
                }
                const int v = w.vc * QR + lv, hq = v / w.n_r, j = v - hq * w.n_r;
                few_store(d.att, c.idx_of[w.seq * a.g.rps + j], (w.kh * group + hq) * HD + ch, c.nlive, v0 / L, v1 / L);
            }
        }
    }
}

template <int HD>
__device__ __forceinline__ void few_attention(FewCtx &c, const Args &a, int layer) {
    const FewAtt f = *c.att;
    for (int it = c.cta; it < f.items; it += c.ncta) {
        const FewItem w = it == c.cta ? *c.first : few_item(c, a, f, it);
        if (it != c.cta) fsync();                        // the scratch and the flag of the item before have been read
        few_attention_item<HD>(c, a, f, w, layer);
    }
}

// End of one draft forward (Eq. 6), as tail_draft: the rows' 1/rms is the LM head's, and all warps copy the hidden rows while
// warp 0 still looks for the best logit (the arg-max, 1/rms, copy and state one after the other: 4.5 us of a 68M draft step
// and 9.5 of a 1.3B one; now 3.3 and 4.5).
__device__ __forceinline__ void few_tail_draft_rows(const FewCtx &c, const Args &a, int s) {
    const DevPtrs &d = a.d;
    const int n_in = c.n_rows[s], half = a.m.cfg.d_model >> 1;
    if (d.st[s].sched) return;                           // with prescribed windows nothing is pre-verified
    float2 *dst = reinterpret_cast<float2 *>(d.hpend + ((size_t)s * (d.block_b + 1) + d.st[s].n_pend) * (2 * half));
    for (int j = 0; j < n_in; ++j) {
        const int r = s * a.g.rps + j;
        const float inv = c.inv[c.idx_of[r]];
        const float2 *x = reinterpret_cast<const float2 *>(d.xres + (size_t)r * (2 * half));
#pragma unroll 4
        for (int i = threadIdx.x; i < half; i += FC_THREADS) {
            const float2 v = __ldcg(x + i), gn = __bfloat1622float2(reinterpret_cast<const __nv_bfloat162 *>(a.m.normf)[i]);
            dst[(size_t)j * half + i] = make_float2(v.x * inv * gn.x, v.y * inv * gn.y);
        }
    }
}
__device__ __forceinline__ void few_tail_draft(const FewCtx &c, const Args &a, int s, int pick) {      // one thread
    const DevPtrs &d = a.d;
    SeqState &st = d.st[s];
    const int n_in = c.n_rows[s], gamma = st.gamma, n_pend = st.n_pend;
    if (!st.sched) {
        for (int j = 0; j < n_in; ++j) d.hpend_e[s * (d.block_b + 1) + n_pend + j] = j == n_in - 1 ? gamma + 1 : 0;
        st.n_pend = n_pend + n_in;
    }
    d.y[(size_t)s * d.gamma_cap + gamma] = pick;
    st.gamma = gamma + 1;
    st.len_D += n_in;
    st.n_draft_fwd += 1;
}

// ------------------------------------------------------------------ the kernel

template <int MAXRT, int HD, int PASS>
__global__ void __launch_bounds__(FEW_THREADS, 1) k_few(const __grid_constant__ Args a) {
    extern __shared__ __align__(1024) unsigned char smem[];
    if (smem_u32(smem) & 1023u) {               // the swizzled weight atoms need this alignment (the same in every block)
        if (threadIdx.x == 0) atomicCAS(a.fb.abort_flag, 0, 13);
        return;
    }
    FewCtx c;
    c.warp = threadIdx.x >> 5; c.lane = threadIdx.x & 31; c.cta = blockIdx.x; c.ncta = gridDim.x;
    c.ring = smem + F_GUARD;
    unsigned char *misc = c.ring + F_SHARED;
    c.wfull = reinterpret_cast<uint64_t *>(misc);
    c.wempty = c.wfull + FNB;
    c.xfull = c.wempty + FNB;
    c.xempty = c.xfull + FXS_MANY;
    c.ready = reinterpret_cast<volatile int32_t *>(c.xempty + FXS_MANY);          // one word, and a pad
    c.slot_at = reinterpret_cast<int32_t *>(c.xempty + FXS_MANY + 1);
    FewOp *ops = reinterpret_cast<FewOp *>(c.slot_at + FNB);                 // [2][N_OPS]
    c.ops = ops;
    c.row_dst = reinterpret_cast<float **>(ops + 2 * N_OPS);
    c.row_pos = reinterpret_cast<int32_t *>(c.row_dst + FEW_ROWS);           // three tables of MAX_ROWS
    c.row_tok = c.row_pos + MAX_ROWS;
    c.idx_of = c.row_tok + MAX_ROWS;
    c.n_rows = c.idx_of + MAX_ROWS;                                          // [MAX_SEQ]
    c.key_start = c.n_rows + MAX_SEQ;                                        // [MAX_SEQ]
    c.row_of = c.key_start + MAX_SEQ;                                        // [FEW_ROWS]
    c.bias_at = c.row_of + FEW_ROWS;
    c.inv = reinterpret_cast<float *>(c.bias_at + FEW_ROWS);
    c.top = reinterpret_cast<Top2 *>(c.inv + FEW_ROWS);                      // [FEW_ROWS]
    c.best = reinterpret_cast<BestD *>(c.top + FEW_ROWS);                    // [FEW_ROWS]
    c.seed = reinterpret_cast<uint64_t *>(c.best + FEW_ROWS);                // [FEW_ROWS]
    c.draw_pos = reinterpret_cast<int32_t *>(c.seed + FEW_ROWS);             // [FEW_ROWS]
    c.flag = c.draw_pos + FEW_ROWS;                                          // 4 words: attention's last arrival, live rows
    c.pick = c.flag + 4;                                                     // [FEW_ROWS]
    c.gamma0 = c.pick + FEW_ROWS;                                            // [FEW_ROWS]
    c.att = reinterpret_cast<FewAtt *>(c.gamma0 + FEW_ROWS);
    c.first = reinterpret_cast<FewItem *>(c.att + 1);
    static_assert(8 * (2 * FNB + 2 * FXS_MANY + 1) + 4 * FNB + 2 * sizeof(FewOp) * N_OPS + 8 * FEW_ROWS + 4 * (3 * MAX_ROWS + 2 * MAX_SEQ + 5 * FEW_ROWS) +
                  (12 + 16 + 8 + 4) * FEW_ROWS + 16 + sizeof(FewAtt) + sizeof(FewItem) <= F_MISC - F_XBYTES, "tables");
    static_assert(sizeof(FewOp) * N_OPS % 8 == 0, "alignment of the pointer table");
    c.xs = reinterpret_cast<float *>(misc + F_MISC - F_XBYTES);
    c.bar_target = 0; c.ok = true; c.stage = 0; c.xstage = 0; c.pass = 0;
    const DevPtrs &d = a.d;
    const ModelDev &m = a.m;
    const Geom &g = a.g;
    const int kind = a.kind;

    // rows of this forward, from the sequence state
    if (threadIdx.x < MAX_ROWS) {
        const int r = threadIdx.x;
        int pos = -1, tok = 0;
        if (r < g.rtot) {
            const RowDesc rd = row_desc(kind, d, r / g.rps, r % g.rps, a.aux);
            if (rd.active) { pos = rd.pos; tok = rd.tok; }
        }
        c.row_pos[r] = pos; c.row_tok[r] = tok;
    }
    if (threadIdx.x == MAX_ROWS) c.flag[2] = *(volatile int32_t *)a.fb.abort_flag;
    if (threadIdx.x == FC_THREADS) {
        for (int i = 0; i < FNB; ++i) { mbar_init(c.wfull + i, 1); mbar_init(c.wempty + i, 2); }
        for (int i = 0; i < FXS_MANY; ++i) { mbar_init(c.xfull + i, 1); mbar_init(c.xempty + i, FW); }
        *c.ready = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        fence_proxy_async();
    }
    __syncthreads();
    if (c.warp == 0) {                          // the live rows, packed
        int n = 0;
        for (int r0 = 0; r0 < g.rtot; r0 += 32) {
            const int r = r0 + c.lane;
            const bool on = r < g.rtot && c.row_pos[r] >= 0;
            const uint32_t mask = __ballot_sync(0xffffffffu, on);
            const int i = n + __popc(mask & ((1u << c.lane) - 1u));
            if (on && i < FEW_ROWS) c.row_of[i] = r;
            if (r < g.rtot) c.idx_of[r] = i;
            n += __popc(mask);
        }
        // (after a wait that gave up nothing is computed: what the forward would read is not complete)
        if (c.lane == 0) c.flag[1] = c.flag[2] != 0 ? -1 : n;
    } else if (c.warp == 1) {
        const int s = c.lane;
        int n = 0, ks = 0;
        if (s < g.batch) {
            for (int j = 0; j < g.rps; ++j) n += c.row_pos[s * g.rps + j] >= 0;
            if (kind == KIND_MB && d.mb_scope != 0 && n > 0) {
                int n_hist = 0;
                while (n_hist < n && c.row_tok[s * g.rps + n_hist] == 0) ++n_hist;
                const int first = c.row_pos[s * g.rps] + n_hist;
                ks = (d.mb_scope == 2 || d.st[s].gamma == d.block_b) ? first : d.st[s].mb_start;
            }
        }
        c.n_rows[s] = n;
        c.key_start[s] = ks;
        const uint32_t on = __ballot_sync(0xffffffffu, n > 0);
        if (s == 0) c.flag[0] = __popc(on);
        if (s < FEW_ROWS) c.gamma0[s] = s < g.batch ? d.st[s].gamma : 0;
    }
    __syncthreads();
    c.nlive = c.flag[1]; c.nlater = c.flag[0];
    if (c.nlive <= 0 || c.nlive > FEW_ROWS) {   // nothing to do, or k_forward's work: the same decision in every block
        if (c.nlive == 0 && c.cta == 0 && threadIdx.x < g.batch) d.n_rows[threadIdx.x] = 0;
        return;
    }
    c.xk = F_XROWS / c.nlive;
    // (in a launch of several forwards the later ones have at most eight rows)
    c.many = MAXRT == 2 && PASS > FEW_SHORT && a.n_fwd == 1 && few_many(c.nlive, m.cfg.d_model);
    c.scratch = c.ring + few_ring(c.many);
    if (threadIdx.x < 2 * N_OPS) {
        const int o = threadIdx.x % N_OPS;
        ops[threadIdx.x] = few_op<PASS>(a.P.op[o], o, c.cta, c.ncta, threadIdx.x < N_OPS ? c.nlive : c.nlater, c.many);
    }
    if (threadIdx.x == 32) {
        const unsigned long long v = ld_acquire_u64(a.fb.bar);
        c.bar_target = v / (unsigned long long)c.ncta * (unsigned long long)c.ncta;
        *reinterpret_cast<unsigned long long *>(c.flag + 2) = c.bar_target;
    }
    __syncthreads();
    c.bar_target = *reinterpret_cast<unsigned long long *>(c.flag + 2);

    if (c.warp == FW) {
        few_weight_producer(c, a.fb, a.P, a.n_fwd, few_ring(c.many), policy_evict_first());
        return;
    }
    if (c.warp == FW + 1) {
        uint64_t keep;
        asm volatile("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(keep));
        if (c.many) few_x_producer<FXS_MANY>(c, a, keep);
        else few_x_producer<FXS>(c, a, keep);
        return;
    }
    if (c.cta == 0 && threadIdx.x < MAX_ROWS) {
        const int r = threadIdx.x;
        if (r < g.batch) d.n_rows[r] = c.n_rows[r];
        if (r < g.rtot) { d.row_pos[r] = c.row_pos[r]; d.row_tok[r] = c.row_tok[r]; }
    }

    int n_stamp = 0;
    auto stamp = [&]() {
        if (a.fb.prof && threadIdx.x == 0 && n_stamp < PROF_STAMPS)
            a.fb.prof[(size_t)c.cta * PROF_STAMPS + n_stamp++] = globaltimer_ns();
    };
    const int nq = n_ops(a.P);
    c.x0 = ops[OP_O].r0; c.xc = ops[OP_O].r1 - ops[OP_O].r0;
    for (int f = 0;;) {                         // the forwards of the launch
        if (threadIdx.x < c.nlive) {                // where the LM-head rows go (read after the barriers of the layers)
            const int i = threadIdx.x, r = c.row_of[i], s = r / g.rps, j = r - s * g.rps, V = m.cfg.vocab;
            float *dst = nullptr;
            int b = -1;
            if (a.P.has_head) {
                if (kind == KIND_DRAFT) {
                    if (j == c.n_rows[s] - 1) dst = d.draft_logits + ((size_t)s * d.gamma_cap + c.gamma0[s] + f) * V;
                } else {
                    dst = d.verify_logits + ((size_t)s * (d.gamma_cap + 1) + j) * V;
                }
                if (m.succ) b = m.succ[c.row_tok[r]];
            }
            c.row_dst[i] = dst; c.bias_at[i] = b;
            const SeqState &st = d.st[s];
            c.draw_pos[i] = dst && st.mode == PACER_SAMPLE && kind != KIND_VERIFY ? c.row_pos[r] + 1 : -1;     // the token behind the row
            c.seed[i] = st.seed;
            c.best[i] = BestD{-INFINITY, 0x7fffffff};
            c.top[i] = Top2{-INFINITY, 0x7fffffff, -INFINITY};
        }
        stamp();
        // input rows: this block's columns of the residual stream, like a residual epilogue
        for (int i = c.warp; i < c.nlive; i += FW) {
            const int r = c.row_of[i];
            float s = 0.f;
            for (int k = 2 * c.lane; k < c.xc; k += 64) {
                const float2 v = few_input(a, c, r, c.x0 + k);
                const __nv_bfloat162 gn = *reinterpret_cast<const __nv_bfloat162 *>(m.norm1 + c.x0 + k);
                s += v.x * v.x + v.y * v.y;
                c.xs[i * c.xc + k] = v.x; c.xs[i * c.xc + k + 1] = v.y;
                few_store(a.fb.xg, i, c.x0 + k, c.nlive, v.x * __low2float(gn), v.y * __high2float(gn));
            }
            s = warp_sum(s);
            if (c.lane == 0) a.fb.ssq[i * c.ncta + c.cta] = s;
        }
        stamp();
        few_grid_barrier(c, a.fb);
        stamp();
        if (threadIdx.x == 0) {
            const FewAtt f = few_att(c, a);
            *c.att = f;
            *c.first = few_item(c, a, f, min(c.cta, f.items - 1));
        }
        fsync();
        for (int q = 0; q < nq; ++q) {
            const int opi = op_index(a.P, q), l = op_layer(a.P, q);
            // opaque in every round: what the compiler could compute from these once for all rounds it would keep in registers
            // that the projections need (68M draft step 90.7 -> 86.5 us, 7B forward of 5 rows 742 -> 727)
            asm volatile("" : "+r"(c.lane), "+r"(c.warp), "+r"(c.nlive), "+r"(c.cta), "+r"(c.ncta), "+r"(c.xk));
            if (opi == OP_QKV && c.warp == FW - 1 && c.cta < c.att->items) few_kv_prefetch(c, a, *c.first, l);
            few_gemm<MAXRT, PASS>(c, a, opi, l);
            stamp();
            few_grid_barrier(c, a.fb);
            stamp();
            if (opi == OP_QKV) {
                few_attention<HD>(c, a, l);
                stamp();
                few_grid_barrier(c, a.fb);
                stamp();
            }
        }
        // Arg-max (lowest index on ties) and gap, a row per warp: the block of a sequence for its rows and, where another forward
        // follows, every block for all of them, so that the next token needs no barrier of its own.
        const bool more = f + 1 < a.n_fwd;
        if (a.P.has_head && (more || c.cta < g.batch)) {
            for (int i = c.warp; i < c.nlive; i += FW) {
                const int r = c.row_of[i], s = r / g.rps;
                const bool own = s == c.cta;
                if (!c.row_dst[i] || !(more || own)) continue;
                Top2 tp{-INFINITY, 0x7fffffff, -INFINITY};
                for (int b = c.lane; b < c.ncta; b += 32) {
                    const float4 v = __ldcg(reinterpret_cast<const float4 *>(a.fb.tile_top) + (size_t)b * FEW_ROWS + i);
                    tp = top2_merge(tp, Top2{v.x, __float_as_int(v.y), v.z});
                }
                tp = few_warp_top2(tp);
                if (c.lane == 0) {
                    const int best = in_vocab(tp.i1, m.cfg.vocab);
                    if (own) { d.row_arg[r] = best; d.row_margin[r] = tp.v1 - tp.v2; }
                    if (kind != KIND_VERIFY && c.draw_pos[i] < 0) c.pick[s] = best;
                }
                if (c.draw_pos[i] >= 0) {           // (one row of the sequence at most)
                    BestD bd{-INFINITY, 0x7fffffff};
                    for (int b = c.lane; b < c.ncta; b += 32) {
                        const BestD *p = few_best(a, c) + (size_t)b * FEW_ROWS + i;
                        bd = best_merge(bd, BestD{__ldcg(&p->v), __ldcg(&p->i)});
                    }
                    bd = few_warp_best(bd);
                    if (c.lane == 0) c.pick[s] = drawn_token(bd, m.cfg.vocab);
                }
            }
            if (kind == KIND_DRAFT && c.cta < g.batch) few_tail_draft_rows(c, a, c.cta);
            fsync();
            if (c.cta < g.batch && threadIdx.x == 0) {
                if (kind == KIND_DRAFT && c.n_rows[c.cta] > 0) few_tail_draft(c, a, c.cta, c.pick[c.cta]);
                if (kind == KIND_VERIFY && a.aux) accept_greedy_seq(d, g, c.cta);
            }
        }
        if (!more) break;
        // the next forward: one row per sequence, the token just chosen behind the last row
        fsync();
        if (threadIdx.x == 0) {
            int n = 0;
            for (int s = 0; s < g.batch; ++s) {
                const int n_r = c.n_rows[s], r = s * g.rps;
                if (n_r == 0) continue;
                c.row_pos[r] += n_r; c.row_tok[r] = c.pick[s];
                c.n_rows[s] = 1; c.idx_of[r] = n; c.row_of[n] = r;
                ++n;
            }
        }
        c.nlive = c.nlater; c.xk = F_XROWS / c.nlive; c.ops = ops + N_OPS;
        ++f;
        fsync();
    }
    if (c.cta < g.batch && (kind == KIND_MB || kind == KIND_AR) && c.warp < MMA_WARPS) {
        Ctx t;                                  // what the tails look at
        t.warp = c.warp; t.lane = c.lane; t.cta = c.cta; t.ncta = c.ncta;
        t.scratch = c.scratch; t.n_rows = c.n_rows; t.row_tok = c.row_tok; t.row_pos = c.row_pos;
        t.inv_rms = reinterpret_cast<float *>(c.scratch) + 1024;             // [MAX_ROWS], beside what the tails use
        if (kind == KIND_MB) tail_mb(t, a, t.cta);
        else tail_ar(t, a, t.cta, c.pick[t.cta]);
    }
    stamp();
}

template <int MAXRT, int HD, int PASS>
static cudaError_t launch_few_variant(const Args &a, int ncta, cudaStream_t st) {
    static bool attr_set[64] = {};           // the opt-in is per device
    constexpr int smem = F_GUARD + F_SHARED + F_MISC;
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= 64 || !attr_set[dev]) {
        e = cudaFuncSetAttribute(k_few<MAXRT, HD, PASS>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
        if (e != cudaSuccess) return e;
        if (dev >= 0 && dev < 64) attr_set[dev] = true;
    }
    void *params[] = {(void *)&a};
    return cudaLaunchCooperativeKernel((const void *)k_few<MAXRT, HD, PASS>, dim3(ncta), dim3(FEW_THREADS), params, smem, st);
}

}  // namespace fwd
