// Host side of the few-row kernel: which variant a forward takes.
#include "fwd_few.h"

#include "few_plan.h"

namespace fwd {

cudaError_t launch_few_narrow8(const Args &a, int ncta, cudaStream_t st);
cudaError_t launch_few_narrow16(const Args &a, int ncta, cudaStream_t st);
cudaError_t launch_few_wide8(const Args &a, int ncta, cudaStream_t st);
cudaError_t launch_few_wide16(const Args &a, int ncta, cudaStream_t st);
cudaError_t launch_few_wider8(const Args &a, int ncta, cudaStream_t st);
cudaError_t launch_few_wider16(const Args &a, int ncta, cudaStream_t st);

bool few_rows_ok(const ModelDev &m, const Geom &g, int kind, int ncta) {
    if (g.batch > FEW_ROWS || (kind != KIND_DRAFT && kind != KIND_VERIFY && kind != KIND_AR && kind != KIND_MB)) return false;
    // this block's columns of the residual stream: in shared memory, and (the two residual projections) in one pass, the shortest
    // being twelve atoms
    static_assert(FEW_XBYTES / (FEW_ROWS * 4) + 16 <= 8 * 12, "a residual projection in one pass");
    const int xc = 2 * ((m.cfg.d_model / 2 + ncta - 1) / ncta);
    return FEW_ROWS * xc * 4 <= FEW_XBYTES;
}

// How long a pass: few_plan.h.  The target's forwards of windows that may have nine and more live rows take long passes whatever
// their size: these variants have five activation stages for such rows (see fwd_few.cuh).
// Where no more than eight rows can be live the code for sixteen is left out (the instruction cache misses less).
cudaError_t launch_few(const Args &a, int ncta, cudaStream_t st) {
    const pacer_model_cfg &k = a.m.cfg;
    const int pass = few_pass_atoms(k.n_layers, a.m.qrows, 2 * k.d_ffn, a.P.has_head ? k.vocab : 0, ncta);
    const bool eight = a.g.rtot <= 8;
    if (pass == FEW_LONGER) return eight ? launch_few_wider8(a, ncta, st) : launch_few_wider16(a, ncta, st);
    if (pass == FEW_LONG || (!eight && (a.kind == KIND_VERIFY || a.kind == KIND_AR)))
        return eight ? launch_few_wide8(a, ncta, st) : launch_few_wide16(a, ncta, st);
    return eight ? launch_few_narrow8(a, ncta, st) : launch_few_narrow16(a, ncta, st);
}

}  // namespace fwd
