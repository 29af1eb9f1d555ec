// Host side of the few-row kernel: which variant a forward takes.
#include "fwd_few.h"

namespace fwd {

cudaError_t launch_few_narrow8(const Args &a, int ncta, cudaStream_t st);
cudaError_t launch_few_narrow16(const Args &a, int ncta, cudaStream_t st);
cudaError_t launch_few_wide8(const Args &a, int ncta, cudaStream_t st);
cudaError_t launch_few_wide16(const Args &a, int ncta, cudaStream_t st);

bool few_rows_ok(const ModelDev &m, const Geom &g, int kind, int ncta) {
    if (g.batch > FEW_ROWS || (kind != KIND_DRAFT && kind != KIND_VERIFY && kind != KIND_AR && kind != KIND_MB)) return false;
    const int xc = 2 * ((m.cfg.d_model / 2 + ncta - 1) / ncta);
    return FEW_ROWS * xc * 4 <= FEW_XBYTES && xc + 16 <= 8 * 12;       // (a pass of twelve atoms: nine and more rows)
}

// Draft steps and pre-verification calls take the variant with short passes, the target's forwards the one with long passes.
// A pass of up to 24 atoms keeps a projection of a wide model in one or two passes, but its accumulators leave the kernel short of
// registers (52 to 80 bytes spilled, none with 16), and a spill in a phase of 3 us is seen: step of the tiny pair with short
// passes everywhere 414 us, with 24 atoms everywhere 429; one token of the 1.5B / 32B pair's target (4 layers) 972 and 909.
// Where no more than eight rows can be live the code for sixteen is left out (the instruction cache misses less).
cudaError_t launch_few(const Args &a, int ncta, cudaStream_t st) {
    if (a.kind == KIND_DRAFT || a.kind == KIND_MB) return a.g.rtot <= 8 ? launch_few_narrow8(a, ncta, st) : launch_few_narrow16(a, ncta, st);
    return a.g.rtot <= 8 ? launch_few_wide8(a, ncta, st) : launch_few_wide16(a, ncta, st);
}

}  // namespace fwd
