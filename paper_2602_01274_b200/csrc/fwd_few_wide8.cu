// k_few for at most 8 live rows, long passes (see few_plan.h), a translation unit of its own like every variant.
#include "fwd_few.cuh"

namespace fwd {
cudaError_t launch_few_wide8(const Args &a, int ncta, cudaStream_t st) {
    return a.m.hd == 64 ? launch_few_variant<1, 64, FEW_LONG>(a, ncta, st) : launch_few_variant<1, 128, FEW_LONG>(a, ncta, st);
}
}  // namespace fwd
