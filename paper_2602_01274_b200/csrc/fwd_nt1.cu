// The forward kernel for 1 eight-row tile.
#define FWD_INSTANTIATE
#include "fwd_kernel.cuh"

namespace fwd {

FWD_VARIANT(1, false, false);
FWD_VARIANT(1, true, false);

}  // namespace fwd
