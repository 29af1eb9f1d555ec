// The forward kernel for groups of 6 eight-row tiles.
#define FWD_INSTANTIATE
#include "fwd_kernel.cuh"

namespace fwd {

FWD_VARIANT(6, false, true);

}  // namespace fwd
