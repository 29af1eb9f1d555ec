// The forward kernel for groups of 8 eight-row tiles.
#define FWD_INSTANTIATE
#include "fwd_kernel.cuh"

namespace fwd {

FWD_VARIANT(8, false, true);

}  // namespace fwd
