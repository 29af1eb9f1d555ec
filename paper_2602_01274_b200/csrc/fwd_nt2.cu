// The forward kernel for 2 eight-row tiles.
#define FWD_INSTANTIATE
#include "fwd_kernel.cuh"

namespace fwd {

FWD_VARIANT(2, false, false);
FWD_VARIANT(2, true, false);

}  // namespace fwd
