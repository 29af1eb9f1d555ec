// The forward kernel for 3 eight-row tiles.
#define FWD_INSTANTIATE
#include "fwd_kernel.cuh"

namespace fwd {

FWD_VARIANT(3, false, false);
FWD_VARIANT(3, true, false);

}  // namespace fwd
