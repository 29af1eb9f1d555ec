// The forward kernel for 4 eight-row tiles.
#define FWD_INSTANTIATE
#include "fwd_kernel.cuh"

namespace fwd {

FWD_VARIANT(4, false, false);
FWD_VARIANT(4, true, false);

}  // namespace fwd
