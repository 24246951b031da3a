// The direct path's kernels of one family: GBG_PARTS BF16 parts (2 or 3) and
// GBG_MODE_A, the LoadMode of op(A); every mode of op(B) and tile shape.
#include "direct_kernel.cuh"

namespace gbg {
template cudaError_t launch_direct_mode<GBG_PARTS, GBG_MODE_A>(const DirectPlan&, int, const DirectArgs&, int64_t,
                                                               cudaStream_t);
template bool direct_mode_fits<GBG_PARTS, GBG_MODE_A>(const DirectPlan&, int);
}  // namespace gbg
