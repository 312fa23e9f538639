// spots_split_ff.cu -- the warp-per-pixel kernels with double-float unit
// geometry, for shots of up to kFfUnits units per pixel (split_unit).
#include "split_kernel.cuh"

namespace nbgb {

template SplitKernel pick_split<true>(const SpotArgs &);

}  // namespace nbgb
