// The tiled kernel in FP32 storage.
#include "lb_tiled.cuh"

namespace lbhb {

template const void* tiled_kernel<float>(int tx, bool sample, int fam);

}  // namespace lbhb
