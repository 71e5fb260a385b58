// The tiled kernel in FP64 storage.
#include "lb_tiled.cuh"

namespace lbhb {

template const void* tiled_kernel<double>(int tx, bool sample, int fam);

}  // namespace lbhb
