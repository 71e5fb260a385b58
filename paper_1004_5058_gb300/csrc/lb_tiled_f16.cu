// The tiled kernel in FP16-shifted storage.
#include "lb_tiled.cuh"

namespace lbhb {

template const void* tiled_kernel<__half>(int tx, bool sample, int fam);

}  // namespace lbhb
