// The tiled kernel in stochastically rounded FP16 storage.
#include "lb_tiled.cuh"

namespace lbhb {

template const void* tiled_kernel<half_sr>(int tx, bool sample, int fam);

}  // namespace lbhb
