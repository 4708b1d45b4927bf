// k_fast_a.cu - FP32 instances of the warp-FFT engine kernels, N = 16, 32, 48, 64, 96, 128, 160.
#include "fast_kernels.cuh"

namespace cpra {

CPRA_WARP_INSTANCES(16, )
CPRA_WARP_INSTANCES(32, )
CPRA_WARP_INSTANCES(48, )
CPRA_WARP_INSTANCES(64, )
CPRA_WARP_INSTANCES(96, )
CPRA_WARP_INSTANCES(128, )
CPRA_WARP_INSTANCES(160, )

}  // namespace cpra
