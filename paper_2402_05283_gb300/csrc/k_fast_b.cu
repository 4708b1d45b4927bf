// k_fast_b.cu - FP32 instances of the warp-FFT engine kernels, N = 192, 256, 320, 384.
#include "fast_kernels.cuh"

namespace cpra {

CPRA_WARP_INSTANCES(192, )
CPRA_WARP_INSTANCES(256, )
CPRA_WARP_INSTANCES(320, )
CPRA_WARP_INSTANCES(384, )

}  // namespace cpra
