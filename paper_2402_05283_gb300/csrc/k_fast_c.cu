// k_fast_c.cu - FP32 instances of the warp-FFT engine kernels, N = 512, 640, 700, 768, 1024.
#include "fast_kernels.cuh"

namespace cpra {

CPRA_WARP_INSTANCES(512, )
CPRA_WARP_INSTANCES(640, )
CPRA_WARP_INSTANCES(700, )
CPRA_WARP_INSTANCES(768, )
CPRA_WARP_INSTANCES(1024, )

}  // namespace cpra
