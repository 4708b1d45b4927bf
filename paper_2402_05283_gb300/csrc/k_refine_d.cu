// k_refine_d.cu - instances of the line passes over volumes, N = 640, 700.
#include "refine_kernels.cuh"

namespace cpra {

CPRA_REFINE_INSTANCES(640, )
CPRA_REFINE_INSTANCES(700, )

}  // namespace cpra
