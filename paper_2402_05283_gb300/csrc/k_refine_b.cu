// k_refine_b.cu - instances of the line passes over volumes, N = 160, 192, 256.
#include "refine_kernels.cuh"

namespace cpra {

CPRA_REFINE_INSTANCES(160, )
CPRA_REFINE_INSTANCES(192, )
CPRA_REFINE_INSTANCES(256, )

}  // namespace cpra
