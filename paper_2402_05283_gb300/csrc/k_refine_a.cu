// k_refine_a.cu - instances of the line passes over volumes, N = 16, 32, 48, 64, 96, 128.
#include "refine_kernels.cuh"

namespace cpra {

CPRA_REFINE_INSTANCES(16, )
CPRA_REFINE_INSTANCES(32, )
CPRA_REFINE_INSTANCES(48, )
CPRA_REFINE_INSTANCES(64, )
CPRA_REFINE_INSTANCES(96, )
CPRA_REFINE_INSTANCES(128, )

}  // namespace cpra
