// k_refine_c.cu - instances of the line passes over volumes, N = 320, 384, 512.
#include "refine_kernels.cuh"

namespace cpra {

CPRA_REFINE_INSTANCES(320, )
CPRA_REFINE_INSTANCES(384, )
CPRA_REFINE_INSTANCES(512, )

}  // namespace cpra
