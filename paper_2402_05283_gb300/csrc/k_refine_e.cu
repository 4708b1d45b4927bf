// k_refine_e.cu - instances of the line passes over volumes, N = 768, 1024.
#include "refine_kernels.cuh"

namespace cpra {

CPRA_REFINE_INSTANCES(768, )
CPRA_REFINE_INSTANCES(1024, )

}  // namespace cpra
