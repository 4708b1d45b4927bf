// k_assemble_b.cu - instances of the assembly kernels, N = 160, 192, 256, 320.
#include "assemble_kernels.cuh"

namespace cpra {

CPRA_ASSEMBLE_INSTANCES(160, )
CPRA_ASSEMBLE_INSTANCES(192, )
CPRA_ASSEMBLE_INSTANCES(256, )
CPRA_ASSEMBLE_INSTANCES(320, )

}  // namespace cpra
