// k_assemble_a.cu - instances of the assembly kernels, N = 16, 32, 48, 64, 96, 128.
#include "assemble_kernels.cuh"

namespace cpra {

CPRA_ASSEMBLE_INSTANCES(16, )
CPRA_ASSEMBLE_INSTANCES(32, )
CPRA_ASSEMBLE_INSTANCES(48, )
CPRA_ASSEMBLE_INSTANCES(64, )
CPRA_ASSEMBLE_INSTANCES(96, )
CPRA_ASSEMBLE_INSTANCES(128, )

}  // namespace cpra
