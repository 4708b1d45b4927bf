// k_assemble_d.cu - instances of the assembly kernels, N = 700, 768, 1024.
#include "assemble_kernels.cuh"

namespace cpra {

CPRA_ASSEMBLE_INSTANCES(700, )
CPRA_ASSEMBLE_INSTANCES(768, )
CPRA_ASSEMBLE_INSTANCES(1024, )

}  // namespace cpra
