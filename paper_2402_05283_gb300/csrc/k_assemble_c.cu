// k_assemble_c.cu - instances of the assembly kernels, N = 384, 512, 640.
#include "assemble_kernels.cuh"

namespace cpra {

CPRA_ASSEMBLE_INSTANCES(384, )
CPRA_ASSEMBLE_INSTANCES(512, )
CPRA_ASSEMBLE_INSTANCES(640, )

}  // namespace cpra
