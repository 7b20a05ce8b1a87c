// resident_newcg.cu -- chip-resident kernels: binary64 Algorithm 2.
#include "resident_kernels.cuh"

namespace lap5 {

LAP5_RESIDENT_KERNELS(newcg, RK_F64_NEWCG)

}  // namespace lap5
