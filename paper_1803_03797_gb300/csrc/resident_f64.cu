// resident_f64.cu -- chip-resident kernels: binary64 Algorithm 1.
#include "resident_kernels.cuh"

namespace lap5 {

LAP5_RESIDENT_KERNELS(f64, RK_F64_CLASSIC)

}  // namespace lap5
