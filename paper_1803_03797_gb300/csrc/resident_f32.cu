// resident_f32.cu -- chip-resident kernels: binary32 Algorithm 1.
#include "resident_kernels.cuh"

namespace lap5 {

LAP5_RESIDENT_KERNELS(f32, RK_F32_CLASSIC)

}  // namespace lap5
