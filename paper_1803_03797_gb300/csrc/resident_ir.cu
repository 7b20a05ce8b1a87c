// resident_ir.cu -- chip-resident kernels: mixed precision.
#include "resident_kernels.cuh"

namespace lap5 {

LAP5_RESIDENT_KERNELS(ir, RK_IR_F32)

}  // namespace lap5
