// Instances of the register y passes (ypass_reg.cuh), part 3.
#include "ypass_reg.cuh"

namespace dda {
DDA_YREG_DEFINE(3, DDA_REG_NONE)
}  // namespace dda
