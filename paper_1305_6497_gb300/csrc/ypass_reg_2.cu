// Instances of the register y passes (ypass_reg.cuh), part 2.
#include "ypass_reg.cuh"

namespace dda {
DDA_YREG_DEFINE(2, DDA_REG_NONE)
}  // namespace dda
