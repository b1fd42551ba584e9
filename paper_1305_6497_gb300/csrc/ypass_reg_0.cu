// Instances of the register y passes (ypass_reg.cuh), part 0.
#include "ypass_reg.cuh"

namespace dda {
DDA_YREG_DEFINE(0)
}  // namespace dda
