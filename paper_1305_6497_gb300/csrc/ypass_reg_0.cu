// Instances of the register y passes (ypass_reg.cuh), part 0 and odd lengths.
#include "ypass_reg.cuh"

namespace dda {
DDA_YREG_DEFINE(0, DDA_XREG_ODD)
}  // namespace dda
