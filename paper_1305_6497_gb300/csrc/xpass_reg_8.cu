// Instances of the register x passes (xpass_reg.cuh), odd lengths.
#include "xpass_reg.cuh"

namespace dda {
DDA_XREG_DEFINE(8, DDA_XREG_ODD, _ODD)
}  // namespace dda
