// Instances of the register x passes (xpass_reg.cuh), part 6.
#include "xpass_reg.cuh"

namespace dda {
DDA_XREG_DEFINE(6)
}  // namespace dda
