// Instances of the register x passes (xpass_reg.cuh), part 7.
#include "xpass_reg.cuh"

namespace dda {
DDA_XREG_DEFINE(7, DDA_XREG_PART7, )
}  // namespace dda
