// Instances of the register x passes (xpass_reg.cuh), part 4.
#include "xpass_reg.cuh"

namespace dda {
DDA_XREG_DEFINE(4, DDA_XREG_PART4, )
}  // namespace dda
