// Instances of the register x passes (xpass_reg.cuh), part 3.
#include "xpass_reg.cuh"

namespace dda {
DDA_XREG_DEFINE(3, DDA_XREG_PART3, )
}  // namespace dda
