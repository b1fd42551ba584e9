// Instances of the register x passes (xpass_reg.cuh), part 6.
#include "xpass_reg.cuh"

namespace dda {
DDA_XREG_DEFINE(6, DDA_XREG_PART6, )
}  // namespace dda
