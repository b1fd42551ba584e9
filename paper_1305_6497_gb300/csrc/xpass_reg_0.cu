// Instances of the register x passes (xpass_reg.cuh), part 0.
#include "xpass_reg.cuh"

namespace dda {
DDA_XREG_DEFINE(0, DDA_XREG_PART0, )
}  // namespace dda
