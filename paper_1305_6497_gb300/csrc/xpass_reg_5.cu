// Instances of the register x passes (xpass_reg.cuh), part 5.
#include "xpass_reg.cuh"

namespace dda {
DDA_XREG_DEFINE(5, DDA_XREG_PART5, )
}  // namespace dda
