// Instances of the register x passes (xpass_reg.cuh), part 2.
#include "xpass_reg.cuh"

namespace dda {
DDA_XREG_DEFINE(2, DDA_XREG_PART2, )
}  // namespace dda
