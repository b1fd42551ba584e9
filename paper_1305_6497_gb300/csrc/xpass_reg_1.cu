// Instances of the register x passes (xpass_reg.cuh), part 1.
#include "xpass_reg.cuh"

namespace dda {
DDA_XREG_DEFINE(1, DDA_XREG_PART1, )
}  // namespace dda
