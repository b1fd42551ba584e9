// Instances of the two-step register z pass (zpass_reg.cuh), part 5.
#include "zpass_reg.cuh"

namespace dda {
DDA_ZREG_DEFINE(5, DDA_REG_NONE)
}  // namespace dda
