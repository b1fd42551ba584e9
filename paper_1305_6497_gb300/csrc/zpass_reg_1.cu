// Instances of the two-step register z pass (zpass_reg.cuh), part 1 and odd lengths.
#include "zpass_reg.cuh"

namespace dda {
DDA_ZREG_DEFINE(1, DDA_XREG_ODD)
}  // namespace dda
