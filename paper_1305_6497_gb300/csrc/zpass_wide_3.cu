// Instances of the FP64 and double-float register z pass (zpass_wide.cuh), part 3.
#include "zpass_wide.cuh"

namespace dda {
DDA_ZWIDE_DEFINE(3)
}  // namespace dda
