// Instances of the FP64 and double-float register z pass (zpass_wide.cuh), part 1.
#include "zpass_wide.cuh"

namespace dda {
DDA_ZWIDE_DEFINE(1)
}  // namespace dda
