// Instances of the FP64 and double-float register z pass (zpass_wide.cuh), part 4.
#include "zpass_wide.cuh"

namespace dda {
DDA_ZWIDE_DEFINE(4)
}  // namespace dda
