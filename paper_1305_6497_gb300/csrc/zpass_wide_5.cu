// Instances of the FP64 and double-float register z pass (zpass_wide.cuh), part 5.
#include "zpass_wide.cuh"

namespace dda {
DDA_ZWIDE_DEFINE(5)
}  // namespace dda
