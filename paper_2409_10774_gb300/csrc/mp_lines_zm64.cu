// The z pass with the Green operator of several cells in FP64.
#include "mp_lines.cuh"

namespace mp {

MP_INSTANTIATE_LINE_MULTI(double, kZReduced)

}  // namespace mp
