// The z pass with the Green operator of one cell in FP64.
#include "mp_lines.cuh"

namespace mp {

MP_INSTANTIATE_LINE(double, kZReduced)

}  // namespace mp
