// The z pass with the Green operator of one cell in FP32.
#include "mp_lines.cuh"

namespace mp {

MP_INSTANTIATE_LINE(float, kZReduced)

}  // namespace mp
