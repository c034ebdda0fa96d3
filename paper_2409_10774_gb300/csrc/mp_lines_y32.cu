// The y passes of one cell in FP32.
#include "mp_lines.cuh"

namespace mp {

MP_INSTANTIATE_LINE(float, kYForward)
MP_INSTANTIATE_LINE(float, kYInverse)

}  // namespace mp
