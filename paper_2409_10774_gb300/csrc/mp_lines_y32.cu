// The y passes in FP32.
#include "mp_lines.cuh"

namespace mp {

MP_INSTANTIATE_LINES(float, kYForward)
MP_INSTANTIATE_LINES(float, kYInverse)

}  // namespace mp
