// The y passes of several cells in FP32.
#include "mp_lines.cuh"

namespace mp {

MP_INSTANTIATE_LINE_MULTI(float, kYForward)
MP_INSTANTIATE_LINE_MULTI(float, kYInverse)

}  // namespace mp
