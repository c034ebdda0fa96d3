// The y passes of several cells in FP64.
#include "mp_lines.cuh"

namespace mp {

MP_INSTANTIATE_LINE_MULTI(double, kYForward)
MP_INSTANTIATE_LINE_MULTI(double, kYInverse)

}  // namespace mp
