// The y passes of one cell in FP64.
#include "mp_lines.cuh"

namespace mp {

MP_INSTANTIATE_LINE(double, kYForward)
MP_INSTANTIATE_LINE(double, kYInverse)

}  // namespace mp
