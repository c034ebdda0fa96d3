// The y passes in FP64.
#include "mp_lines.cuh"

namespace mp {

MP_INSTANTIATE_LINES(double, kYForward)
MP_INSTANTIATE_LINES(double, kYInverse)

}  // namespace mp
