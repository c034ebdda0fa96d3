// The z passes with the Green operator in FP64.
#include "mp_lines.cuh"

namespace mp {

MP_INSTANTIATE_LINES(double, kZReduced)
MP_INSTANTIATE_LINES(double, kZFull)

}  // namespace mp
