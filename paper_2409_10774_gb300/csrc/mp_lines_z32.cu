// The z passes with the Green operator in FP32.
#include "mp_lines.cuh"

namespace mp {

MP_INSTANTIATE_LINES(float, kZReduced)
MP_INSTANTIATE_LINES(float, kZFull)

}  // namespace mp
