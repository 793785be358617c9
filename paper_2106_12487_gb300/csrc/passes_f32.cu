// Mixed-radix passes, FP32 fields.
#include "passes_launch.cuh"

namespace bloch {
BLOCH_INST_PASSES_Z(float)
BLOCH_INST_PASSES_AXIS(float)
BLOCH_INST_PASSES_X(float)
template void pass_x<float>(bloch_plan*, int, int, cplx_t<float>*, float, const double2*, int);
}  // namespace bloch
