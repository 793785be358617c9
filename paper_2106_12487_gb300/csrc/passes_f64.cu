// Mixed-radix passes, FP64 fields.
#include "passes_launch.cuh"

namespace bloch {
BLOCH_INST_PASSES_Z(double)
BLOCH_INST_PASSES_AXIS(double)
BLOCH_INST_PASSES_X(double)
template void pass_x<double>(bloch_plan*, int, int, cplx_t<double>*, double, const double2*, int);
}  // namespace bloch
