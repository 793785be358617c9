// Mixed-radix passes, float-float fields, x passes.
#include "passes_launch.cuh"

namespace bloch {
BLOCH_INST_PASSES_X(dfloat)
}  // namespace bloch
