// Mixed-radix passes, float-float fields, z passes.
#include "passes_launch.cuh"

namespace bloch {
BLOCH_INST_PASSES_Z(dfloat)
}  // namespace bloch
