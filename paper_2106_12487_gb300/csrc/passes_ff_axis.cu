// Mixed-radix passes, float-float fields, plain y and z passes.
#include "passes_launch.cuh"

namespace bloch {
BLOCH_INST_PASSES_AXIS(dfloat)
}  // namespace bloch
