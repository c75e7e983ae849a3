// Multi-step backward-Euler kernel of the heat operator with direct FP32 solves
// in one precision form (FP32-pair refinement; device code in pit_direct.cuh).
#include "pit_direct.cuh"

namespace pit {
PIT_DIRECT_PREC(pair, PAIR)
}  // namespace pit
