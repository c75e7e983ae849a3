// Multi-step backward-Euler kernel of the heat operator with direct FP32 solves
// in one precision form (FP64 refinement; device code in pit_direct.cuh).
#include "pit_direct.cuh"

namespace pit {
PIT_DIRECT_PREC(mixed, MIXED)
}  // namespace pit
