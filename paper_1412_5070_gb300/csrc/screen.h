// screen.h -- the arithmetic of the primitive screen (kernel_common.cuh says what
// it weighs).  Also compiles as plain C++ (a test exercises it on the CPU).
#pragma once

#include "auxgrid.cuh"

namespace f12k {

// Growth of a kernel with distance, tabulated at this step (screening).
constexpr double kGrowStep = 0.05, kGrowMax = 120.0;

// Entry of a table of n for a distance of x steps: the next one up, the last one
// past the end.  (Clamped before the conversion: a distance past 2^31 steps,
// 1e8 bohr, gave the least int once one was added to the largest.)
F12_HD inline int grow_index(float x, int n) { return (int)fminf(x, (float)(n - 2)) + 1; }

}  // namespace f12k
