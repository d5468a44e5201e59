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
F12_HD inline int grow_index(double x, int n) { return (int)fmin(x, (double)(n - 2)) + 1; }

// A primitive quartet of Schwarz product v (below limit) at distance R = sqrt(u),
// 1/xi = iv, is negligible when v Gamma < limit,
//   Gamma = max over w = 0, 0.5, .., 3 (units of 1/sqrt(xi)) of G(R + w) e^{-xi w^2}
// (e^{-xi w^2} = e^{-k^2/4} at the k-th sample), G from its table g of n entries.
F12_HD inline bool screen_negligible(double v, double u, double iv, double limit, const double *g, int n) {
  const double R = sqrt(u), hw = 0.5 * sqrt(iv);
  double gam = 0.0, w = 1.0, q = 0.77880078307140487;   // e^{-k^2/4} from one sample to the next
#ifdef __CUDACC__
#pragma unroll 1   // (seldom taken: kept small beside the code that is)
#endif
  for (int k = 0; k < 7; ++k) {
    gam = fmax(gam, g[grow_index((R + k * hw) * (1.0 / kGrowStep), n)] * w);
    w *= q;
    q *= 0.60653065971263342;
  }
  return v * gam < limit;
}

// The same, its outcome taken from single precision where that settles it: a
// distance rounded there is off by at most one entry of the table, so Gamma by at
// most the largest ratio of neighbouring entries (and a little for the
// roundings), and lo and hi are limit over and times that.  1: negligible, 0: not,
// -1: to be weighed in double precision.
F12_HD inline int screen_single(double v, double u, double iv, double lo, double hi, const float *g, int n) {
  const float R = sqrtf((float)u), hw = 0.5f * sqrtf((float)iv);
  constexpr float kOverlap[7] = {1.0f, 0.77880078307140487f, 0.36787944117144233f, 0.10539922456186433f,
                                 0.018315638888734179f, 0.0019304541362277093f, 0.00012340980408667956f};
  float gam = 0.0f;
#ifdef __CUDACC__
#pragma unroll
#endif
  for (int k = 0; k < 7; ++k) gam = fmaxf(gam, g[grow_index((R + k * hw) * (float)(1.0 / kGrowStep), n)] * kOverlap[k]);
  const double w = v * (double)gam;
  return w < lo ? 1 : w >= hi && gam < 3e38f ? 0 : -1;
}
// that ratio of a table (one that leaves the range of numbers settles nothing)
inline double screen_band(const double *g, int n) {
  double r = 1.0;
  for (int i = 0; i + 1 < n; ++i) r = fmax(r, g[i + 1] / g[i]);
  return fmin(r * (1.0 + 1e-5), 1e300);
}

}  // namespace f12k
