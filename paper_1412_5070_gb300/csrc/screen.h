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

// The same, its outcome taken from single precision where that settles it,
// without an FP64 instruction: the logarithms of v and Gamma against lim =
// log2(limit).  Their roundings are within kScreenSlack; a distance rounded there
// (2.5e-7 of it) is in the next entry of the table only within 2e-3 of one, and
// Gamma then off by at most the largest ratio of neighbouring entries, 2^band.
// 1: negligible, 0: not, -1: to be weighed in double precision.
constexpr float kScreenSlack = 2e-4f;
F12_HD inline int screen_single(double v, double u, double iv, float lim, const float *g, int n, float band) {
  const float R = sqrtf((float)u), hw = 0.5f * sqrtf((float)iv);
  constexpr float kOverlap[7] = {1.0f, 0.77880078307140487f, 0.36787944117144233f, 0.10539922456186433f,
                                 0.018315638888734179f, 0.0019304541362277093f, 0.00012340980408667956f};
  float gam = 0.0f;
  bool edge = false;
#ifdef __CUDACC__
#pragma unroll
#endif
  for (int k = 0; k < 7; ++k) {
    const float x = (R + k * hw) * (float)(1.0 / kGrowStep);
    edge = edge || fabsf(x - rintf(x)) < 2e-3f;
    gam = fmaxf(gam, g[grow_index(x, n)] * kOverlap[k]);
  }
  const int h = f12dev::grid_hi(v), m = 0x3f800000 | (h & 0xFFFFF) << 3;   // (its mantissa as a float in [1, 2))
#ifdef __CUDA_ARCH__
  const float t = (float)((h >> 20) - 1023) + __log2f(__int_as_float(m)) + __log2f(gam);
#else
  float f;
  std::memcpy(&f, &m, sizeof f);
  const float t = (float)((h >> 20) - 1023) + log2f(f) + log2f(gam);
#endif
  const float d = kScreenSlack + (edge ? band : 0.0f);
  return !(gam < 3e38f) ? -1 : t < lim - d ? 1 : t >= lim + d ? 0 : -1;
}
// band of a table (one that leaves the range of numbers settles next to nothing)
inline float screen_band(const double *g, int n) {
  double r = 1.0;
  for (int i = 0; i + 1 < n; ++i) r = fmax(r, g[i + 1] / g[i]);
  return (float)fmin(log2(r), 1e4);
}

}  // namespace f12k
