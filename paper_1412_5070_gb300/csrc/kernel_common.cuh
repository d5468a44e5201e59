// kernel_common.cuh -- types and helpers shared by the library's kernel
// translation units (f12int.cu: pair data, screening, auxiliary stage,
// general contraction, host API; thin.cu: the thin contraction kernels).
#pragma once

#include <cuda_runtime.h>

#include <cstdint>

#include "auxgrid.cuh"
#include "screen.h"

namespace f12k {

constexpr int kLaux = 14;                          // highest radial order (I5 of f shells)
constexpr int kSMs = 152;                          // of a GB300
constexpr int kPartPitch = 16;                     // doubles per family-partial row (128 bytes, whole sectors)
constexpr int kSkipKey = 24 * (kLaux + 1) * 34;    // work-item key of a primitive quartet the screen drops

// Pair data of a basis as the kernels see it (shell-pair tables of Sec. 2.2).
struct PairView {
  const int *pair_start;     // [nshell*nshell + 1] first primitive pair of shell pair (i,j)
  const double *pp_p;        // exponent sum p
  const double *pp_P;        // [6*npp] centre P as heavy centre H (3) + offset P - H (3)
  const double *pp_ab;       // [4*npp] exponents a, b, 1/p, pi^{5/4} p^{-3/2}
  const int64_t *pp_eoff;    // offset into epool of this primitive pair's tables
  const double *epool;       // E (3 dims) then F (3 dims), each (la+1)(lb+1)(la+lb+1)
  const int *shell_l;
  int nshell;
  const double *qprim;       // [npp] primitive Schwarz factors of the class, or null
  const double *grow;        // [ngrow] growth G(i kGrowStep) of the class's kernel, or null (no growth)
  const float *grow32;       // the same in single precision, and its band (screen.h)
  float grow_band;
  int ngrow;
};

// A list of shell quartets.  In a batch (qslot != null) every quartet names a
// slot, which gives the pair data of its basis and the output array of its
// request; counts then live in device memory (count_dev[0] quartets,
// count_dev[1] primitive quartets), so one captured launch sequence serves
// every batch.
struct QuartetView {
  const int32_t *quartets;     // [n][4]
  const int64_t *pq_off;       // [n+1] first primitive quartet of each shell quartet
  int64_t n;
  const int64_t *count_dev;    // batch: {n, pq_off[n]} on the device, else null
  const int32_t *qslot;        // batch: slot of each quartet, else null
  const PairView *slot_view;   // batch: pair data per slot
  double *const *slot_out;     // batch: output array per slot
};


// One block of contraction work: quartet q (index into the list), range split
// of |nsplit| (nsplit < 0: the quartet is listed with its pairs swapped).
struct CTask {
  int32_t q;
  int16_t split, nsplit;
};

__host__ __device__ __forceinline__ int nh_count(int L) { return (L + 1) * (L + 2) * (L + 3) / 6; }
__host__ __device__ __forceinline__ int ncart(int l) { return (l + 1) * (l + 2) / 2; }
// index of the Hermite triple (t, u, v) in order of t+u+v, then decreasing t, then v
__host__ __device__ __forceinline__ int hidx(int t, int u, int v) {
  int s = t + u + v, w = s - t;
  return s * (s + 1) * (s + 2) / 6 + w * (w + 1) / 2 + v;
}

// X_PQ component k = Q - P = (H_cd - H_ab) + (offset_cd - offset_ab).
__device__ __forceinline__ double pair_sep(const double *ppP, int pab, int pcd, int k) {
  return (ppP[6 * pcd + k] - ppP[6 * pab + k]) + (ppP[6 * pcd + 3 + k] - ppP[6 * pab + 3 + k]);
}

// Where a class's auxiliary functions come from, when not family by family:
// the grid (auxgrid.cuh), or for I1 the table of the Boys function.
struct GridView {
  const double *cells;   // null: no grid
  const double *xt;
  const double *boys;    // null: not the Coulomb kernel
  __host__ __device__ bool direct() const { return cells || boys; }
};

// g_n, n <= L, of a primitive quartet, u = |P - Q|^2: with
//   g_n = pi^{5/2}/(sqrt(p+q) pq) hat g_n = pi^{5/2} (pq)^{-3/2} [sqrt(xi) hat g_n]
// and 1/xi = 1/p + 1/q both factors come from the pairs' tables without a
// division or a square root (some 60 FP64 instructions, a tenth of a thin
// primitive quartet's).
template <int L>
__device__ __forceinline__ void aux_direct(const GridView &G, const PairView &PV, int pab, int pcd, double u,
                                           double *g) {
  const double v = PV.pp_ab[4 * pab + 2] + PV.pp_ab[4 * pcd + 2];
  if (G.boys) f12dev::boys_eval<L, true>(G.boys, v, u, L, g);
  else f12dev::grid_eval<L, true>(G.cells, f12dev::grid_point(G.xt, v, u), L, g);
  const double pref = PV.pp_ab[4 * pab + 3] * PV.pp_ab[4 * pcd + 3];
#pragma unroll
  for (int l = 0; l <= L; ++l) g[l] *= pref;
}
__host__ __device__ constexpr int aux_direct_fmas(const bool boys, int L) {
  return boys ? f12dev::BY_NT - 1 + L : f12dev::grid_fmas(L);
}

constexpr double kPrimScreen = 1e-26;
constexpr float kPrimScreenLog2 = -86.37013f;   // its binary logarithm

// Primitive quartets whose Schwarz product is below kPrimScreen are skipped:
// the skipped contributions stay below the absolute accuracy that elements
// just above 1e-12 need for a relative error of 1e-10.  The diagonal
// integrals behind qprim sample the kernel at short range; a kernel that
// grows with r (Eq. rs12 with B > 0: I2, I3 like e^{Br}, k4 = f f' and
// k6 = f_r f'_r like e^{2Br}) is larger at the separation R = |P - Q| of the
// two charge distributions, whose overlap e^{-xi w^2} reaches out to R + w.
// A candidate is weighed, as the shell screen weighs a shell quartet, by the
// growth Gamma that its overlap reaches (screen.h).  The weighing is in single
// precision, and in double where that does not settle it (few of the
// candidates): in double precision throughout, its square roots, taken by the
// whole warp whenever one lane has a candidate, were a third of the thin
// contraction's FP64 instructions.
__device__ __forceinline__ bool prim_negligible(const PairView &PV, int pab, int pcd, double u) {
  if (!PV.qprim) return false;
  const double v = PV.qprim[pab] * PV.qprim[pcd];
  if (v >= kPrimScreen) return false;
  if (!PV.grow32) return true;
  const double iv = PV.pp_ab[4 * pab + 2] + PV.pp_ab[4 * pcd + 2];
  const int s = screen_single(v, u, iv, kPrimScreenLog2, PV.grow32, PV.ngrow, PV.grow_band);
  return s >= 0 ? s == 1 : screen_negligible(v, u, iv, kPrimScreen, PV.grow, PV.ngrow);
}

// Thin contraction (thin_*.cu): quartets of total order L <= kThinL (I5:
// L <= kThinL5), one warp per shell quartet, always in FP64 (on the mixed
// path too: there it is faster than the FP32 general kernel).
constexpr int kThinL = 3, kThinL5 = 2;
constexpr int kThinWarps = 4;
using ThinKernel = void (*)(PairView, QuartetView, int, int64_t, GridView, const CTask *, int64_t, const int64_t *,
                            const int *, const double *, double *, const int64_t *, unsigned long long *);
// The instance for class key (la << 6 | lb << 4 | lc << 2 | ld), or null.
ThinKernel thin_kernel(int key, bool i5);
// Index of a thin class key among the thin keys of its class kind (the batch
// engine's launch slot), -1 if the key is not thin there.
int thin_slot(int key, bool i5);
constexpr int kThinKeys = 35;   // thin keys of the classes other than I5 (15 for I5)
__host__ __device__ inline bool thin_quartet(int key, int cls) {
  const int L = ((key >> 6) & 3) + ((key >> 4) & 3) + ((key >> 2) & 3) + (key & 3);
  return L <= (cls == 5 ? kThinL5 : kThinL);
}

}  // namespace f12k
