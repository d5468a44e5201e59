// f12int.cu -- CUDA kernels and C ABI of the F12 integral library (sm_103a).
//
// Stages (arXiv:1412.5070, Sec. 2):
//   1. shell-pair data: p, P, and the Hermite expansion coefficients
//      E_t^{ij} (Eq. AB, Eqs. Erec0-Erect) with their AB derivatives
//      F_t^{ij} = dE_t^{ij}/dAB_x for I5, one thread per primitive pair,
//      resident in device memory for the life of the basis;
//   2. auxiliary functions g_n = D_Q^n B_i per primitive quartet: a point of the
//      factor's grid (auxgrid.cuh; the Boys table for I1), inside the kernels of
//      stage 3; the points of a basis that the grid does not hold go family by
//      family through the work items of aux.cuh;
//   3. the Hermite integrals R_tuv = d^t/dQx^t d^u/dQy^u d^v/dQz^v B_i
//      (Eq. ri) by the Cartesian recursion for a radial function
//        R^(n)_{t+1,u,v} = t R^(n+1)_{t-1,u,v} + X_QP R^(n+1)_{t,u,v},
//      which holds because d/dQx D_Q^n B = X_QP D_Q^{n+1} B: one thread per
//      primitive quartet (contract.cuh; in the registers of thin.cuh at low order);
//   4. the contraction of Eq. ii (inner ket sum, then bra sum, or the mirror
//      image where that is cheaper) and for I5 the combination of Eq. I5byI3_,
//      accumulated over primitive quartets.
#include <cuda_runtime.h>

#include <algorithm>
#include <chrono>
#include <cmath>
#include <condition_variable>
#include <cstdint>
#include <cstdio>
#include <cstring>
#include <deque>
#include <cstdlib>
#include <map>
#include <memory>
#include <mutex>
#include <new>
#include <thread>
#include <unordered_map>
#include <vector>

#include <nvtx3/nvToolsExt.h>

#include "../../include/f12int.h"
#include "aux.cuh"
#include "kernel_common.cuh"
#include "auxtab.h"
#include "grid.h"
#include "hoststage.h"
#include "perdevice.h"
#include "scratchcut.h"
#include "termlist.h"
#include "tickets.h"

using namespace f12dev;
using namespace f12k;

namespace {

constexpr int LSH = 3;                 // highest shell angular momentum
constexpr int NHMAX = 680;             // Hermite indices with t+u+v <= 14
constexpr int BLOCK_AUX = 64;
constexpr int NSIDE = 8;               // side streams of a call's contraction launches


// ---------------------------------------------------------------------------
// device status word bits: 1 = an auxiliary series hit its length cap,
// 4 = a quartet needs a radial order above LAUX


// ------------------------------------------------------------ pair builder --
// E_0^{00} = exp(-(ab/p) X_AB^2)  (Eq. Erec0); upward in i and j with
//   E_t^{i+1,j} = E_{t-1}^{ij}/(2p) + X_PA E_t^{ij} + (t+1) E_{t+1}^{ij}
//   E_t^{i,j+1} = E_{t-1}^{ij}/(2p) + X_PB E_t^{ij} + (t+1) E_{t+1}^{ij}
// (the standard McMurchie-Davidson form equivalent to Eqs. Ereci-Erect, whose
// printed j-recursion carries a stray factor).  F = dE/dAB_x follows by
// differentiating every step: dX_PA/dAB = -b/p, dX_PB/dAB = a/p,
// dE_0^{00}/dAB = -(2ab/p) X_AB E_0^{00}.
__global__ void k_build_pairs(int npp, const int *pp_shell_a, const int *pp_shell_b, const int *pp_prim_a,
                              const int *pp_prim_b, const double *centers, const int *shell_l,
                              const double *exps, const double *coefs, double *pp_p, double *pp_P,
                              double *pp_ab, const int64_t *pp_eoff, double *epool) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= npp) return;
  int sa = pp_shell_a[i], sb = pp_shell_b[i];
  int la = shell_l[sa], lb = shell_l[sb];
  double a = exps[pp_prim_a[i]], b = exps[pp_prim_b[i]];
  double da = coefs[pp_prim_a[i]], db = coefs[pp_prim_b[i]];
  double p = a + b;
  pp_p[i] = p;
  pp_ab[4 * i] = a;
  pp_ab[4 * i + 1] = b;
  pp_ab[4 * i + 2] = 1.0 / p;
  pp_ab[4 * i + 3] = 4.1825133983795991 / (p * sqrt(p));   // pi^{5/4} p^{-3/2}
  const int nt = la + lb + 1;
  const int n1 = (la + 1) * (lb + 1) * nt;
  double *E = epool + pp_eoff[i];
  double *F = E + 3 * n1;
  // P is kept as the centre of the larger exponent H plus the offset P - H,
  // and X_PA, X_PB come from X_AB: both stay exact (zero) for one-centre
  // pairs, and X_PQ formed from them keeps its relative accuracy when P and
  // Q nearly coincide; the parity cancellations of one-centre blocks rely on
  // that.
  const bool heavy_a = a >= b;
  for (int k = 0; k < 3; ++k) {
    double A = centers[3 * sa + k], B = centers[3 * sb + k];
    double XAB = A - B, XPA = -(b / p) * XAB, XPB = (a / p) * XAB;
    pp_P[6 * i + k] = heavy_a ? A : B;
    pp_P[6 * i + 3 + k] = heavy_a ? XPA : XPB;
    double K = exp(-a * b / p * XAB * XAB);
    double scale = (k == 0) ? da * db : 1.0;
    double *Ek = E + k * n1, *Fk = F + k * n1;
    for (int j = 0; j < n1; ++j) Ek[j] = Fk[j] = 0.0;
#define EI(ii, jj, t) Ek[((ii) * (lb + 1) + (jj)) * nt + (t)]
#define FI(ii, jj, t) Fk[((ii) * (lb + 1) + (jj)) * nt + (t)]
    EI(0, 0, 0) = K;
    FI(0, 0, 0) = -2.0 * a * b / p * XAB * K;
    const double h = 0.5 / p;
    for (int ii = 0; ii <= la; ++ii) {
      if (ii > 0) {
        for (int t = 0; t <= ii; ++t) {
          double e = XPA * EI(ii - 1, 0, t), f = XPA * FI(ii - 1, 0, t) - b / p * EI(ii - 1, 0, t);
          if (t > 0) {
            e += h * EI(ii - 1, 0, t - 1);
            f += h * FI(ii - 1, 0, t - 1);
          }
          if (t + 1 <= ii - 1) {
            e += (t + 1) * EI(ii - 1, 0, t + 1);
            f += (t + 1) * FI(ii - 1, 0, t + 1);
          }
          EI(ii, 0, t) = e;
          FI(ii, 0, t) = f;
        }
      }
      for (int jj = 1; jj <= lb; ++jj) {
        for (int t = 0; t <= ii + jj; ++t) {
          double e = XPB * EI(ii, jj - 1, t), f = XPB * FI(ii, jj - 1, t) + a / p * EI(ii, jj - 1, t);
          if (t > 0) {
            e += h * EI(ii, jj - 1, t - 1);
            f += h * FI(ii, jj - 1, t - 1);
          }
          if (t + 1 <= ii + jj - 1) {
            e += (t + 1) * EI(ii, jj - 1, t + 1);
            f += (t + 1) * FI(ii, jj - 1, t + 1);
          }
          EI(ii, jj, t) = e;
          FI(ii, jj, t) = f;
        }
      }
    }
#undef EI
#undef FI
    for (int j = 0; j < n1; ++j) {
      Ek[j] *= scale;
      Fk[j] *= scale;
    }
  }
}

// ------------------------------------------------------------------- aux --
__device__ __forceinline__ int64_t qv_count(const QuartetView &QV) { return QV.count_dev ? QV.count_dev[0] : QV.n; }

// Pair data of quartet q: the kernel's own view, or the slot's in a batch
// (a compile-time choice, so that the single-basis kernels keep their view in
// the parameter space).
template <bool BATCH>
__device__ __forceinline__ const PairView &qv_view(const PairView &PV, const QuartetView &QV, int64_t q) {
  if constexpr (BATCH) return QV.slot_view[QV.qslot[q]];
  else return PV;
}


__device__ __forceinline__ int64_t find_quartet(const int64_t *off, int64_t n, int64_t pq) {
  int64_t lo = 0, hi = n - 1;
  while (lo < hi) {
    int64_t mid = (lo + hi + 1) >> 1;
    if (off[mid] <= pq) lo = mid; else hi = mid - 1;
  }
  return lo;
}

// Work items of the auxiliary stage: item = (primitive quartet of the chunk) * nf + family.
struct ItemGeom {
  double xi, D, u;
  int L;
  int iab, icd;
  const PairView *pv;
};

template <bool BATCH>
__device__ __forceinline__ ItemGeom item_geometry(const PairView &PV0, const QuartetView &QV, int cls, int64_t pq) {
  int64_t q = find_quartet(QV.pq_off, qv_count(QV), pq);
  const PairView &PV = qv_view<BATCH>(PV0, QV, q);
  const int32_t *s = QV.quartets + 4 * q;
  const int ns = PV.nshell;
  int ab = s[0] * ns + s[1], cd = s[2] * ns + s[3];
  int npcd = PV.pair_start[cd + 1] - PV.pair_start[cd];
  int64_t r = pq - QV.pq_off[q];
  int iab = PV.pair_start[ab] + (int)(r / npcd);
  int icd = PV.pair_start[cd] + (int)(r % npcd);
  ItemGeom g;
  g.iab = iab;
  g.icd = icd;
  g.pv = &PV;
  g.L = PV.shell_l[s[0]] + PV.shell_l[s[1]] + PV.shell_l[s[2]] + PV.shell_l[s[3]] + (cls == 5 ? 2 : 0);
  double p = PV.pp_p[iab], qq = PV.pp_p[icd];
  double X = pair_sep(PV.pp_P, iab, icd, 0), Y = pair_sep(PV.pp_P, iab, icd, 1), Z = pair_sep(PV.pp_P, iab, icd, 2);
  g.u = X * X + Y * Y + Z * Z;
  g.D = sqrt(g.u);
  g.xi = p * qq / (p + qq);
  return g;
}

__device__ __forceinline__ int item_key(int f, int L, int bin) { return (f * (LAUX + 1) + L) * NZBIN + bin; }
constexpr int SKIP_KEY = kSkipKey;   // last key: negligible primitive quartets
static_assert(kSkipKey == MAXFAM * (LAUX + 1) * NZBIN, "the skip key follows the item keys");
static_assert(kLaux == LAUX, "one highest radial order");

// Pass 1: key of every item and a histogram of the keys.
// Items of a list: (pq_off[n] - pq0) * nf, from the device counts in a batch.
__device__ __forceinline__ int64_t item_count(const QuartetView &QV, int nf, int64_t pq0, int64_t nitems) {
  return QV.count_dev ? (QV.count_dev[1] - pq0) * nf : nitems;
}

// hist[key] += 1 for every active lane, one atomic per distinct key of the warp
__device__ __forceinline__ void hist_add(unsigned int *hist, int key) {
  const unsigned grp = __match_any_sync(__activemask(), key);
  if ((int)(threadIdx.x & 31) == __ffs(grp) - 1) atomicAdd(&hist[key], (unsigned)__popc(grp));
}

// Pass 1: key of every item and a histogram of the keys.  One thread per
// primitive quartet (its geometry serves all of its families).
template <bool BATCH>
__global__ void k_items_classify(Tables T, PairView PV, QuartetView QV, int cls, int64_t pq0, int64_t nitems,
                                 int *keys, unsigned int *hist) {
  const int kcls = cls == 5 ? 3 : cls;
  const int nf = T.nfam[kcls];
  if (nf <= 0) return;   // a class the factor leaves out (never scheduled)
  const int64_t npq = item_count(QV, nf, pq0, nitems) / nf;
  for (int64_t r = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; r < npq;
       r += (int64_t)gridDim.x * blockDim.x) {
    ItemGeom g = item_geometry<BATCH>(PV, QV, cls, pq0 + r);
    const bool skip = prim_negligible(*g.pv, g.iab, g.icd, g.u);
    for (int f = 0; f < nf; ++f) {
      const FamDev &F = T.fam[T.fam0[kcls] + f];
      const int key = skip ? SKIP_KEY : item_key(f, min(g.L, LAUX), item_bin(F, g.xi, g.D, g.L));
      keys[r * nf + f] = key;
      hist_add(hist, key);
    }
  }
}

// Pass 2: exclusive scan of the histogram (one block).
__global__ void k_items_scan(unsigned int *hist, int nkeys) {
  __shared__ unsigned int part[1024];
  const int tid = threadIdx.x, nt = blockDim.x;
  const int per = (nkeys + nt - 1) / nt;
  unsigned int s = 0;
  for (int i = tid * per; i < min(nkeys, (tid + 1) * per); ++i) s += hist[i];
  part[tid] = s;
  __syncthreads();
  if (tid == 0) {
    unsigned int run = 0;
    for (int i = 0; i < nt; ++i) {
      unsigned int v = part[i];
      part[i] = run;
      run += v;
    }
  }
  __syncthreads();
  unsigned int run = part[tid];
  for (int i = tid * per; i < min(nkeys, (tid + 1) * per); ++i) {
    unsigned int v = hist[i];
    hist[i] = run;
    run += v;
  }
}

// Pass 3: scatter item indices into key order (order inside a key is free:
// every item is evaluated independently, so results do not depend on it).
__global__ void k_items_scatter(QuartetView QV, int nf, int64_t pq0, const int *keys, unsigned int *cursor,
                                int64_t nitems, unsigned int *order) {
  const int64_t nit = item_count(QV, nf, pq0, nitems);
  const int lane = threadIdx.x & 31;
  for (int64_t it = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; it < nit;
       it += (int64_t)gridDim.x * blockDim.x) {
    // one atomic per distinct key of the warp; lanes take consecutive slots
    const int key = keys[it];
    const unsigned grp = __match_any_sync(__activemask(), key);
    const int leader = __ffs(grp) - 1;
    unsigned base = 0;
    if (lane == leader) base = atomicAdd(&cursor[key], (unsigned)__popc(grp));
    base = __shfl_sync(grp, base, leader);
    order[base + __popc(grp & ((1u << lane) - 1u))] = (unsigned int)it;
  }
}

// Pass 4: one family's contribution to hat g_l (l <= L) per item, into
// part[item * kPartPitch + l], in key order; the row is written up to the end
// of the 32-byte sector that holds order L (zeros past L), so that no sector
// is left partly written.  The families evaluated by
// quadrature (b < 0 or a lowest power below -1, FamDev::quad) are left to a
// second launch of the same kernel with QUAD = true (family_quad), made only
// when the factor has such families.
template <bool BATCH, bool QUAD>
__device__ __forceinline__ unsigned long long items_eval_one(Tables T, PairView PV, QuartetView QV, int cls,
                                                             int64_t pq0, int64_t it, const int *keys, double *part,
                                                             unsigned int *status) {
  // a primitive quartet the screen dropped (decided once, by the classify
  // pass) is never read by the contraction
  if (keys[it] == SKIP_KEY) return 0;
  const int kcls = cls == 5 ? 3 : cls;
  const int nf = T.nfam[kcls];
  const int64_t pq = pq0 + it / nf;
  const int f = (int)(it % nf);
  const FamDev &F = T.fam[T.fam0[kcls] + f];
  if ((F.quad != 0) != QUAD) return 0;   // the other launch's family
  ItemGeom g = item_geometry<BATCH>(PV, QV, cls, pq);
  if (g.L > LAUX) {
    atomicOr(status, 4u);
    return 0;
  }
  double out[LAUX + 1];
  for (int l = 0; l <= g.L; ++l) out[l] = 0.0;
  unsigned long long nfma = 0;
  int bad = family_eval<QUAD>(T, F, g.xi, g.D, g.L, out, &nfma);
  if (bad) atomicOr(status, 1u);
  double2 *o = reinterpret_cast<double2 *>(part + it * kPartPitch);
  for (int l = 0; l <= (g.L | 3); l += 2)
    o[l >> 1] = make_double2(l <= g.L ? out[l] : 0.0, l + 1 <= g.L ? out[l + 1] : 0.0);
  return nfma;
}

template <bool BATCH, bool QUAD = false>
__global__ void k_items_eval(Tables T, PairView PV, QuartetView QV, int cls, int64_t pq0, int64_t nitems,
                             const unsigned int *order, const int *keys, double *part, unsigned int *status,
                             unsigned long long *fma_total) {
  unsigned long long nfma = 0;
  if constexpr (BATCH) {
    const int64_t nit = item_count(QV, T.nfam[cls == 5 ? 3 : cls], pq0, nitems);
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < nit; t += (int64_t)gridDim.x * blockDim.x)
      nfma += items_eval_one<BATCH, QUAD>(T, PV, QV, cls, pq0, order[t], keys, part, status);
  } else {
    const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (t < nitems) nfma = items_eval_one<BATCH, QUAD>(T, PV, QV, cls, pq0, order[t], keys, part, status);
  }
  // warp-aggregated count of the core multiply-adds (series terms and quadrature nodes)
  if (fma_total) {
    for (int o = 16; o > 0; o >>= 1) nfma += __shfl_down_sync(0xffffffffu, nfma, o);
    if ((threadIdx.x & 31) == 0 && nfma) atomicAdd(fma_total, nfma);
  }
}



// hat g_n at given (xi, D) points (no prefactor), for the aux-stage tests:
// from the grid where it holds the point, else family by family.
__global__ void k_aux_points(Tables T, GridView G, const unsigned char *ok, int cls, int64_t npts, const double *xi,
                             const double *D, int nmax, double *out, unsigned int *status) {
  int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= npts) return;
  double g[LAUX + 1];
  if (G.boys) {
    const double is = 1.0 / sqrt(xi[i]);
    boys_eval<LAUX, false>(G.boys, 1.0 / xi[i], D[i] * D[i], nmax, g);
    for (int n = 0; n <= nmax; ++n) out[i * (nmax + 1) + n] = is * g[n];
    return;
  }
  if (G.cells) {
    const GridPoint pt = grid_point(G.xt, 1.0 / xi[i], D[i] * D[i]);
    if (pt.cell >= 0 && ok[pt.cell]) {
      const double is = 1.0 / sqrt(xi[i]);
      if (nmax <= 4) grid_eval<4, false>(G.cells, pt, nmax, g);
      else if (nmax <= 8) grid_eval<8, false>(G.cells, pt, nmax, g);
      else grid_eval<LAUX, false>(G.cells, pt, nmax, g);
      for (int n = 0; n <= nmax; ++n) out[i * (nmax + 1) + n] = is * g[n];
      return;
    }
  }
  int bad = aux_eval(T, cls == 5 ? 3 : cls, xi[i], D[i], nmax, g);
  if (bad) atomicOr(status, 1u);
  for (int n = 0; n <= nmax; ++n) out[i * (nmax + 1) + n] = g[n];
}

}  // namespace

#include "contract.cuh"

// ================================================================ host API ==

namespace {
struct Engine;   // batched requests (engine.cuh)
}

// Where the arrays of a planned list lie, on the device and in its host staging.
struct ListLayout {
  size_t offsets, pqoff, rowoff, tasks, bytes;   // (the quartets are first)
  ListLayout(int64_t n, int64_t nthin, int64_t ntask) {
    offsets = (16 * (size_t)n + 15) & ~(size_t)15;
    pqoff = offsets + 8 * (size_t)n;
    rowoff = pqoff + 8 * ((size_t)n + 1);
    tasks = rowoff + 8 * ((size_t)nthin + 1);
    bytes = tasks + sizeof(CTask) * (size_t)ntask;
  }
};

// Page-locked memory of HostStage (hoststage.h).
struct PageLocked {
  static bool alloc(void **p, size_t bytes) {
    if (cudaHostAlloc(p, bytes, cudaHostAllocDefault) == cudaSuccess) return true;
    cudaGetLastError();
    return false;
  }
  static void free(void *p) { cudaFreeHost(p); }
};
using HostStage = f12host::HostStage<PageLocked>;

struct f12int_ctx {
  int device = 0;
  size_t budget = 0;
  size_t used = 0;
  cudaStream_t stream = nullptr;
  int64_t launches = 0;
  unsigned int *d_status = nullptr;
  // factor tables
  bool factor_ready = false;
  FamDev *d_fam = nullptr;
  double *d_coef = nullptr;
  GroupDev *d_grp = nullptr;
  size_t grp_bytes = 0;
  double *d_jtab = nullptr;   // start-value tables of the series families
  size_t jtab_bytes = 0;
  Tables tables{};
  const double *boys = nullptr;   // the device's table of the Boys function
  size_t fam_bytes = 0, coef_bytes = 0;
  std::shared_ptr<const f12grid::AuxGrid> grid;   // the factor's auxiliary grids (null: none)
  // basis
  struct BasisData {
    int nshell = 0;
    int *d_shell_l = nullptr;
    double *d_centers = nullptr;
    int *d_pair_start = nullptr;
    double *d_pp_p = nullptr, *d_pp_P = nullptr, *d_pp_ab = nullptr, *d_epool = nullptr;
    int64_t *d_pp_eoff = nullptr;
    std::vector<int> l, nprim, pair_start;
    std::vector<int> type, type_l, type_nprim;   // per shell: its type, (l, primitives); per type
    std::vector<double> centers, exps, coefs;
    size_t bytes = 0;
    bool prim_screen = true;            // false for the internal per-primitive basis
    double *d_qprim[7] = {nullptr};     // primitive Schwarz factors per class (lazily built)
    std::vector<double> pair_bound[7];  // shell-pair bounds sqrt(max |(ab|k|ab)|) per class (lazily built)
    std::vector<double> pair_cen;       // [nshell^2][3] centre of the most diffuse primitive pair
    std::vector<double> pair_pmin;      // [nshell^2] its exponent sum
    double exp_lo = 0.0, exp_hi = 0.0;  // range of the exponents: that of xi = pq/(p+q), p = a + b
    double dmax = 0.0;                  // bound of the distances between primitive centres
    bool grid_ok[7] = {false, false, false, false, false, false, false};   // the grid serves (basis, class)
  };
  std::deque<BasisData> bases;   // deque: growing it never moves existing entries
  // scratch of compute_class (grown on demand, bounded by the budget)
  unsigned char *d_list = nullptr;   // a planned list (ListLayout)
  HostStage stage{true};             // its staging on the host
  HostStage static_stage{false};     // that of f12int_compute_class_static
  int *d_keys = nullptr;
  unsigned *d_order = nullptr, *d_hist = nullptr;
  double *d_part = nullptr;
  double *d_rows = nullptr;      // Hermite rows of a chunk
  size_t rows_cap = 0;
  // the contraction launches of a call are independent of one another: they
  // run on these streams, between two events on the call's
  cudaStream_t side[NSIDE] = {nullptr};
  cudaEvent_t fork = nullptr, join[NSIDE] = {nullptr};
  size_t list_cap = 0, keys_cap = 0, order_cap = 0, hist_cap = 0, part_cap = 0;
  // optional per-kernel timing (events on the launching stream) and counters
  bool timing = false;
  unsigned long long *d_fma = nullptr;
  double aux_ms = 0.0, contract_ms = 0.0;
  int64_t aux_launches = 0, contract_launches = 0;
  std::vector<std::pair<cudaEvent_t, cudaEvent_t>> ev_aux, ev_con, ev_pool;
  std::mutex mu;
  std::recursive_mutex bounds_mu;   // first-time primitive and shell-pair bounds
  bool cls_ok[7] = {false, false, false, false, false, false, false};   // classes the factor supports
  bool cls_quad[7] = {false, false, false, false, false, false, false};   // classes with quadrature families
  // growth of each class's kernel with distance (screening estimate):
  // kgrow[cls][i] = G(i * kGrowStep), see screen_estimate
  std::vector<double> kgrow[7];
  // the same tables on the device for the primitive screen ([7][kgrow_n]);
  // in both precisions; grows[cls]: the kernel of cls grows (G > 1 somewhere)
  double *d_kgrow = nullptr;
  float *d_kgrow32 = nullptr;
  float grow_band[7] = {0.0f};
  size_t kgrow_bytes = 0;
  int kgrow_n = 0;
  bool grows[7] = {false, false, false, false, false, false, false};
  int series_cap = KMAX;   // f12int_set_series_cap
  double plan_ms = 0.0;    // host planning of compute_class calls (f12int_host_stats)
  int64_t plan_calls = 0;
  Engine *engine = nullptr;
};

namespace {

// The status of a CUDA call that failed.  Its error is taken off the thread's last
// one: it is reported here, and a retry with less memory (or the next call) must
// not find it after its own launches.
int cuda_fail(cudaError_t e) {
  cudaGetLastError();
  if (e == cudaErrorMemoryAllocation) return F12INT_ENOMEM;
  return F12INT_ECUDA;
}

#define CK(call)                                    \
  do {                                              \
    cudaError_t e_ = (call);                        \
    if (e_ != cudaSuccess) return cuda_fail(e_);    \
  } while (0)

template <class T>
int dalloc(f12int_ctx *ctx, T **p, size_t bytes) {
  if (bytes == 0) bytes = 8;
  if (ctx->budget && ctx->used + bytes > ctx->budget) return F12INT_ENOMEM;
  cudaError_t e = cudaMalloc((void **)p, bytes);
  if (e != cudaSuccess) return cuda_fail(e);
  ctx->used += bytes;
  return F12INT_OK;
}

template <class T>
void dfree(f12int_ctx *ctx, T *&p, size_t bytes) {
  if (p) {
    cudaFree(p);
    ctx->used -= std::min(ctx->used, bytes ? bytes : (size_t)8);
    p = nullptr;
  }
}

// Copy to the device, or clear there, complete when they return: a plain
// cudaMemcpy from pageable memory (and cudaMemset) may return while its last part
// is still to come on the legacy stream, which non-blocking streams do not wait for.
cudaError_t upload(void *dst, const void *src, size_t bytes, cudaStream_t st) {
  const cudaError_t e = cudaMemcpyAsync(dst, src, bytes, cudaMemcpyHostToDevice, st);
  return e == cudaSuccess ? cudaStreamSynchronize(st) : e;
}
cudaError_t clear(void *dst, size_t bytes, cudaStream_t st) {
  const cudaError_t e = cudaMemsetAsync(dst, 0, bytes, st);
  return e == cudaSuccess ? cudaStreamSynchronize(st) : e;
}

cudaStream_t pick_stream(f12int_ctx *ctx, void *s) { return s ? (cudaStream_t)s : ctx->stream; }

// NVTX range over a host scope (the stages of a call, visible in a profiler's
// timeline; free when no tool is attached)
struct NvtxRange {
  explicit NvtxRange(const char *name) { nvtxRangePushA(name); }
  ~NvtxRange() { nvtxRangePop(); }
  NvtxRange(const NvtxRange &) = delete;
  NvtxRange &operator=(const NvtxRange &) = delete;
};

// The pair data of a basis as the kernels see it, for class cls: with the
// primitive screen (its Schwarz factors and the kernel's growth table) when
// screen is set and the factors exist.
PairView pair_view(const f12int_ctx *ctx, const f12int_ctx::BasisData &B, int cls, bool screen) {
  PairView v{B.d_pair_start, B.d_pp_p, B.d_pp_P, B.d_pp_ab, B.d_pp_eoff, B.d_epool, B.d_shell_l, B.nshell,
             nullptr, nullptr, nullptr, 0.0f, 0};
  if (screen && B.d_qprim[cls]) {
    v.qprim = B.d_qprim[cls];
    if (ctx->grows[cls] && ctx->d_kgrow) {
      v.grow = ctx->d_kgrow + (size_t)cls * ctx->kgrow_n;
      v.grow32 = ctx->d_kgrow32 + (size_t)cls * ctx->kgrow_n;
      v.grow_band = ctx->grow_band[cls];
      v.ngrow = ctx->kgrow_n;
    }
  }
  return v;
}

static_assert(BY_LSTRIDE == MT_NA * MT_NX * MT_NT && BY_NT == MT_NT && BY_XMAX <= (MT_NX - 1) * MT_DX && MT_DX == 0.5,
              "boys_eval reads the Kummer table");

// How a class of a basis gets its auxiliary functions: I1 from the Boys
// table, the others from the grid if it holds every (xi, D) of the basis,
// else family by family.  A lowered series cap (a test aid) keeps to the
// series.
GridView class_view(const f12int_ctx *ctx, int cls) {
  if (ctx->series_cap < KMAX) return GridView{nullptr, nullptr, nullptr};
  if (cls == 1) return GridView{nullptr, nullptr, ctx->boys};
  const int k = cls == 5 ? 3 : cls;
  if (!ctx->grid || !ctx->grid->cells[k]) return GridView{nullptr, nullptr, nullptr};
  return GridView{ctx->grid->cells[k], ctx->grid->xt, nullptr};
}
GridView grid_view(const f12int_ctx *ctx, const f12int_ctx::BasisData &B, int cls) {
  return cls == 1 || B.grid_ok[cls] ? class_view(ctx, cls) : GridView{nullptr, nullptr, nullptr};
}

void mark_grid(const f12int_ctx *ctx, f12int_ctx::BasisData &B) {
  for (int c = 2; c <= 6; ++c)
    B.grid_ok[c] = ctx->grid && ctx->cls_ok[c] && f12grid::covers(*ctx->grid, c, B.exp_lo, B.exp_hi, B.dmax);
}

f12host::PerDevice<const double *> g_tables;

// Fills the constant tables of the current device; *boys: the Kummer table's
// rows of a = 1.
int upload_constants(const double **boys) {
  unsigned tuv[NHMAX];
  for (int s = 0; s <= 14; ++s)
    for (int t = s; t >= 0; --t)
      for (int v = 0; v <= s - t; ++v) {
        const int u = s - t - v;
        tuv[hidx(t, u, v)] = (unsigned)(t | u << 4 | v << 8);
      }
  const HostPairTabs &pt = pair_tabs();
  if (pt.term.size() > (size_t)PT_TERMS) return F12INT_ECUDA;
  CK(cudaMemcpyToSymbol(d_pt, pt.pt, sizeof(pt.pt)));
  CK(cudaMemcpyToSymbol(d_pt_term, pt.term.data(), sizeof(uint2) * pt.term.size()));
  static AuxConst ac;
  fill_aux_const(ac);
  CK(cudaMemcpyToSymbol(c_cratio, ac.cratio, sizeof(ac.cratio)));
  CK(cudaMemcpyToSymbol(c_inv_dfact, ac.inv_dfact, sizeof(ac.inv_dfact)));
  CK(cudaMemcpyToSymbol(d_kum_inv, ac.kum_inv, sizeof(ac.kum_inv)));
  CK(cudaMemcpyToSymbol(d_sm1_ratio, ac.sm1_ratio, sizeof(ac.sm1_ratio)));
  CK(cudaMemcpyToSymbol(d_cser, ac.cser, sizeof(ac.cser)));
  CK(cudaMemcpyToSymbol(d_vstep, ac.vstep, sizeof(ac.vstep)));
  CK(cudaMemcpyToSymbol(d_quarter, ac.quarter, sizeof(ac.quarter)));
  CK(cudaMemcpyToSymbol(d_htuv, tuv, sizeof(tuv)));
  CK(cudaMemcpyToSymbol(c_gh_x, ac.gh_x, sizeof(ac.gh_x)));
  CK(cudaMemcpyToSymbol(c_gh_w, ac.gh_w, sizeof(ac.gh_w)));
  CK(cudaMemcpyToSymbol(c_gl_x, ac.gl_x, sizeof(ac.gl_x)));
  CK(cudaMemcpyToSymbol(c_gl_w, ac.gl_w, sizeof(ac.gl_w)));
  {
    // the Kummer table of the b = 0 families (13.5 MB), kept for the process
    std::vector<double> kt;
    fill_kummer_table(kt);
    double *dk = nullptr;
    CK(cudaMalloc(&dk, sizeof(double) * kt.size()));
    const double *dkc = dk;
    cudaError_t e = cudaMemcpyAsync(dk, kt.data(), sizeof(double) * kt.size(), cudaMemcpyHostToDevice, nullptr);
    if (e == cudaSuccess) e = cudaMemcpyToSymbol(d_mtab, &dkc, sizeof(dkc));
    if (e == cudaSuccess) e = cudaDeviceSynchronize();   // (the symbols' copies above as well)
    if (e != cudaSuccess) {
      cudaFree(dk);
      return cuda_fail(e);
    }
    *boys = dk + (size_t)1 * MT_NX * MT_NT;   // a = (1 + 1)/2
  }
  return F12INT_OK;
}

bool finite_factor(const f12int_factor &f) {
  return std::isfinite(f.c0) && std::isfinite(f.rho) && std::isfinite(f.B) && std::isfinite(f.mu);
}

// A factor given as terms: 1..64 finite terms with g >= 0, not all zero.
int check_terms(const f12int_term *t, int n, f12::TermList &out) {
  if (!t || n < 1 || n > 64) return F12INT_EINVAL;
  out.clear();
  for (int i = 0; i < n; ++i) {
    const f12int_term &u = t[i];
    if (!std::isfinite(u.c) || !std::isfinite(u.a) || !std::isfinite(u.b) || !std::isfinite(u.g) || u.g < 0.0)
      return F12INT_EDOMAIN;
    out.push_back({u.c, u.a, u.b, u.g});
  }
  f12::simplify(out);
  return out.empty() ? F12INT_EDOMAIN : F12INT_OK;
}

int check_factor(const f12int_factor &f) {
  if (!finite_factor(f)) return F12INT_EDOMAIN;
  if (!(f.mu > 0.0) || f.c0 < 0.0 || f.n < 0 || f.n > 20) return F12INT_EDOMAIN;
  if (f.c0 > 0.0 && !(f.rho + 2.0 * f.n + 2.0 > 0.0)) return F12INT_EDOMAIN;
  return F12INT_OK;
}

}  // namespace

extern "C" {

static void collect_events(f12int_ctx *ctx);

const char *f12int_strerror(int status) {
  switch (status) {
    case F12INT_OK: return "ok";
    case F12INT_EINVAL: return "invalid argument";
    case F12INT_ENOMEM: return "device memory budget exceeded";
    case F12INT_EDOMAIN: return "correlation-factor parameters outside the supported domain";
    case F12INT_ENOTREADY: return "basis or correlation factor not set";
    case F12INT_ETIMEOUT: return "timed out";
    case F12INT_ECUDA: return "CUDA runtime error";
    case F12INT_EDEVICE: return "device-side check failed";
    default: return "unknown status";
  }
}

int f12int_create(f12int_ctx **out, int device, size_t hbm_budget_bytes, void *cuda_stream) {
  if (!out) return F12INT_EINVAL;
  *out = nullptr;
  int ndev = 0;
  CK(cudaGetDeviceCount(&ndev));
  if (device < 0 || device >= ndev) return F12INT_EINVAL;
  CK(cudaSetDevice(device));
  f12int_ctx *ctx = new (std::nothrow) f12int_ctx();
  if (!ctx) return F12INT_ENOMEM;
  ctx->device = device;
  ctx->budget = hbm_budget_bytes;
  ctx->stream = (cudaStream_t)cuda_stream;
  int rc = g_tables.get(device, &ctx->boys, [](const double *&boys) { return upload_constants(&boys); });
  if (rc == F12INT_OK) rc = dalloc(ctx, &ctx->d_status, sizeof(unsigned int));
  if (rc == F12INT_OK && clear(ctx->d_status, sizeof(unsigned int), ctx->stream) != cudaSuccess) rc = F12INT_ECUDA;
  for (int i = 0; i < NSIDE && rc == F12INT_OK; ++i)
    if (cudaStreamCreateWithFlags(&ctx->side[i], cudaStreamNonBlocking) != cudaSuccess ||
        cudaEventCreateWithFlags(&ctx->join[i], cudaEventDisableTiming) != cudaSuccess)
      rc = F12INT_ECUDA;
  if (rc == F12INT_OK && cudaEventCreateWithFlags(&ctx->fork, cudaEventDisableTiming) != cudaSuccess) rc = F12INT_ECUDA;
  if (rc != F12INT_OK) {
    f12int_destroy(ctx);
    return rc;
  }
  *out = ctx;
  return F12INT_OK;
}

static void engine_shutdown(f12int_ctx *ctx);
static bool engine_idle(f12int_ctx *ctx);
static void engine_factor_changed(f12int_ctx *ctx);

int f12int_destroy(f12int_ctx *ctx) {
  if (!ctx) return F12INT_EINVAL;
  cudaSetDevice(ctx->device);
  engine_shutdown(ctx);
  cudaDeviceSynchronize();
  for (auto &b : ctx->bases) {
    cudaFree(b.d_shell_l);
    cudaFree(b.d_centers);
    cudaFree(b.d_pair_start);
    cudaFree(b.d_pp_p);
    cudaFree(b.d_pp_P);
    cudaFree(b.d_pp_ab);
    cudaFree(b.d_epool);
    cudaFree(b.d_pp_eoff);
    for (int c = 0; c < 7; ++c) cudaFree(b.d_qprim[c]);
  }
  cudaFree(ctx->d_fam);
  cudaFree(ctx->d_coef);
  cudaFree(ctx->d_grp);
  cudaFree(ctx->d_jtab);
  cudaFree(ctx->d_kgrow);
  cudaFree(ctx->d_kgrow32);
  cudaFree(ctx->d_list);
  cudaFree(ctx->d_keys);
  cudaFree(ctx->d_order);
  cudaFree(ctx->d_hist);
  cudaFree(ctx->d_part);
  cudaFree(ctx->d_rows);
  for (int i = 0; i < NSIDE; ++i) {
    if (ctx->side[i]) cudaStreamDestroy(ctx->side[i]);
    if (ctx->join[i]) cudaEventDestroy(ctx->join[i]);
  }
  if (ctx->fork) cudaEventDestroy(ctx->fork);
  cudaFree(ctx->d_status);
  cudaFree(ctx->d_fma);
  ctx->stage.release();
  ctx->static_stage.release();
  for (auto &e : ctx->ev_pool) {
    cudaEventDestroy(e.first);
    cudaEventDestroy(e.second);
  }
  delete ctx;
  return F12INT_OK;
}

int64_t f12int_launch_count(const f12int_ctx *ctx) { return ctx ? ctx->launches : -1; }

int f12int_set_timing(f12int_ctx *ctx, int on) {
  if (!ctx) return F12INT_EINVAL;
  std::lock_guard<std::mutex> lk(ctx->mu);
  CK(cudaSetDevice(ctx->device));
  if (on && !ctx->d_fma) {
    int rc = dalloc(ctx, &ctx->d_fma, 2 * sizeof(unsigned long long));
    if (rc != F12INT_OK) return rc;
    CK(clear(ctx->d_fma, 2 * sizeof(unsigned long long), ctx->stream));
  }
  ctx->timing = on != 0;
  return F12INT_OK;
}

int f12int_kernel_stats(f12int_ctx *ctx, int reset, double *stats) {
  if (!ctx || !stats) return F12INT_EINVAL;
  std::lock_guard<std::mutex> lk(ctx->mu);
  CK(cudaSetDevice(ctx->device));
  CK(cudaStreamSynchronize(ctx->stream));
  collect_events(ctx);
  unsigned long long cnt[2] = {0, 0};
  if (ctx->d_fma) CK(cudaMemcpy(cnt, ctx->d_fma, sizeof(cnt), cudaMemcpyDeviceToHost));
  stats[0] = ctx->aux_ms;
  stats[1] = (double)ctx->aux_launches;
  stats[2] = ctx->contract_ms;
  stats[3] = (double)ctx->contract_launches;
  stats[4] = 2.0 * (double)cnt[0];
  stats[5] = (double)cnt[1];
  if (reset) {
    ctx->aux_ms = ctx->contract_ms = 0.0;
    ctx->aux_launches = ctx->contract_launches = 0;
    if (ctx->d_fma) CK(clear(ctx->d_fma, sizeof(cnt), ctx->stream));
  }
  return F12INT_OK;
}

int f12int_host_stats(f12int_ctx *ctx, int reset, double *stats) {
  if (!ctx || !stats) return F12INT_EINVAL;
  std::lock_guard<std::mutex> lk(ctx->mu);
  stats[0] = ctx->plan_ms;
  stats[1] = (double)ctx->plan_calls;
  if (reset) {
    ctx->plan_ms = 0.0;
    ctx->plan_calls = 0;
  }
  return F12INT_OK;
}

int f12int_set_series_cap(f12int_ctx *ctx, int kmax) {
  if (!ctx || kmax < 0) return F12INT_EINVAL;
  if (!engine_idle(ctx)) return F12INT_EINVAL;   // submitted requests use the current tables
  std::lock_guard<std::mutex> lk(ctx->mu);
  ctx->series_cap = kmax == 0 ? KMAX : std::min(kmax, KMAX);
  ctx->tables.kcap = ctx->series_cap;
  engine_factor_changed(ctx);
  return F12INT_OK;
}

int f12int_device_status(f12int_ctx *ctx) {
  if (!ctx) return F12INT_EINVAL;
  std::lock_guard<std::mutex> lk(ctx->mu);
  CK(cudaSetDevice(ctx->device));
  unsigned int h = 0;
  CK(cudaMemcpyAsync(&h, ctx->d_status, sizeof(h), cudaMemcpyDeviceToHost, ctx->stream));
  CK(cudaStreamSynchronize(ctx->stream));
  CK(cudaMemsetAsync(ctx->d_status, 0, sizeof(unsigned int), ctx->stream));
  CK(cudaStreamSynchronize(ctx->stream));
  return h ? F12INT_EDEVICE : F12INT_OK;
}

}  // extern "C"

// x^{2l+2} (D_r^l k)(x) of a kernel from its families.
static double kernel_radial_value(const f12::TermList &kt, int l, double x) {
  std::vector<f12::Family> fl = f12::families(kt);
  double s = 0.0;
  for (const f12::Family &fam0 : fl) {
    f12::Family cur = fam0;
    for (int k = 0; k < l; ++k) cur = f12::radial_derivative(cur);
    // x^{2l+2} * sum_j P_j x^{a0 - 2l + j} e^{b x - g x^2}, with a0 the original lowest power
    double poly = 0.0;
    for (size_t j = cur.poly.size(); j-- > 0;) poly = poly * x + cur.poly[j];
    s += poly * std::pow(x, fam0.a0 + 2.0) * std::exp(fam0.b * x - fam0.g * x * x);
  }
  return s;
}

extern "C" {

int f12int_kernel_radial(int cls, const f12int_factor *f, const f12int_factor *fprime, int l, double x,
                         double *value) {
  if (!f || !value || cls < 1 || cls > 6 || l < 0 || l > LAUX || !(x > 0.0)) return F12INT_EINVAL;
  const f12int_factor &fp = fprime ? *fprime : *f;
  int rc = check_factor(*f);
  if (rc == F12INT_OK) rc = check_factor(fp);
  if (rc != F12INT_OK) return rc;
  f12::Factor F1{f->c0, f->rho, f->B, f->mu, f->n}, F2{fp.c0, fp.rho, fp.B, fp.mu, fp.n};
  *value = kernel_radial_value(f12::kernel_terms(cls, F1, F2), l, x);
  return F12INT_OK;
}

}  // extern "C"

static int factor_class_flags(const f12::TermList &T1, const f12::TermList &T2, int *flags) {
  f12::TermList kt[NCLASS];
  for (int cls = 1; cls <= 6; ++cls)
    if (cls != 5) kt[cls] = f12::kernel_terms(cls, T1, T2);
  ClassTables ct;
  if (!build_class_tables(kt, ct)) return F12INT_EDOMAIN;
  flags[0] = 0;
  for (int c = 1; c <= 6; ++c) flags[c] = ct.supported[c] ? (ct.quad[c] ? 3 : 1) : 0;
  return F12INT_OK;
}

extern "C" {

int f12int_factor_classes(const f12int_factor *f, const f12int_factor *fprime, int *flags) {
  if (!f || !flags) return F12INT_EINVAL;
  const f12int_factor &fp = fprime ? *fprime : *f;
  int rc = check_factor(*f);
  if (rc == F12INT_OK) rc = check_factor(fp);
  if (rc != F12INT_OK) return rc;
  f12::Factor F1{f->c0, f->rho, f->B, f->mu, f->n}, F2{fp.c0, fp.rho, fp.B, fp.mu, fp.n};
  return factor_class_flags(f12::factor_terms(F1), f12::factor_terms(F2), flags);
}

int f12int_factor_classes_terms(const f12int_term *f, int nf, const f12int_term *fprime, int nfp, int *flags) {
  if (!flags) return F12INT_EINVAL;
  f12::TermList T1, T2;
  int rc = check_terms(f, nf, T1);
  if (rc == F12INT_OK) rc = fprime ? check_terms(fprime, nfp, T2) : (T2 = T1, F12INT_OK);
  if (rc != F12INT_OK) return rc;
  return factor_class_flags(T1, T2, flags);
}

int f12int_kernel_radial_terms(int cls, const f12int_term *f, int nf, const f12int_term *fprime, int nfp, int l,
                               double x, double *value) {
  if (!value || cls < 1 || cls > 6 || l < 0 || l > LAUX || !(x > 0.0)) return F12INT_EINVAL;
  f12::TermList T1, T2;
  int rc = check_terms(f, nf, T1);
  if (rc == F12INT_OK) rc = fprime ? check_terms(fprime, nfp, T2) : (T2 = T1, F12INT_OK);
  if (rc != F12INT_OK) return rc;
  *value = kernel_radial_value(f12::kernel_terms(cls, T1, T2), l, x);
  return F12INT_OK;
}

}  // extern "C"

// Screening estimate of a quartet: bound(ab) bound(cd) Gamma.  The diagonal
// blocks behind bound() sample the kernel at short range only; the F12
// kernels with B > 0 grow with r (Eq. rs12), so a quartet whose charge
// distributions lie R apart is larger by about the kernel's size there
// relative to short range.  With G(x) = max(1, max_{1 <= s <= x} |k(s)| /
// max_{1/2 <= s <= 3/2} |k(s)|) (G = 1 for 1/r), the overlap of the two
// distributions, exp(-xi w^2) at distance R + w, weighs the growth:
//   Gamma = max over w = 0, 0.5, .., 3 (in units of 1/sqrt(xi)) of
//           G(R + w) exp(-xi w^2),
// with R and xi = pq/(p+q) from each pair's most diffuse primitive pair.
// I5 (whose kinetic transform raises a quartet by about the bra exponents
// over the I3 diagonal it borrows) and I6 (whose f_r f'_r diagonal can cancel
// at short range) carry a further factor 8; on the 12-atom s/p/d sample the
// largest ratio of a quartet to its unscaled estimate was 55 (I5) and 49 (I6).
constexpr double kScreenSafety[7] = {1.0, 1.0, 1.0, 1.0, 1.0, 8.0, 8.0};
static std::vector<double> growth_table(const f12::TermList &t) {
  auto kval = [&](double x) {
    double v = 0.0;
    for (const f12::Term &u : t) v += u.c * std::pow(x, u.a) * std::exp(u.b * x - u.g * x * x);
    return std::fabs(v);
  };
  double kref = 0.0;
  for (double x = 0.5; x <= 1.5 + 1e-12; x += 0.01) kref = std::max(kref, kval(x));
  const int n = (int)(kGrowMax / kGrowStep) + 1;
  std::vector<double> g((size_t)n, 1.0);
  double run = 0.0;
  for (int i = 0; i < n; ++i) {
    const double x = i * kGrowStep;
    if (x >= 1.0) run = std::max(run, kval(x));
    g[i] = kref > 0.0 ? std::max(1.0, run / kref) : 1.0;
  }
  return g;
}

static double screen_estimate(const f12int_ctx *ctx, const f12int_ctx::BasisData &B, int cls, int a, int b, int c,
                              int d) {
  const std::vector<double> &pb = B.pair_bound[cls == 5 ? 3 : cls];
  const int ns = B.nshell;
  const size_t ab = (size_t)a * ns + b, cd = (size_t)c * ns + d;
  const double q = pb[ab] * pb[cd];
  const std::vector<double> &g = ctx->kgrow[cls];
  if (q == 0.0 || g.empty()) return q * kScreenSafety[cls];
  double r2 = 0.0;
  for (int k = 0; k < 3; ++k) {
    const double dx = B.pair_cen[3 * ab + k] - B.pair_cen[3 * cd + k];
    r2 += dx * dx;
  }
  const double p = B.pair_pmin[ab], qq = B.pair_pmin[cd];
  const double xi = p * qq / (p + qq), R = std::sqrt(r2), w1 = 1.0 / std::sqrt(xi);
  double gam = 1.0;
  for (int k = 0; k <= 6; ++k) {
    const double w = 0.5 * k * w1;
    const size_t i = std::min(g.size() - 1, (size_t)((R + w) / kGrowStep) + 1);
    gam = std::max(gam, g[i] * std::exp(-xi * w * w));
  }
  return q * gam * kScreenSafety[cls];
}

// The part of f12int_set_factor(_terms) after validation: kernels, families,
// upload, and the bounds and schedules that depend on the factor.
static int set_factor_lists(f12int_ctx *ctx, const f12::TermList &T1, const f12::TermList &T2) {
  if (!engine_idle(ctx)) return F12INT_EINVAL;   // submitted requests still use the current factor
  std::lock_guard<std::mutex> lk(ctx->mu);
  CK(cudaSetDevice(ctx->device));
  int rc = F12INT_OK;
  f12::TermList kt[NCLASS];
  for (int cls = 1; cls <= 6; ++cls)
    if (cls != 5) kt[cls] = f12::kernel_terms(cls, T1, T2);
  ClassTables ct;
  if (!build_class_tables(kt, ct)) return F12INT_EDOMAIN;
  // The tables are replaced one after the other: until all of them are there the
  // context has no factor, and a call after a failure below is refused
  // (F12INT_ENOTREADY) instead of reading freed tables or the former grid.
  ctx->factor_ready = false;
  ctx->tables = Tables{};
  ctx->grid.reset();
  for (auto &b : ctx->bases) mark_grid(ctx, b);
  engine_factor_changed(ctx);
  const std::vector<FamDev> &fams = ct.fams;
  const std::vector<double> &coef = ct.coef;
  Tables T{};
  for (int c = 0; c < NCLASS; ++c) {
    T.nfam[c] = ct.nfam[c];
    T.fam0[c] = ct.fam0[c];
  }
  // upload
  dfree(ctx, ctx->d_fam, ctx->fam_bytes);
  dfree(ctx, ctx->d_coef, ctx->coef_bytes);
  dfree(ctx, ctx->d_grp, ctx->grp_bytes);
  dfree(ctx, ctx->d_jtab, ctx->jtab_bytes);
  ctx->d_grp = nullptr;
  ctx->d_jtab = nullptr;
  ctx->fam_bytes = fams.size() * sizeof(FamDev);
  ctx->coef_bytes = coef.size() * sizeof(double);
  ctx->grp_bytes = ct.groups.size() * sizeof(GroupDev);
  ctx->jtab_bytes = ct.jtab.size() * sizeof(double);
  rc = dalloc(ctx, &ctx->d_fam, ctx->fam_bytes);
  if (rc == F12INT_OK) rc = dalloc(ctx, &ctx->d_coef, ctx->coef_bytes);
  if (rc == F12INT_OK && ctx->grp_bytes) rc = dalloc(ctx, &ctx->d_grp, ctx->grp_bytes);
  if (rc == F12INT_OK && ctx->jtab_bytes) rc = dalloc(ctx, &ctx->d_jtab, ctx->jtab_bytes);
  if (rc != F12INT_OK) return rc;
  CK(upload(ctx->d_fam, fams.data(), ctx->fam_bytes, ctx->stream));
  CK(upload(ctx->d_coef, coef.data(), ctx->coef_bytes, ctx->stream));
  if (ctx->grp_bytes)
    CK(upload(ctx->d_grp, ct.groups.data(), ctx->grp_bytes, ctx->stream));
  if (ctx->jtab_bytes)
    CK(upload(ctx->d_jtab, ct.jtab.data(), ctx->jtab_bytes, ctx->stream));
  T.fam = ctx->d_fam;
  T.coef = ctx->d_coef;
  T.grp = ctx->d_grp;
  T.jtab = ctx->d_jtab;
  T.kcap = ctx->series_cap;
  ctx->tables = T;
  for (int c = 1; c <= 6; ++c) {
    ctx->cls_ok[c] = ct.supported[c];
    ctx->cls_quad[c] = ct.quad[c];
  }
  for (auto &b : ctx->bases)   // the primitive bounds depend on the factor
    for (int c = 0; c < 7; ++c)
      if (b.d_qprim[c]) {
        cudaFree(b.d_qprim[c]);
        b.d_qprim[c] = nullptr;
      }
  for (auto &b : ctx->bases)   // and so do the shell-pair bounds
    for (int c = 0; c < 7; ++c) b.pair_bound[c].clear();
  for (int c = 1; c <= 6; ++c) ctx->kgrow[c] = growth_table(kt[c == 5 ? 3 : c]);
  {
    dfree(ctx, ctx->d_kgrow, ctx->kgrow_bytes);
    dfree(ctx, ctx->d_kgrow32, ctx->kgrow_bytes / 2);
    ctx->kgrow_n = (int)ctx->kgrow[1].size();
    std::vector<double> all((size_t)7 * ctx->kgrow_n, 1.0);
    std::vector<float> single(all.size(), 1.0f);
    for (int c = 1; c <= 6; ++c) {
      ctx->grows[c] = false;
      ctx->grow_band[c] = screen_band(ctx->kgrow[c].data(), ctx->kgrow_n);
      for (int i = 0; i < ctx->kgrow_n; ++i) {
        const double g = ctx->kgrow[c][i];
        all[(size_t)c * ctx->kgrow_n + i] = g;
        single[(size_t)c * ctx->kgrow_n + i] = g < 3e38 ? (float)g : INFINITY;
        ctx->grows[c] = ctx->grows[c] || g > 1.0;
      }
    }
    ctx->kgrow_bytes = sizeof(double) * all.size();
    rc = dalloc(ctx, &ctx->d_kgrow, ctx->kgrow_bytes);
    if (rc == F12INT_OK) rc = dalloc(ctx, &ctx->d_kgrow32, ctx->kgrow_bytes / 2);
    if (rc != F12INT_OK) return rc;
    CK(upload(ctx->d_kgrow, all.data(), ctx->kgrow_bytes, ctx->stream));
    CK(upload(ctx->d_kgrow32, single.data(), ctx->kgrow_bytes / 2, ctx->stream));
  }
  {
    f12::TermList gk[7];
    for (int c = 1; c <= 6; ++c) gk[c] = kt[c];
    ctx->grid = f12grid::acquire(ctx->device, gk, ctx->cls_ok, ctx->stream);
    for (auto &b : ctx->bases) mark_grid(ctx, b);
  }
  ctx->factor_ready = true;
  return F12INT_OK;
}

extern "C" {

int f12int_set_factor(f12int_ctx *ctx, const f12int_factor *f, const f12int_factor *fprime) {
  if (!ctx || !f) return F12INT_EINVAL;
  const f12int_factor &fp = fprime ? *fprime : *f;
  int rc = check_factor(*f);
  if (rc == F12INT_OK) rc = check_factor(fp);
  if (rc != F12INT_OK) return rc;
  f12::Factor F1{f->c0, f->rho, f->B, f->mu, f->n}, F2{fp.c0, fp.rho, fp.B, fp.mu, fp.n};
  return set_factor_lists(ctx, f12::factor_terms(F1), f12::factor_terms(F2));
}

int f12int_set_factor_terms(f12int_ctx *ctx, const f12int_term *f, int nf, const f12int_term *fprime, int nfp) {
  if (!ctx) return F12INT_EINVAL;
  f12::TermList T1, T2;
  int rc = check_terms(f, nf, T1);
  if (rc == F12INT_OK) rc = fprime ? check_terms(fprime, nfp, T2) : (T2 = T1, F12INT_OK);
  if (rc != F12INT_OK) return rc;
  return set_factor_lists(ctx, T1, T2);
}

int f12int_set_basis(f12int_ctx *ctx, int nshell, const double *centers, const int *l, const int *nprim,
                     const double *exps, const double *coefs, int *basis_id) {
  if (!ctx || nshell <= 0 || !centers || !l || !nprim || !exps || !coefs || !basis_id) return F12INT_EINVAL;
  int nptot = 0;
  for (int i = 0; i < nshell; ++i) {
    if (l[i] < 0 || l[i] > LSH || nprim[i] < 1) return F12INT_EINVAL;
    for (int k = 0; k < 3; ++k)
      if (!std::isfinite(centers[3 * i + k])) return F12INT_EINVAL;
    nptot += nprim[i];
  }
  for (int i = 0; i < nptot; ++i)
    if (!(exps[i] > 0.0) || !std::isfinite(exps[i]) || !std::isfinite(coefs[i])) return F12INT_EINVAL;
  std::lock_guard<std::mutex> lk(ctx->mu);
  CK(cudaSetDevice(ctx->device));
  f12int_ctx::BasisData B;
  B.nshell = nshell;
  B.l.assign(l, l + nshell);
  B.nprim.assign(nprim, nprim + nshell);
  B.centers.assign(centers, centers + 3 * nshell);
  B.exps.assign(exps, exps + nptot);
  B.coefs.assign(coefs, coefs + nptot);
  std::vector<int> poff(nshell);
  for (int i = 0, o = 0; i < nshell; ++i) {
    poff[i] = o;
    o += nprim[i];
  }
  {
    std::map<std::pair<int, int>, int> types;
    for (int i = 0; i < nshell; ++i) {
      const auto it = types.emplace(std::make_pair(l[i], nprim[i]), (int)types.size());
      if (it.second) {
        B.type_l.push_back(l[i]);
        B.type_nprim.push_back(nprim[i]);
      }
      B.type.push_back(it.first->second);
    }
  }
  // primitive pairs of every ordered shell pair (i, j), i outer
  std::vector<int> sa, sb, pa, pb;
  std::vector<int64_t> eoff;
  B.pair_start.assign((size_t)nshell * nshell + 1, 0);
  int64_t epos = 0;
  for (int i = 0; i < nshell; ++i)
    for (int j = 0; j < nshell; ++j) {
      B.pair_start[(size_t)i * nshell + j] = (int)sa.size();
      int n1 = (l[i] + 1) * (l[j] + 1) * (l[i] + l[j] + 1);
      for (int x = 0; x < nprim[i]; ++x)
        for (int y = 0; y < nprim[j]; ++y) {
          sa.push_back(i);
          sb.push_back(j);
          pa.push_back(poff[i] + x);
          pb.push_back(poff[j] + y);
          eoff.push_back(epos);
          epos += 6 * n1;
        }
    }
  B.pair_start[(size_t)nshell * nshell] = (int)sa.size();
  const int npp = (int)sa.size();
  // most diffuse primitive pair of every shell pair (screening geometry)
  B.pair_cen.assign((size_t)nshell * nshell * 3, 0.0);
  B.pair_pmin.assign((size_t)nshell * nshell, 0.0);
  for (int i = 0; i < nshell; ++i)
    for (int j = 0; j < nshell; ++j) {
      double ea = exps[poff[i]], eb = exps[poff[j]];
      for (int x = 1; x < nprim[i]; ++x) ea = std::min(ea, exps[poff[i] + x]);
      for (int y = 1; y < nprim[j]; ++y) eb = std::min(eb, exps[poff[j] + y]);
      const size_t k = (size_t)i * nshell + j;
      B.pair_pmin[k] = ea + eb;
      for (int d = 0; d < 3; ++d)
        B.pair_cen[3 * k + d] = (ea * centers[3 * i + d] + eb * centers[3 * j + d]) / (ea + eb);
    }
  // device buffers
  int *d_sa = nullptr, *d_sb = nullptr, *d_pa = nullptr, *d_pb = nullptr;
  double *d_exps = nullptr, *d_coefs = nullptr;
  int rc = F12INT_OK;
  size_t bytes = 0;
  auto A = [&](auto **p, size_t n) {
    if (rc != F12INT_OK) return;
    rc = dalloc(ctx, p, n);
    bytes += n;
  };
  A(&B.d_shell_l, sizeof(int) * nshell);
  A(&B.d_centers, sizeof(double) * 3 * nshell);
  A(&B.d_pair_start, sizeof(int) * B.pair_start.size());
  A(&B.d_pp_p, sizeof(double) * npp);
  A(&B.d_pp_P, sizeof(double) * 6 * npp);
  A(&B.d_pp_ab, sizeof(double) * 4 * npp);
  A(&B.d_pp_eoff, sizeof(int64_t) * npp);
  A(&B.d_epool, sizeof(double) * std::max<int64_t>(epos, 1));
  B.bytes = bytes;
  size_t tmpb = 0;
  auto At = [&](auto **p, size_t n) {
    if (rc != F12INT_OK) return;
    rc = dalloc(ctx, p, n);
    tmpb += n;
  };
  At(&d_sa, sizeof(int) * npp);
  At(&d_sb, sizeof(int) * npp);
  At(&d_pa, sizeof(int) * npp);
  At(&d_pb, sizeof(int) * npp);
  At(&d_exps, sizeof(double) * nptot);
  At(&d_coefs, sizeof(double) * nptot);
  if (rc == F12INT_OK) {
    cudaStream_t st = ctx->stream;
    cudaMemcpyAsync(B.d_shell_l, l, sizeof(int) * nshell, cudaMemcpyHostToDevice, st);
    cudaMemcpyAsync(B.d_centers, centers, sizeof(double) * 3 * nshell, cudaMemcpyHostToDevice, st);
    cudaMemcpyAsync(B.d_pair_start, B.pair_start.data(), sizeof(int) * B.pair_start.size(), cudaMemcpyHostToDevice, st);
    cudaMemcpyAsync(B.d_pp_eoff, eoff.data(), sizeof(int64_t) * npp, cudaMemcpyHostToDevice, st);
    cudaMemcpyAsync(d_sa, sa.data(), sizeof(int) * npp, cudaMemcpyHostToDevice, st);
    cudaMemcpyAsync(d_sb, sb.data(), sizeof(int) * npp, cudaMemcpyHostToDevice, st);
    cudaMemcpyAsync(d_pa, pa.data(), sizeof(int) * npp, cudaMemcpyHostToDevice, st);
    cudaMemcpyAsync(d_pb, pb.data(), sizeof(int) * npp, cudaMemcpyHostToDevice, st);
    cudaMemcpyAsync(d_exps, exps, sizeof(double) * nptot, cudaMemcpyHostToDevice, st);
    cudaMemcpyAsync(d_coefs, coefs, sizeof(double) * nptot, cudaMemcpyHostToDevice, st);
    int nb = (npp + 127) / 128;
    k_build_pairs<<<nb, 128, 0, st>>>(npp, d_sa, d_sb, d_pa, d_pb, B.d_centers, B.d_shell_l, d_exps, d_coefs,
                                      B.d_pp_p, B.d_pp_P, B.d_pp_ab, B.d_pp_eoff, B.d_epool);
    ctx->launches++;
    cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) rc = cuda_fail(e);
  }
  dfree(ctx, d_sa, sizeof(int) * npp);
  dfree(ctx, d_sb, sizeof(int) * npp);
  dfree(ctx, d_pa, sizeof(int) * npp);
  dfree(ctx, d_pb, sizeof(int) * npp);
  dfree(ctx, d_exps, sizeof(double) * nptot);
  dfree(ctx, d_coefs, sizeof(double) * nptot);
  if (rc != F12INT_OK) {
    cudaFree(B.d_shell_l);
    cudaFree(B.d_centers);
    cudaFree(B.d_pair_start);
    cudaFree(B.d_pp_p);
    cudaFree(B.d_pp_P);
    cudaFree(B.d_pp_ab);
    cudaFree(B.d_pp_eoff);
    cudaFree(B.d_epool);
    ctx->used -= std::min(ctx->used, B.bytes);
    return rc;
  }
  B.exp_lo = *std::min_element(exps, exps + nptot);
  B.exp_hi = *std::max_element(exps, exps + nptot);
  {
    // every primitive centre lies between two shells: the diagonal of the
    // box of the shells bounds their distances
    double d2 = 0.0;
    for (int k = 0; k < 3; ++k) {
      double lo = centers[k], hi = centers[k];
      for (int i = 1; i < nshell; ++i) {
        lo = std::min(lo, centers[3 * i + k]);
        hi = std::max(hi, centers[3 * i + k]);
      }
      d2 += (hi - lo) * (hi - lo);
    }
    B.dmax = std::sqrt(d2);
  }
  mark_grid(ctx, B);
  ctx->bases.push_back(std::move(B));
  *basis_id = (int)ctx->bases.size() - 1;
  return F12INT_OK;
}

static int ensure_buf(f12int_ctx *ctx, void **p, size_t *cap, size_t bytes) {
  if (*cap >= bytes) return F12INT_OK;
  if (*p) {
    cudaFree(*p);
    ctx->used -= std::min(ctx->used, *cap);
    *p = nullptr;
    *cap = 0;
  }
  size_t want = std::max(bytes, (size_t)1 << 16);
  int rc = dalloc(ctx, (char **)p, want);
  if (rc == F12INT_OK) *cap = want;
  return rc;
}

static std::pair<cudaEvent_t, cudaEvent_t> take_events(f12int_ctx *ctx) {
  if (!ctx->ev_pool.empty()) {
    auto e = ctx->ev_pool.back();
    ctx->ev_pool.pop_back();
    return e;
  }
  std::pair<cudaEvent_t, cudaEvent_t> e{nullptr, nullptr};
  cudaEventCreate(&e.first);
  cudaEventCreate(&e.second);
  return e;
}

// After the stream has drained: add the timed launches to the totals.
static void collect_events(f12int_ctx *ctx) {
  for (auto &e : ctx->ev_aux) {
    float ms = 0.f;
    if (cudaEventElapsedTime(&ms, e.first, e.second) == cudaSuccess) ctx->aux_ms += ms;
    ctx->ev_pool.push_back(e);
  }
  for (auto &e : ctx->ev_con) {
    float ms = 0.f;
    if (cudaEventElapsedTime(&ms, e.first, e.second) == cudaSuccess) ctx->contract_ms += ms;
    ctx->ev_pool.push_back(e);
  }
  ctx->ev_aux.clear();
  ctx->ev_con.clear();
}

// items of the auxiliary stage per chunk (bounds the scratch memory)
static const int64_t kItemChunk = (int64_t)32 << 20;
// doubles of Hermite rows per chunk (1 GB)
static const int64_t kRowChunk = (int64_t)128 << 20;
static const int kNKeys = MAXFAM * (LAUX + 1) * NZBIN + 1;

}  // extern "C"

// Work one contraction block should carry at most, in multiply-adds: a longer
// one would keep an SM busy while the others idle at the end of a launch.
constexpr double kTaskFmas = 2e6;

// A block of this many cycles (0.5 ms) is long enough for the order of launches
// to matter.
constexpr double kPoleCycles = 1e6;

// A planned list: quartets in the working order -- those of the general
// contraction first, by launch group (precision, threads, shared memory within
// a factor of two), then decreasing work per task (the longest blocks start
// first), then the thin ones by class key -- and the launches over them.
struct ListPlan {
  struct Group {           // quartets [first, end) of one launch
    int64_t first, end;
    int nthr;
    size_t smem;
    bool fp32;
    int thin;              // class key, or -1
    double longest, warps; // estimated cycles of its longest block, and of all its warps together
  };
  std::vector<Group> groups;
  int64_t n = 0, nthin = 0;            // quartets; first thin one
  // runs of quartets of one kind, in the working order
  struct Run {
    int64_t first, count, npq, npab, pitch;   // primitive quartets, outer pairs and row doubles of one quartet
    int64_t pq0, row0, task0;                 // of the first
    int nsplit;
    bool swap, thin;
  };
  std::vector<Run> runs, kind_run;            // (kind_run: by the index in kid)
  int64_t ntask = 0, npq = 0, nrow = 0;       // totals
  int64_t big_pq = 1, big_row = 1;            // largest quartet, largest bra pair's rows
  std::vector<int32_t> kid;                   // kind of every quartet of the list
  std::vector<std::vector<int64_t>> at;       // per part of the list and kind: where its quartets go
  // filled by plan_fill
  int32_t *quartets = nullptr;                // [4 n]
  int64_t *offsets = nullptr, *pqoff = nullptr, *rowoff = nullptr;   // [n], [n + 1], [nthin + 1] (may be null)
  CTask *tasks = nullptr;                     // [ntask], quartet by quartet
  const Run &run_of(int64_t q) const {
    size_t lo = 0, hi = runs.size() - 1;
    while (lo < hi) {
      const size_t mid = (lo + hi + 1) / 2;
      if (runs[mid].first <= q) lo = mid;
      else hi = mid - 1;
    }
    return runs[lo];
  }
  int64_t tfirst(int64_t q) const {
    if (q >= n) return ntask;
    const Run &r = run_of(q);
    return r.task0 + (q - r.first) * r.nsplit;
  }
};

// Plans the list hq0.  fp32(s): the mixed path's choice for quartet s; fewest:
// as few tasks as fit in shared memory.  Returns F12INT_EINVAL for a shell index
// out of range.  Every quartet of the same kind (types of the four shells, FP32
// or not) has the same plan: the kinds are planned once, ordered, and the
// quartets placed run by run in their list order (a counting sort, its passes
// over the list on several cores when it is long).
template <class Fp32>
static int plan_kinds(const f12int_ctx::BasisData &B, int cls, int64_t n, const int32_t *hq0, Fp32 fp32, ListPlan &P,
                      bool fewest = false) {
  struct Kind {
    int64_t key;
    int la, lb, lc, ld, f32;
    int64_t nab, ncd, count, first;
    bool thin, swap;   // swap: listed as (cd|ab), the bra inner
    ContractShape shape;
    ContractPlan pl;
    double work;
    int tier;
  };
  std::vector<Kind> kinds;
  P = ListPlan{};
  P.n = n;
  const int ns = B.nshell;
  const int64_t T = (int64_t)B.type_l.size();
  double total = 0.0;   // multiply-adds of the general contraction
  auto make_kind = [&](int64_t code) {
    Kind k{};
    k.key = code;
    k.f32 = (int)(code & 1);
    int64_t c = code >> 1;
    int t[4];
    for (int i = 3; i >= 0; --i) {
      t[i] = (int)(c % T);
      c /= T;
    }
    k.la = B.type_l[(size_t)t[0]];
    k.lb = B.type_l[(size_t)t[1]];
    k.lc = B.type_l[(size_t)t[2]];
    k.ld = B.type_l[(size_t)t[3]];
    k.nab = (int64_t)B.type_nprim[(size_t)t[0]] * B.type_nprim[(size_t)t[1]];
    k.ncd = (int64_t)B.type_nprim[(size_t)t[2]] * B.type_nprim[(size_t)t[3]];
    k.thin = thin_quartet(k.la << 6 | k.lb << 4 | k.lc << 2 | k.ld, cls);
    k.swap = !k.thin && bra_inner(k.la, k.lb, k.lc, k.ld, cls, k.nab, k.ncd);
    k.shape = contract_shape(k.la, k.lb, k.lc, k.ld, cls, k.swap);
    if (k.swap) std::swap(k.nab, k.ncd);   // outer, inner
    kinds.push_back(k);
  };
  // code of a quartet, -1 for a shell out of range
  auto code_of = [&](const int32_t *s) -> int64_t {
    for (int k = 0; k < 4; ++k)
      if (s[k] < 0 || s[k] >= ns) return -1;
    const int *t = B.type.data();
    const int64_t c = ((t[s[0]] * T + t[s[1]]) * T + t[s[2]]) * T + t[s[3]];
    const bool thin = thin_quartet(B.l[s[0]] << 6 | B.l[s[1]] << 4 | B.l[s[2]] << 2 | B.l[s[3]], cls);
    return 2 * c + (thin ? 0 : fp32(s));   // (the thin kernel is FP64)
  };
  P.kid.resize((size_t)n);
  const int parts = n >= 65536 ? 8 : 1;
  auto part_begin = [&](int t) { return n * t / parts; };
  const double ncode = 2.0 * (double)T * (double)T * (double)T * (double)T;
  if (ncode <= std::max(4096.0, 4.0 * (double)n)) {
    std::vector<unsigned char> seen((size_t)ncode, 0);
    std::atomic<bool> bad{false};
    parallel_for(parts, [&](int t) {
      for (int64_t i = part_begin(t); i < part_begin(t + 1); ++i) {
        const int64_t c = code_of(hq0 + 4 * i);
        if (c < 0) {
          bad = true;
          return;
        }
        P.kid[(size_t)i] = (int32_t)c;
        if (!__atomic_load_n(&seen[(size_t)c], __ATOMIC_RELAXED)) __atomic_store_n(&seen[(size_t)c], 1, __ATOMIC_RELAXED);
      }
    });
    if (bad) return F12INT_EINVAL;
    std::vector<int32_t> map((size_t)ncode, -1);
    for (size_t c = 0; c < seen.size(); ++c)
      if (seen[c]) {
        map[c] = (int32_t)kinds.size();
        make_kind((int64_t)c);
      }
    P.at.assign((size_t)parts, std::vector<int64_t>(kinds.size(), 0));
    parallel_for(parts, [&](int t) {
      std::vector<int64_t> &cnt = P.at[(size_t)t];
      for (int64_t i = part_begin(t); i < part_begin(t + 1); ++i) {
        int32_t &k = P.kid[(size_t)i];
        k = map[(size_t)k];
        ++cnt[(size_t)k];
      }
    });
  } else {   // a short list of many types of shells: open-addressing map from code to kind
    std::vector<int64_t> slot_key(4096, -1);
    std::vector<int32_t> slot_val(4096, -1);
    size_t mask = slot_key.size() - 1;
    auto find = [&](const std::vector<int64_t> &keys, size_t m, int64_t key) {
      size_t h = (size_t)((uint64_t)key * 0x9E3779B97F4A7C15ull >> 40) & m;
      while (keys[h] != -1 && keys[h] != key) h = (h + 1) & m;
      return h;
    };
    for (int64_t i = 0; i < n; ++i) {
      const int64_t key = code_of(hq0 + 4 * i);
      if (key < 0) return F12INT_EINVAL;
      size_t h = find(slot_key, mask, key);
      if (slot_key[h] == -1) {
        if (kinds.size() * 2 >= slot_key.size()) {   // grow and rehash
          std::vector<int64_t> nk(slot_key.size() * 2, -1);
          std::vector<int32_t> nv(slot_key.size() * 2, -1);
          for (size_t t = 0; t < slot_key.size(); ++t)
            if (slot_key[t] != -1) {
              const size_t g = find(nk, nk.size() - 1, slot_key[t]);
              nk[g] = slot_key[t];
              nv[g] = slot_val[t];
            }
          slot_key.swap(nk);
          slot_val.swap(nv);
          mask = slot_key.size() - 1;
          h = find(slot_key, mask, key);
        }
        slot_key[h] = key;
        slot_val[h] = (int32_t)kinds.size();
        make_kind(key);
      }
      P.kid[(size_t)i] = slot_val[h];
    }
    P.at.assign((size_t)parts, std::vector<int64_t>(kinds.size(), 0));
    parallel_for(parts, [&](int t) {
      for (int64_t i = part_begin(t); i < part_begin(t + 1); ++i) ++P.at[(size_t)t][(size_t)P.kid[(size_t)i]];
    });
  }
  for (size_t k = 0; k < kinds.size(); ++k)
    for (const auto &c : P.at) kinds[k].count += c[k];
  for (const Kind &k : kinds)
    if (!k.thin) total += (double)k.count * (double)(k.nab * k.ncd) * task_fmas(k.shape, k.ncd, k.shape.ncd());
  // about a dozen tasks per SM where the list has the work for it (a block's
  // result does not depend on how a quartet is cut into ranges)
  const double target = fewest ? 1e300 : std::min(kTaskFmas, std::max(5e4, total / (kSMs * 12)));
  for (Kind &k : kinds) {
    k.pl = ContractPlan{32, 1, 0};
    if (k.thin) {
      k.work = (double)(k.nab * k.ncd);
      continue;
    }
    k.pl = contract_plan(k.shape, k.nab * k.ncd, k.ncd, k.f32 ? 4 : 8, target, fewest);
    if (k.pl.smem == 0) return F12INT_EINVAL;
    k.work = (double)(k.nab * k.ncd) * task_fmas(k.shape, k.ncd, (k.shape.ncd() + k.pl.nsplit - 1) / k.pl.nsplit);
    k.tier = 0;
    while (((size_t)8192 << k.tier) < k.pl.smem) ++k.tier;
  }
  std::vector<int32_t> order(kinds.size());
  for (size_t g = 0; g < kinds.size(); ++g) order[g] = (int32_t)g;
  std::sort(order.begin(), order.end(), [&](int32_t x, int32_t y) {
    const Kind &a = kinds[(size_t)x], &b = kinds[(size_t)y];
    if (a.thin != b.thin) return b.thin;
    const int ka = a.la << 6 | a.lb << 4 | a.lc << 2 | a.ld, kb = b.la << 6 | b.lb << 4 | b.lc << 2 | b.ld;
    if (a.thin) return ka != kb ? ka < kb : (a.work != b.work ? a.work > b.work : a.key < b.key);
    if (a.f32 != b.f32) return a.f32 < b.f32;
    if (a.tier != b.tier) return a.tier > b.tier;
    if (a.pl.nthr != b.pl.nthr) return a.pl.nthr > b.pl.nthr;
    if (a.work != b.work) return a.work > b.work;
    return a.key < b.key;
  });
  int64_t run = 0;
  std::vector<int32_t> place(kinds.size());   // kind -> run
  for (size_t at = 0; at < order.size(); ++at) {
    Kind &k = kinds[(size_t)order[at]];
    const int thin = k.thin ? k.la << 6 | k.lb << 4 | k.lc << 2 | k.ld : -1;
    if (P.groups.empty() || P.groups.back().thin != thin ||
        (!k.thin && (P.groups.back().fp32 != (k.f32 != 0) || P.groups.back().nthr != k.pl.nthr ||
                     kinds[(size_t)order[at - 1]].tier != k.tier)))
      P.groups.push_back(ListPlan::Group{run, run, k.pl.nthr, 0, k.f32 != 0, thin, 0.0, 0.0});
    ListPlan::Group &G = P.groups.back();
    G.smem = std::max(G.smem, k.pl.smem);
    // cycles of a block (a thin quartet's warp): a primitive quartet's staging or
    // grid point, and the chain of a thread's multiply-adds
    const double cycles = k.thin ? 650.0 * (double)(k.nab * k.ncd + 31)
                                 : 300.0 * (double)(k.nab * k.ncd) + 150.0 * k.work / k.pl.nthr;
    G.longest = std::max(G.longest, cycles);
    G.warps += cycles * (double)(k.count * k.pl.nsplit) * (k.thin ? 1.0 : k.pl.nthr / 32.0);
    k.first = run;
    ListPlan::Run r{};
    r.first = run;
    r.count = k.count;
    r.npq = k.nab * k.ncd;
    r.npab = k.nab;
    r.pitch = k.thin ? 0 : r.npq * row_pitch(k.shape.L());
    r.pq0 = P.npq;
    r.row0 = P.nrow;
    r.task0 = P.ntask;
    r.nsplit = k.pl.nsplit;
    r.swap = k.swap;
    r.thin = k.thin;
    place[(size_t)order[at]] = (int32_t)P.runs.size();
    P.runs.push_back(r);
    run += k.count;
    P.npq += k.count * r.npq;
    P.nrow += k.count * r.pitch;
    P.ntask += k.count * r.nsplit;
    P.big_pq = std::max(P.big_pq, r.npq);
    if (!k.thin) P.big_row = std::max(P.big_row, r.pitch / r.npab);
    G.end = run;
    if (!k.thin) P.nthin = run;
  }
  // where each part of the list puts its quartets of a kind
  for (size_t k = 0; k < kinds.size(); ++k) {
    int64_t pos = kinds[k].first;
    for (auto &c : P.at) {
      const int64_t cnt = c[k];
      c[k] = pos;
      pos += cnt;
    }
  }
  // (the arrays stay by kind: runs of a kind are found through place)
  {
    std::vector<ListPlan::Run> by_kind(P.runs.size());
    for (size_t k = 0; k < kinds.size(); ++k) by_kind[k] = P.runs[(size_t)place[k]];
    P.kind_run.swap(by_kind);
  }
  return F12INT_OK;
}

// Writes the planned list into the caller's arrays.
static void plan_fill(ListPlan &P, const int32_t *hq0, const int64_t *ho0, int32_t *quartets, int64_t *offsets,
                      int64_t *pqoff, int64_t *rowoff, CTask *tasks) {
  P.quartets = quartets;
  P.offsets = offsets;
  P.pqoff = pqoff;
  P.rowoff = rowoff;
  P.tasks = tasks;
  const int parts = (int)P.at.size();
  parallel_for(parts, [&](int t) {
    std::vector<int64_t> &at = P.at[(size_t)t];
    for (int64_t i = P.n * t / parts; i < P.n * (t + 1) / parts; ++i) {
      const size_t k = (size_t)P.kid[(size_t)i];
      const ListPlan::Run &r = P.kind_run[k];
      const int64_t q = at[k]++, in = q - r.first;
      const int flip = r.swap ? 2 : 0;
      for (int c = 0; c < 4; ++c) quartets[4 * q + c] = hq0[4 * i + (c ^ flip)];
      offsets[q] = ho0[i];
      pqoff[q] = r.pq0 + in * r.npq;
      if (rowoff && !r.thin) rowoff[q] = r.row0 + in * r.pitch;
      CTask *tk = tasks + r.task0 + in * r.nsplit;
      const int16_t mark = (int16_t)(r.swap ? -r.nsplit : r.nsplit);
      for (int sp = 0; sp < r.nsplit; ++sp) tk[sp] = CTask{(int32_t)q, (int16_t)sp, mark};
    }
  });
  pqoff[P.n] = P.npq;
  if (rowoff) rowoff[P.nthin] = P.nrow;
}

// Device arrays that a planned list runs with.
struct ListBufs {
  const int32_t *quartets;
  const int64_t *offsets, *pqoff, *rowoff;
  const CTask *tasks;
  int *keys;
  unsigned *order, *hist;
  double *part, *rows;
  int64_t keys_cap, part_cap, rows_cap;   // ints, doubles, doubles
  int64_t part_thin;                      // doubles of D.part when no rows are in use
  int pitch = 0;                          // > 0: every row takes so many doubles (rowoff unused)
};

// Queue the list's kernels on st: the thin contraction, and chunk by chunk of
// the general one the auxiliary functions, the Hermite rows and the
// contraction.  F12INT_ENOMEM when the buffers do not hold one
// bra primitive pair of a general quartet, or one thin quartet.
static int launch_list(f12int_ctx *ctx, const ListPlan &P, const ListBufs &D, const PairView &PV, const GridView &G,
                       int cls, double *out_dev, cudaStream_t st, bool timing) {
  const int nf = ctx->tables.nfam[cls == 5 ? 3 : cls];
  QuartetView QV{D.quartets, D.pqoff, P.n, nullptr, nullptr, nullptr, nullptr};
  const bool direct = G.direct();
  unsigned long long *fma_aux = timing ? ctx->d_fma : nullptr, *fma_con = timing ? ctx->d_fma + 1 : nullptr;
  std::pair<cudaEvent_t, cudaEvent_t> ev{nullptr, nullptr};
  auto time_begin = [&] {
    if (!timing) return;
    ev = take_events(ctx);
    cudaEventRecord(ev.first, st);
  };
  auto time_end = [&](bool aux) {
    if (!timing) return;
    cudaEventRecord(ev.second, st);
    (aux ? ctx->ev_aux : ctx->ev_con).push_back(ev);
    (aux ? ctx->aux_launches : ctx->contract_launches)++;
  };
  // The independent launches go round the side streams between fork and join.
  // Launches whose longest block takes a good part of the whole list's time
  // (quartets of thousands of primitive quartets and few entries: a few blocks of
  // milliseconds each) go first, and every launch then to the stream with the
  // least before it: in the list's order, smallest blocks last, they had the GPU
  // to themselves in the end (2000 mixed I4 quartets of one molecule 20.4 ms, so 18.2; 3000 f-shell
  // I2 quartets 3.18 and 3.04).  Lists without such launches keep their order
  // (sorting every launch by its longest block: 17.6 and 3.24 ms).
  double all_warps = 0.0;
  for (const ListPlan::Group &g : P.groups) all_warps += g.warps;
  const double pole = 0.25 * all_warps / (kSMs * 16);   // cycles, at 16 warps an SM
  auto is_pole = [&](const ListPlan::Group &g) { return g.longest > std::max(pole, kPoleCycles); };
  bool poles = false;
  std::vector<int> launch_order;
  for (int pass = 0; pass < 2; ++pass)
    for (size_t i = 0; i < P.groups.size(); ++i)
      if (is_pole(P.groups[i]) == (pass == 0)) {
        launch_order.push_back((int)i);
        poles = poles || pass == 0;
      }
  unsigned used = 0;            // side streams that carry launches since the last join
  unsigned waits = 0;           // ... that wait for the last fork
  double load[NSIDE] = {0.0};
  auto fork = [&] {
    waits = 0;
    if (!poles) std::fill(load, load + NSIDE, 0.0);
    return cudaEventRecord(ctx->fork, st) == cudaSuccess;
  };
  auto side = [&](const ListPlan::Group &g) -> cudaStream_t {
    const int i = (int)(std::min_element(load, load + NSIDE) - load);
    load[i] += poles ? std::max(g.longest, g.warps / (kSMs * 16)) : 1.0;
    if (!(waits >> i & 1)) cudaStreamWaitEvent(ctx->side[i], ctx->fork, 0);
    waits |= 1u << i;
    used |= 1u << i;
    return ctx->side[i];
  };
  auto join = [&] {
    for (int i = 0; i < NSIDE; ++i)
      if (used >> i & 1) {
        cudaEventRecord(ctx->join[i], ctx->side[i]);
        cudaStreamWaitEvent(st, ctx->join[i], 0);
      }
    used = 0;
    std::fill(load, load + NSIDE, 0.0);
  };
  // items of the primitive quartets [pq0, pq1), family by family, into D.part
  auto items = [&](int64_t pq0, int64_t pq1) -> int {
    const int64_t nitems = (pq1 - pq0) * nf;
    CK(cudaMemsetAsync(D.hist, 0, sizeof(unsigned) * kNKeys, st));
    const unsigned nb = (unsigned)((nitems + BLOCK_AUX - 1) / BLOCK_AUX);
    const unsigned nbq = (unsigned)((pq1 - pq0 + BLOCK_AUX - 1) / BLOCK_AUX);
    k_items_classify<false><<<nbq, BLOCK_AUX, 0, st>>>(ctx->tables, PV, QV, cls, pq0, nitems, D.keys, D.hist);
    k_items_scan<<<1, 1024, 0, st>>>(D.hist, kNKeys);
    k_items_scatter<<<nb, BLOCK_AUX, 0, st>>>(QV, nf, pq0, D.keys, D.hist, nitems, D.order);
    time_begin();
    k_items_eval<false><<<nb, BLOCK_AUX, 0, st>>>(ctx->tables, PV, QV, cls, pq0, nitems, D.order, D.keys, D.part,
                                                  ctx->d_status, fma_aux);
    if (ctx->cls_quad[cls]) {
      k_items_eval<false, true><<<nb, BLOCK_AUX, 0, st>>>(ctx->tables, PV, QV, cls, pq0, nitems, D.order, D.keys,
                                                          D.part, ctx->d_status, fma_aux);
      ctx->launches++;
    }
    time_end(true);
    ctx->launches += 4;
    CK(cudaGetLastError());
    return F12INT_OK;
  };
  // thin quartets [qa, qb) of the list; pq0: the first primitive quartet of D.part
  auto thin = [&](int64_t qa, int64_t qb, int64_t pq0) -> int {
    for (int gi : launch_order) {
      const ListPlan::Group &g = P.groups[(size_t)gi];
      const int64_t a = std::max(qa, g.first), b = std::min(qb, g.end);
      if (g.thin < 0 || a >= b) continue;
      const ThinKernel kern = thin_kernel(g.thin, cls == 5);
      if (!kern) return F12INT_EINVAL;
      const int64_t nt = b - a;   // one task each
      kern<<<(unsigned)((nt + kThinWarps - 1) / kThinWarps), 32 * kThinWarps, 0, side(g)>>>(
          PV, QV, direct ? 1 : nf, pq0, G, D.tasks + P.tfirst(a), nt, nullptr, D.keys, D.part, out_dev,
          D.offsets, fma_con);
      ctx->launches++;
      CK(cudaGetLastError());
    }
    return F12INT_OK;
  };
  // general quartets [qa, qb), bra primitive pairs [i0, i1) (-1: all); row0: the
  // first double of D.rows
  auto general = [&](int64_t qa, int64_t qb, int64_t pq0, int64_t row0, int i0, int i1) -> int {
    for (int gi : launch_order) {
      const ListPlan::Group &g = P.groups[(size_t)gi];
      const int64_t a = std::max(qa, g.first), b = std::min(qb, g.end);
      if (g.thin >= 0 || a >= b) continue;
      const int64_t t0 = P.tfirst(a), nt = P.tfirst(b) - t0;
      const auto kern = g.fp32 ? k_contract<false, float> : k_contract<false, double>;
      if (g.smem > 48 * 1024)
        CK(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemMax));   // (one value for every thread)
      kern<<<(unsigned)nt, g.nthr, g.smem, side(g)>>>(PV, QV, cls, direct ? 1 : nf, pq0, D.tasks + t0, nt, nullptr,
                                                     D.keys, RowView{D.rows, D.rowoff, row0, D.pitch}, out_dev,
                                                     D.offsets, i0, i1, fma_con);
      ctx->launches++;
      CK(cudaGetLastError());
    }
    return F12INT_OK;
  };
  auto hermite = [&](int64_t pq0, int64_t pq1, int64_t row0, int64_t part0) -> int {
    const unsigned nb = (unsigned)((pq1 - pq0 + BLOCK_AUX - 1) / BLOCK_AUX);
    if (direct) {
      time_begin();
      k_hermite_rows<false, true><<<nb, BLOCK_AUX, 0, st>>>(G, PV, QV, cls, 1, pq0, pq1 - pq0, D.keys, nullptr,
                                                            RowView{D.rows, D.rowoff, row0, D.pitch}, fma_aux);
      time_end(true);
    } else {
      k_hermite_rows<false, false><<<nb, BLOCK_AUX, 0, st>>>(G, PV, QV, cls, nf, pq0, pq1 - pq0,
                                                             D.keys + (pq0 - part0) * nf,
                                                             D.part + (pq0 - part0) * nf * kPartPitch,
                                                             RowView{D.rows, D.rowoff, row0, D.pitch}, nullptr);
    }
    ctx->launches++;
    CK(cudaGetLastError());
    return F12INT_OK;
  };
  int rc = F12INT_OK;
  if (direct) {
    // the thin contraction needs none of the rows: it runs beside them
    if (P.nthin < P.n) {
      if (!fork()) return F12INT_ECUDA;
      time_begin();
      rc = thin(P.nthin, P.n, 0);
      if (P.nthin == 0 || timing) join();
      time_end(false);
      if (rc != F12INT_OK) return rc;
    }
  }
  // first double of the rows of quartet q, and their end, in the list's order
  auto row_of = [&](int64_t q) -> int64_t { return D.pitch ? P.pqoff[q] * D.pitch : P.rowoff[q]; };
  auto row_end = [&](int64_t q) -> int64_t { return D.pitch ? P.pqoff[q + 1] * D.pitch : P.rowoff[q + 1]; };
  const int64_t per_pq = (int64_t)std::max(nf, 1) * kPartPitch;
  const int64_t fit = direct ? (int64_t)1 << 60 : D.part_cap / per_pq;          // primitive quartets whose items fit
  int64_t part0 = 0, part1 = 0;   // family path: primitive quartets whose items are in D.part
  for (int64_t qa = 0; qa < P.nthin && rc == F12INT_OK;) {
    const int64_t pq0 = P.pqoff[qa], npq = P.pqoff[qa + 1] - pq0, row0 = row_of(qa);
    const bool fits = row_end(qa) - row0 <= D.rows_cap && npq <= fit && (!direct || npq <= D.keys_cap);
    if (fits) {
      if (!direct && pq0 >= part1) {   // items of as many quartets as fit
        int64_t qe = qa + 1;
        while (qe < P.nthin && P.pqoff[qe + 1] - pq0 <= fit) ++qe;
        part0 = pq0;
        part1 = P.pqoff[qe];
        rc = items(part0, part1);
        if (rc != F12INT_OK) break;
      }
      int64_t qb = qa + 1;
      while (qb < P.nthin && row_end(qb) - row0 <= D.rows_cap &&
             (direct ? P.pqoff[qb + 1] - pq0 <= D.keys_cap : P.pqoff[qb + 1] <= part1))
        ++qb;
      rc = hermite(pq0, P.pqoff[qb], row0, part0);
      if (rc == F12INT_OK && !fork()) rc = F12INT_ECUDA;
      if (rc != F12INT_OK) break;
      time_begin();
      rc = general(qa, qb, direct ? pq0 : part0, row0, -1, -1);
      join();
      time_end(false);
      qa = qb;
      continue;
    }
    // one quartet larger than the scratch: a few of its bra primitive pairs at a time
    const int64_t npab = P.run_of(qa).npab;
    const int64_t npcd = npq / npab, per = (row_end(qa) - row0) / npab;   // doubles of one bra pair's rows
    int64_t step = std::min<int64_t>(D.rows_cap / per, fit / npcd);
    if (direct) step = std::min<int64_t>(step, D.keys_cap / npcd);
    if (step < 1) return F12INT_ENOMEM;
    for (int64_t i0 = 0; i0 < npab && rc == F12INT_OK; i0 += step) {
      const int64_t i1 = std::min(npab, i0 + step), a = pq0 + i0 * npcd, b = pq0 + i1 * npcd;
      if (!direct) rc = items(a, b);
      if (rc == F12INT_OK) rc = hermite(a, b, row0 + i0 * per, a);
      if (rc == F12INT_OK && !fork()) rc = F12INT_ECUDA;
      if (rc != F12INT_OK) break;
      time_begin();
      rc = general(qa, qa + 1, a, row0 + i0 * per, (int)i0, (int)i1);
      join();
      time_end(false);
    }
    part1 = 0;
    ++qa;
  }
  for (int64_t qa = P.nthin; !direct && qa < P.n && rc == F12INT_OK;) {   // family path: the thin quartets
    const int64_t pq0 = P.pqoff[qa], most = D.part_thin / per_pq;
    int64_t qb = qa + 1;
    while (qb < P.n && P.pqoff[qb + 1] - pq0 <= most) ++qb;
    if (P.pqoff[qb] - pq0 > most) return F12INT_ENOMEM;
    rc = items(pq0, P.pqoff[qb]);
    if (rc == F12INT_OK && !fork()) rc = F12INT_ECUDA;
    if (rc != F12INT_OK) break;
    time_begin();
    rc = thin(qa, qb, pq0);
    join();
    time_end(false);
    qa = qb;
  }
  join();   // (an error's or a thin launch's that is still on a side stream)
  return rc;
}

extern "C" {

// Primitive Schwarz factors Q_ab = sqrt(max |(ab|k|ab)|) of every primitive
// pair of the basis for class cls (the I3 kernel for I5), from the diagonal
// blocks of a basis in which every primitive is its own shell.
static int ensure_prim_bounds(f12int_ctx *ctx, int basis_id, int cls) {
  std::lock_guard<std::recursive_mutex> blk(ctx->bounds_mu);
  {
    f12int_ctx::BasisData &B = ctx->bases[basis_id];
    if (!B.prim_screen || B.d_qprim[cls]) return F12INT_OK;
  }
  const int dcls = cls == 5 ? 3 : cls;
  std::vector<double> cen, ex, co;
  std::vector<int> ll, np1;
  std::vector<int> poff;
  int nprim_tot = 0;
  {
    const f12int_ctx::BasisData &B = ctx->bases[basis_id];
    for (int s = 0; s < B.nshell; ++s) {
      poff.push_back(nprim_tot);
      for (int k = 0; k < B.nprim[s]; ++k) {
        cen.insert(cen.end(), {B.centers[3 * s], B.centers[3 * s + 1], B.centers[3 * s + 2]});
        ll.push_back(B.l[s]);
        np1.push_back(1);
        ex.push_back(B.exps[nprim_tot]);
        co.push_back(B.coefs[nprim_tot]);
        ++nprim_tot;
      }
    }
  }
  int pid = -1;
  int rc = f12int_set_basis(ctx, nprim_tot, cen.data(), ll.data(), np1.data(), ex.data(), co.data(), &pid);
  if (rc != F12INT_OK) return rc;
  ctx->bases[pid].prim_screen = false;
  std::vector<int32_t> hq;
  std::vector<int64_t> off;
  int64_t tot = 0;
  for (int a = 0; a < nprim_tot; ++a)
    for (int b = 0; b <= a; ++b) {
      hq.insert(hq.end(), {a, b, a, b});
      off.push_back(tot);
      int nab = ncart(ll[a]) * ncart(ll[b]);
      tot += (int64_t)nab * nab;
    }
  const int64_t nq = (int64_t)off.size();
  int32_t *dq = nullptr;
  int64_t *doff = nullptr;
  double *dout = nullptr;
  std::vector<double> hout((size_t)tot);
  rc = dalloc(ctx, &dq, sizeof(int32_t) * hq.size());
  if (rc == F12INT_OK) rc = dalloc(ctx, &doff, sizeof(int64_t) * nq);
  if (rc == F12INT_OK) rc = dalloc(ctx, &dout, sizeof(double) * tot);
  cudaStream_t st = ctx->stream;
  if (rc == F12INT_OK &&
      (cudaMemcpyAsync(dq, hq.data(), sizeof(int32_t) * hq.size(), cudaMemcpyHostToDevice, st) != cudaSuccess ||
       cudaMemcpyAsync(doff, off.data(), sizeof(int64_t) * nq, cudaMemcpyHostToDevice, st) != cudaSuccess))
    rc = F12INT_ECUDA;
  if (rc == F12INT_OK) rc = f12int_compute_class(ctx, pid, dcls, dq, nq, dout, doff, st);
  if (rc == F12INT_OK &&
      (cudaMemcpyAsync(hout.data(), dout, sizeof(double) * tot, cudaMemcpyDeviceToHost, st) != cudaSuccess ||
       cudaStreamSynchronize(st) != cudaSuccess))
    rc = F12INT_ECUDA;
  dfree(ctx, dq, sizeof(int32_t) * hq.size());
  dfree(ctx, doff, sizeof(int64_t) * nq);
  dfree(ctx, dout, sizeof(double) * tot);
  // release the per-primitive basis (it is the last one)
  {
    f12int_ctx::BasisData &P = ctx->bases[pid];
    cudaFree(P.d_shell_l);
    cudaFree(P.d_centers);
    cudaFree(P.d_pair_start);
    cudaFree(P.d_pp_p);
    cudaFree(P.d_pp_P);
    cudaFree(P.d_pp_ab);
    cudaFree(P.d_pp_eoff);
    cudaFree(P.d_epool);
    ctx->used -= std::min(ctx->used, P.bytes);
    if (pid == (int)ctx->bases.size() - 1) ctx->bases.pop_back();
  }
  if (rc != F12INT_OK) return rc;
  std::vector<double> qps((size_t)nprim_tot * nprim_tot, 0.0);
  int64_t k = 0;
  for (int a = 0; a < nprim_tot; ++a)
    for (int b = 0; b <= a; ++b, ++k) {
      int nab = ncart(ll[a]) * ncart(ll[b]);
      double m = 0.0;
      for (int64_t i = 0; i < (int64_t)nab * nab; ++i) m = std::max(m, std::fabs(hout[off[k] + i]));
      qps[(size_t)a * nprim_tot + b] = qps[(size_t)b * nprim_tot + a] = std::sqrt(m);
    }
  f12int_ctx::BasisData &B = ctx->bases[basis_id];
  const int npp = B.pair_start.back();
  std::vector<double> qpp((size_t)npp);
  for (int a = 0; a < B.nshell; ++a)
    for (int b = 0; b < B.nshell; ++b) {
      int i = B.pair_start[(size_t)a * B.nshell + b];
      for (int x = 0; x < B.nprim[a]; ++x)
        for (int y = 0; y < B.nprim[b]; ++y, ++i) qpp[i] = qps[(size_t)(poff[a] + x) * nprim_tot + poff[b] + y];
    }
  double *d = nullptr;
  rc = dalloc(ctx, &d, sizeof(double) * npp);
  if (rc != F12INT_OK) return rc;
  if (upload(d, qpp.data(), sizeof(double) * npp, ctx->stream) != cudaSuccess) {
    dfree(ctx, d, sizeof(double) * npp);
    return F12INT_ECUDA;
  }
  B.d_qprim[cls] = d;
  return F12INT_OK;
}

static int compute_class_impl(f12int_ctx *ctx, int basis_id, int cls, const int32_t *quartets_dev, int64_t n,
                              double *out_dev, const int64_t *offsets_dev, void *cuda_stream, double fp32_below,
                              bool prim_screen = true);
static int ensure_pair_bounds(f12int_ctx *ctx, int basis_id, int cls);

int f12int_compute_class(f12int_ctx *ctx, int basis_id, int cls, const int32_t *quartets_dev, int64_t n,
                         double *out_dev, const int64_t *offsets_dev, void *cuda_stream) {
  return compute_class_impl(ctx, basis_id, cls, quartets_dev, n, out_dev, offsets_dev, cuda_stream, 0.0);
}

int f12int_compute_class_mixed(f12int_ctx *ctx, int basis_id, int cls, const int32_t *quartets_dev, int64_t n,
                               double *out_dev, const int64_t *offsets_dev, double fp32_below, void *cuda_stream) {
  if (!(fp32_below >= 0.0)) return F12INT_EINVAL;
  return compute_class_impl(ctx, basis_id, cls, quartets_dev, n, out_dev, offsets_dev, cuda_stream, fp32_below);
}

}  // extern "C"

static int compute_class_impl(f12int_ctx *ctx, int basis_id, int cls, const int32_t *quartets_dev, int64_t n,
                              double *out_dev, const int64_t *offsets_dev, void *cuda_stream, double fp32_below,
                              bool prim_screen) {
  if (!ctx) return F12INT_EINVAL;
  if (cls < 1 || cls > 6 || n < 0) return F12INT_EINVAL;
  if (basis_id < 0 || basis_id >= (int)ctx->bases.size()) return F12INT_ENOTREADY;
  if (!ctx->factor_ready) return F12INT_ENOTREADY;
  if (!ctx->cls_ok[cls]) return F12INT_EDOMAIN;
  if (n == 0) return F12INT_OK;
  if (!quartets_dev || !out_dev || !offsets_dev) return F12INT_EINVAL;
  {
    int rc0 = ensure_prim_bounds(ctx, basis_id, cls);
    if (rc0 == F12INT_OK && fp32_below > 0.0) rc0 = ensure_pair_bounds(ctx, basis_id, cls);
    if (rc0 != F12INT_OK) return rc0;
  }
  std::lock_guard<std::mutex> lk(ctx->mu);
  CK(cudaSetDevice(ctx->device));
  const f12int_ctx::BasisData &B = ctx->bases[basis_id];
  cudaStream_t st = pick_stream(ctx, cuda_stream);
  NvtxRange call_range("f12int.compute_class");
  const auto t_plan0 = std::chrono::steady_clock::now();
  std::unique_ptr<NvtxRange> plan_range(new NvtxRange("f12int.plan"));
  // host staging: the list as given, then as planned (one copy each way)
  HostStage &hs = ctx->stage;
  if (!hs.reserve(24 * (size_t)n)) return F12INT_ENOMEM;
  CK(cudaMemcpyAsync(hs.p, quartets_dev, sizeof(int32_t) * 4 * n, cudaMemcpyDeviceToHost, st));
  CK(cudaMemcpyAsync(hs.p + 16 * n, offsets_dev, sizeof(int64_t) * n, cudaMemcpyDeviceToHost, st));
  CK(cudaStreamSynchronize(st));
  ListPlan P;
  // mixed path: contraction in FP32 below the bound
  int rc = plan_kinds(B, cls, n, (const int32_t *)hs.p, [&](const int32_t *s) {
    return fp32_below > 0.0 && screen_estimate(ctx, B, cls, s[0], s[1], s[2], s[3]) < fp32_below ? 1 : 0;
  }, P);
  if (rc != F12INT_OK) return rc;
  const ListLayout at(n, P.nthin, P.ntask);
  if (!hs.reserve(24 * (size_t)n + at.bytes, 24 * (size_t)n)) return F12INT_ENOMEM;
  unsigned char *list = hs.p + 24 * (size_t)n;
  plan_fill(P, (const int32_t *)hs.p, (const int64_t *)(hs.p + 16 * n), (int32_t *)list, (int64_t *)(list + at.offsets),
            (int64_t *)(list + at.pqoff), (int64_t *)(list + at.rowoff), (CTask *)(list + at.tasks));
  const GridView G = grid_view(ctx, B, cls);
  const int64_t nf = std::max(1, ctx->tables.nfam[cls == 5 ? 3 : cls]);
  const int64_t npq = P.npq, npq_gen = P.pqoff[P.nthin];
  const int64_t big_pq = P.big_pq, big_row = P.big_row;   // largest quartet, bra pair's rows
  rc = ensure_buf(ctx, (void **)&ctx->d_list, &ctx->list_cap, at.bytes);
  if (rc != F12INT_OK) return rc;
  ListBufs D{(const int32_t *)ctx->d_list, (const int64_t *)(ctx->d_list + at.offsets),
             (const int64_t *)(ctx->d_list + at.pqoff), (const int64_t *)(ctx->d_list + at.rowoff),
             (const CTask *)(ctx->d_list + at.tasks)};
  // scratch of one chunk: Hermite rows to kRowChunk doubles, on the family path
  // also the items; under a budget no more than an item per family would take
  const int64_t all_rows = P.nrow;
  if (G.direct()) {
    int64_t want = std::min(all_rows, kRowChunk);
    if (ctx->budget) want = std::min(want, npq * nf * 17);
    D.rows_cap = std::max(want, all_rows ? big_row : 0);
    D.keys_cap = std::min(npq_gen, std::max(D.rows_cap / 36 + 1, big_pq));
  } else {
    D.part_cap = std::min(npq, std::max(big_pq, kItemChunk / nf)) * nf * kPartPitch;
    D.part_thin = D.part_cap;
    D.keys_cap = D.part_cap / kPartPitch;
    D.rows_cap = std::max(std::min(all_rows, kRowChunk / 4), all_rows ? big_row : 0);
    rc = ensure_buf(ctx, (void **)&ctx->d_order, &ctx->order_cap, sizeof(unsigned) * (size_t)D.keys_cap);
    if (rc == F12INT_OK) rc = ensure_buf(ctx, (void **)&ctx->d_part, &ctx->part_cap, sizeof(double) * (size_t)D.part_cap);
    if (rc == F12INT_OK) rc = ensure_buf(ctx, (void **)&ctx->d_hist, &ctx->hist_cap, sizeof(unsigned) * kNKeys);
  }
  if (rc == F12INT_OK) rc = ensure_buf(ctx, (void **)&ctx->d_keys, &ctx->keys_cap, sizeof(int) * (size_t)D.keys_cap);
  if (rc == F12INT_OK) {
    rc = ensure_buf(ctx, (void **)&ctx->d_rows, &ctx->rows_cap, sizeof(double) * (size_t)D.rows_cap);
    while (rc == F12INT_ENOMEM && !G.direct() && D.rows_cap > big_row) {   // the family path's rows take what is left
      D.rows_cap = std::max(big_row, D.rows_cap / 4);
      rc = ensure_buf(ctx, (void **)&ctx->d_rows, &ctx->rows_cap, sizeof(double) * (size_t)D.rows_cap);
    }
  }
  if (rc != F12INT_OK) return rc;
  D.keys = ctx->d_keys;
  D.order = ctx->d_order;
  D.hist = ctx->d_hist;
  D.part = ctx->d_part;
  D.rows = ctx->d_rows;
  CK(cudaMemcpyAsync(ctx->d_list, list, at.bytes, cudaMemcpyHostToDevice, st));
  plan_range.reset();
  ctx->plan_ms += std::chrono::duration<double, std::milli>(std::chrono::steady_clock::now() - t_plan0).count();
  ctx->plan_calls++;
  rc = launch_list(ctx, P, D, pair_view(ctx, B, cls, B.prim_screen && prim_screen), G, cls, out_dev, st, ctx->timing);
  if (rc != F12INT_OK) {
    cudaStreamSynchronize(st);   // the queued copies read the staging buffer
    for (cudaStream_t t : ctx->side) cudaStreamSynchronize(t);
    return rc;
  }
  // keep the host buffer alive until the copy has been consumed
  CK(cudaStreamSynchronize(st));
  if (ctx->timing) collect_events(ctx);
  return F12INT_OK;
}

extern "C" {

int f12int_aux(f12int_ctx *ctx, int cls, int64_t npts, const double *xi_dev, const double *D_dev, int nmax,
               double *out_dev, void *cuda_stream) {
  if (!ctx || cls < 1 || cls > 6 || npts < 0 || nmax < 0 || nmax > LAUX) return F12INT_EINVAL;
  if (!ctx->factor_ready) return F12INT_ENOTREADY;
  if (!ctx->cls_ok[cls]) return F12INT_EDOMAIN;
  if (npts == 0) return F12INT_OK;
  if (!xi_dev || !D_dev || !out_dev) return F12INT_EINVAL;
  std::lock_guard<std::mutex> lk(ctx->mu);
  CK(cudaSetDevice(ctx->device));
  cudaStream_t st = pick_stream(ctx, cuda_stream);
  int64_t nb = (npts + BLOCK_AUX - 1) / BLOCK_AUX;
  const GridView G = class_view(ctx, cls);
  const unsigned char *ok = G.cells ? ctx->grid->ok[cls == 5 ? 3 : cls] : nullptr;
  k_aux_points<<<(unsigned)nb, BLOCK_AUX, 0, st>>>(ctx->tables, G, ok, cls, npts, xi_dev, D_dev, nmax, out_dev,
                                                   ctx->d_status);
  ctx->launches++;
  CK(cudaGetLastError());
  return F12INT_OK;
}

// Shell-pair bounds bound(ab) = sqrt(max |(ab|k|ab)|) over the diagonal block
// (the I3 kernel for I5), cached per basis and class.
static int ensure_pair_bounds(f12int_ctx *ctx, int basis_id, int cls) {
  const int dcls = cls == 5 ? 3 : cls;
  std::lock_guard<std::recursive_mutex> blk(ctx->bounds_mu);
  if (!ctx->bases[basis_id].pair_bound[dcls].empty()) return F12INT_OK;
  const f12int_ctx::BasisData &B = ctx->bases[basis_id];
  const int ns = B.nshell;
  // diagonal blocks (ab|ab) for a >= b
  std::vector<int32_t> hq;
  std::vector<int64_t> off;
  int64_t tot = 0;
  for (int a = 0; a < ns; ++a)
    for (int b = 0; b <= a; ++b) {
      hq.insert(hq.end(), {a, b, a, b});
      off.push_back(tot);
      int nab = ncart(B.l[a]) * ncart(B.l[b]);
      tot += (int64_t)nab * nab;
    }
  const int64_t nq = (int64_t)off.size();
  int32_t *dq = nullptr;
  int64_t *doff = nullptr;
  double *dout = nullptr;
  int rc = dalloc(ctx, &dq, sizeof(int32_t) * hq.size());
  if (rc == F12INT_OK) rc = dalloc(ctx, &doff, sizeof(int64_t) * nq);
  if (rc == F12INT_OK) rc = dalloc(ctx, &dout, sizeof(double) * tot);
  std::vector<double> hout((size_t)tot);
  if (rc == F12INT_OK) {
    cudaStream_t st = ctx->stream;
    if (cudaMemcpyAsync(dq, hq.data(), sizeof(int32_t) * hq.size(), cudaMemcpyHostToDevice, st) != cudaSuccess ||
        cudaMemcpyAsync(doff, off.data(), sizeof(int64_t) * nq, cudaMemcpyHostToDevice, st) != cudaSuccess)
      rc = F12INT_ECUDA;
    // the diagonal blocks themselves can be far below the primitive screen
    // (a pair's bound multiplies a partner's that may be large), so they are
    // computed without it
    if (rc == F12INT_OK)
      rc = compute_class_impl(ctx, basis_id, dcls, dq, nq, dout, doff, st, 0.0, /*prim_screen=*/false);
    if (rc == F12INT_OK &&
        (cudaMemcpyAsync(hout.data(), dout, sizeof(double) * tot, cudaMemcpyDeviceToHost, st) != cudaSuccess ||
         cudaStreamSynchronize(st) != cudaSuccess))
      rc = F12INT_ECUDA;
  }
  dfree(ctx, dq, sizeof(int32_t) * hq.size());
  dfree(ctx, doff, sizeof(int64_t) * nq);
  dfree(ctx, dout, sizeof(double) * tot);
  if (rc != F12INT_OK) return rc;
  std::vector<double> bound((size_t)ns * ns, 0.0);
  int64_t k = 0;
  for (int a = 0; a < ns; ++a)
    for (int b = 0; b <= a; ++b, ++k) {
      int nab = ncart(B.l[a]) * ncart(B.l[b]);
      double m = 0.0;
      for (int64_t i = 0; i < (int64_t)nab * nab; ++i) m = std::max(m, std::fabs(hout[off[k] + i]));
      bound[(size_t)a * ns + b] = bound[(size_t)b * ns + a] = std::sqrt(m);
    }
  ctx->bases[basis_id].pair_bound[dcls] = std::move(bound);
  return F12INT_OK;
}

int f12int_pair_bounds(f12int_ctx *ctx, int basis_id, int cls, double *bounds_out) {
  if (!ctx || cls < 1 || cls > 6 || !bounds_out) return F12INT_EINVAL;
  if (basis_id < 0 || basis_id >= (int)ctx->bases.size() || !ctx->factor_ready) return F12INT_ENOTREADY;
  int rc = ensure_pair_bounds(ctx, basis_id, cls);
  if (rc != F12INT_OK) return rc;
  const std::vector<double> &b = ctx->bases[basis_id].pair_bound[cls == 5 ? 3 : cls];
  std::memcpy(bounds_out, b.data(), sizeof(double) * b.size());
  return F12INT_OK;
}

int f12int_quartet_estimates(f12int_ctx *ctx, int basis_id, int cls, const int32_t *quartets, int64_t n,
                             double *est_out) {
  if (!ctx || cls < 1 || cls > 6 || n < 0 || (n > 0 && (!quartets || !est_out))) return F12INT_EINVAL;
  if (basis_id < 0 || basis_id >= (int)ctx->bases.size() || !ctx->factor_ready) return F12INT_ENOTREADY;
  int rc = ensure_pair_bounds(ctx, basis_id, cls);
  if (rc != F12INT_OK) return rc;
  const f12int_ctx::BasisData &B = ctx->bases[basis_id];
  for (int64_t i = 0; i < n; ++i) {
    const int32_t *q = quartets + 4 * i;
    for (int k = 0; k < 4; ++k)
      if (q[k] < 0 || q[k] >= B.nshell) return F12INT_EINVAL;
    est_out[i] = screen_estimate(ctx, B, cls, q[0], q[1], q[2], q[3]);
  }
  return F12INT_OK;
}

int f12int_screen(f12int_ctx *ctx, int basis_id, int cls, double thresh, int32_t *quartets_out, int64_t cap,
                  int64_t *n_out) {
  if (!ctx || cls < 1 || cls > 6 || !n_out || cap < 0 || (cap > 0 && !quartets_out)) return F12INT_EINVAL;
  if (basis_id < 0 || basis_id >= (int)ctx->bases.size() || !ctx->factor_ready) return F12INT_ENOTREADY;
  if (!(thresh >= 0.0)) return F12INT_EINVAL;
  int rc = ensure_pair_bounds(ctx, basis_id, cls);
  if (rc != F12INT_OK) return rc;
  const f12int_ctx::BasisData &B = ctx->bases[basis_id];
  const int ns = B.nshell;
  const std::vector<double> &bound = B.pair_bound[cls == 5 ? 3 : cls];
  std::vector<std::pair<int, int>> pairs;
  for (int a = 0; a < ns; ++a)
    for (int b = 0; b <= a; ++b) pairs.emplace_back(a, b);
  int64_t cnt = 0;
  const std::vector<double> &g = ctx->kgrow[cls];
  const double gmax = g.empty() ? 1.0 : g.back();   // G is non-decreasing
  for (size_t i = 0; i < pairs.size(); ++i) {
    size_t jend = (cls == 5) ? pairs.size() : i + 1;
    double bi = bound[(size_t)pairs[i].first * ns + pairs[i].second];
    for (size_t j = 0; j < jend; ++j) {
      double bj = bound[(size_t)pairs[j].first * ns + pairs[j].second];
      const double q = bi * bj;
      if (q >= thresh ||
          (q * gmax * kScreenSafety[cls] >= thresh &&
           screen_estimate(ctx, B, cls, pairs[i].first, pairs[i].second, pairs[j].first, pairs[j].second) >=
               thresh)) {
        if (cnt < cap) {
          quartets_out[4 * cnt] = pairs[i].first;
          quartets_out[4 * cnt + 1] = pairs[i].second;
          quartets_out[4 * cnt + 2] = pairs[j].first;
          quartets_out[4 * cnt + 3] = pairs[j].second;
        }
        ++cnt;
      }
    }
  }
  *n_out = cnt;
  return F12INT_OK;
}

}  // extern "C"

// ===================================================== static-scratch variant ==
// Callers that must not allocate device memory while they run (for example a
// host application that reserves all device memory up front for its own
// pool, or a latency-sensitive service in which the device-wide
// synchronisation of a cudaMalloc would stall work on other streams) use
// f12int_compute_class_static.  It runs the same kernels as
// f12int_compute_class but takes every scratch buffer from the file-scope
// array below, which each GPU that loads the library holds until exit.

#define F12INT_STATIC_SCRATCH_BYTES ((size_t)64 << 20)

static __device__ __align__(256) unsigned char g_static_scratch[F12INT_STATIC_SCRATCH_BYTES];

namespace {

// Device address of g_static_scratch, resolved once per device.  In host code
// the array's name is only a stand-in; the address must come from
// cudaGetSymbolAddress with the device current.
std::mutex g_static_mu;
void *g_static_addr[64] = {nullptr};

int static_scratch_address(int device, unsigned char **out) {
  if (device < 0 || device >= 64) return F12INT_EINVAL;
  std::lock_guard<std::mutex> lk(g_static_mu);
  if (!g_static_addr[device]) {
    void *p = nullptr;
    cudaError_t e = cudaGetSymbolAddress(&p, g_static_scratch);
    if (e != cudaSuccess || !p) return F12INT_ECUDA;
    g_static_addr[device] = p;
  }
  *out = (unsigned char *)g_static_addr[device];
  return F12INT_OK;
}

size_t align256(size_t x) { return (x + 255) & ~(size_t)255; }

}  // namespace

extern "C" int f12int_compute_class_static(f12int_ctx *ctx, int basis_id, int cls, const int32_t *quartets_dev,
                                           int64_t n, double *out_dev, const int64_t *offsets_dev,
                                           void *cuda_stream) {
  if (!ctx) return F12INT_EINVAL;
  if (cls < 1 || cls > 6 || n < 0) return F12INT_EINVAL;
  if (basis_id < 0 || basis_id >= (int)ctx->bases.size()) return F12INT_ENOTREADY;
  if (!ctx->factor_ready) return F12INT_ENOTREADY;
  if (!ctx->cls_ok[cls]) return F12INT_EDOMAIN;
  if (n == 0) return F12INT_OK;
  if (!quartets_dev || !out_dev || !offsets_dev) return F12INT_EINVAL;
  // a first bound on the list length, before anything is read back
  const size_t per_quartet = sizeof(int32_t) * 4 + sizeof(int64_t) * 2 + sizeof(CTask);
  if ((size_t)n > F12INT_STATIC_SCRATCH_BYTES / per_quartet) return F12INT_EINVAL;
  std::lock_guard<std::mutex> lk(ctx->mu);
  CK(cudaSetDevice(ctx->device));
  unsigned char *base = nullptr;
  int rc = static_scratch_address(ctx->device, &base);
  if (rc != F12INT_OK) return rc;
  const f12int_ctx::BasisData &B = ctx->bases[basis_id];
  cudaStream_t st = pick_stream(ctx, cuda_stream);
  // (never page-locked: locking and unlocking pages waits for the device's other
  // streams, which a caller of this entry point must not see)
  HostStage &hs = ctx->static_stage;
  if (!hs.reserve(24 * (size_t)n)) return F12INT_ENOMEM;
  CK(cudaMemcpyAsync(hs.p, quartets_dev, sizeof(int32_t) * 4 * n, cudaMemcpyDeviceToHost, st));
  CK(cudaMemcpyAsync(hs.p + 16 * n, offsets_dev, sizeof(int64_t) * n, cudaMemcpyDeviceToHost, st));
  CK(cudaStreamSynchronize(st));
  ListPlan P;
  auto fp64 = [](const int32_t *) { return 0; };
  rc = plan_kinds(B, cls, n, (const int32_t *)hs.p, fp64, P);
  if (rc != F12INT_OK) return rc;
  // layout of the array: quartets, offsets and primitive offsets in the
  // working order, the key histogram and the task list (all sized exactly
  // now), then the scratch of one chunk.  Every size check happens here,
  // before anything is queued, so that an F12INT_EINVAL leaves the array and
  // the output untouched.
  auto fixed_bytes = [&] {
    return align256(sizeof(int32_t) * 4 * (size_t)n) + align256(sizeof(int64_t) * (size_t)n) +
           align256(sizeof(int64_t) * ((size_t)n + 1)) + align256(sizeof(unsigned) * kNKeys) +
           align256(sizeof(CTask) * (size_t)P.ntask);
  };
  const int64_t nf = std::max(1, ctx->tables.nfam[cls == 5 ? 3 : cls]);
  const GridView G = grid_view(ctx, B, cls);
  int64_t pitch = 4, big_in = 0;   // of the general quartets: row doubles, inner pairs
  for (const ListPlan::Run &r : P.runs)
    if (!r.thin) {
      big_in = std::max(big_in, r.npq / r.npab);
      pitch = std::max(pitch, r.pitch / r.npq);
    }
  f12host::ScratchCut cut;
  auto room = [&]() -> int64_t {   // bytes of the chunk's scratch, negative when the list does not fit
    return (int64_t)F12INT_STATIC_SCRATCH_BYTES - (int64_t)fixed_bytes() - 4 * 256;
  };
  auto fits = [&] { return f12host::scratch_cut(room(), G.direct(), nf, kPartPitch, P.big_pq, big_in, pitch, &cut); };
  if (!fits()) {   // fewer and longer tasks leave more of the array
    rc = plan_kinds(B, cls, n, (const int32_t *)hs.p, fp64, P, /*fewest=*/true);
    if (rc != F12INT_OK) return rc;
    if (!fits()) return F12INT_EINVAL;
  }
  const ListLayout at(n, 0, P.ntask);   // (no row offsets: every row at one pitch)
  if (!hs.reserve(24 * (size_t)n + at.bytes, 24 * (size_t)n)) return F12INT_ENOMEM;
  unsigned char *list = hs.p + 24 * (size_t)n;
  plan_fill(P, (const int32_t *)hs.p, (const int64_t *)(hs.p + 16 * n), (int32_t *)list, (int64_t *)(list + at.offsets),
            (int64_t *)(list + at.pqoff), nullptr, (CTask *)(list + at.tasks));
  int32_t *d_q = (int32_t *)base;
  int64_t *d_o = (int64_t *)(base + align256(sizeof(int32_t) * 4 * (size_t)n));
  int64_t *d_pq = (int64_t *)((unsigned char *)d_o + align256(sizeof(int64_t) * (size_t)n));
  unsigned *d_hist = (unsigned *)((unsigned char *)d_pq + align256(sizeof(int64_t) * ((size_t)n + 1)));
  CTask *d_tk = (CTask *)((unsigned char *)d_hist + align256(sizeof(unsigned) * kNKeys));
  unsigned char *scratch = (unsigned char *)d_tk + align256(sizeof(CTask) * (size_t)P.ntask);
  ListBufs D{d_q, d_o, d_pq, nullptr, d_tk};
  D.pitch = (int)pitch;
  D.hist = d_hist;
  D.keys = (int *)scratch;
  D.keys_cap = cut.keys_cap;
  D.rows_cap = cut.rows_cap;
  unsigned char *next = scratch + align256(sizeof(int) * (size_t)cut.keys_cap);
  if (G.direct()) {
    D.rows = (double *)next;
  } else {
    D.order = (unsigned *)next;
    D.part = (double *)(next + align256(sizeof(unsigned) * (size_t)cut.keys_cap));
    D.part_thin = cut.part_thin;
    D.part_cap = cut.part_cap;
    D.rows = D.part + D.part_cap;
  }
  CK(cudaMemcpyAsync(d_tk, P.tasks, sizeof(CTask) * (size_t)P.ntask, cudaMemcpyHostToDevice, st));
  CK(cudaMemcpyAsync(d_q, P.quartets, sizeof(int32_t) * 4 * n, cudaMemcpyHostToDevice, st));
  CK(cudaMemcpyAsync(d_o, P.offsets, sizeof(int64_t) * n, cudaMemcpyHostToDevice, st));
  CK(cudaMemcpyAsync(d_pq, P.pqoff, sizeof(int64_t) * (n + 1), cudaMemcpyHostToDevice, st));
  // the primitive screen of f12int_compute_class when its table for this
  // (basis, class) exists already (building it would allocate); without it
  // every primitive quartet is evaluated
  const int rc_launch = launch_list(ctx, P, D, pair_view(ctx, B, cls, B.prim_screen), G, cls, out_dev, st, false);
  // the staging buffer is free again once the queued copies are consumed, and
  // on an error nothing of this call is still running when it returns
  cudaError_t e = cudaStreamSynchronize(st);
  if (rc_launch != F12INT_OK)
    for (cudaStream_t t : ctx->side) cudaStreamSynchronize(t);
  if (rc_launch != F12INT_OK) return rc_launch;
  if (e != cudaSuccess) return cuda_fail(e);
  return F12INT_OK;
}

#include "engine.cuh"
