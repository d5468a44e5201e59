// contract.cuh -- the general contraction: quartets whose total order is past
// the thin kernel's (thin.cuh).
//
// Two kernels.  The Hermite rows: one thread per primitive quartet forms g_n
// and R_tuv (Eq. ri) by the Cartesian recursion and writes R^(0) as a row.
// The contraction: one block per (shell quartet, range of components);
// the rows of several ket primitive pairs are staged in shared memory and
// every thread owns entries (bra Hermite index, ket component) of the ket sum
// of Eq. ii, then elements of the bra sum.
//
// Both are bound by the FP64 pipe, which takes 16 cycles of an SM per warp
// instruction whether one lane works or 32: a warp that forms g_n, the square
// roots of its prefactor and the recursion's small levels together spends
// several times the instructions of 32 threads that each do their own.
// Measured on 200,000 I4 quartets of s/p/d shells (three primitives each): 35 ms
// with one kernel whose warps took a primitive quartet each, 4.3 ms of rows (89%
// of the pipe) and 7.9 ms of contraction so; 600,000 I5 quartets run their large
// launches at 78-90% of the pipe.  Launches of a few small blocks are bound by a
// thread's chain of loads and multiply-adds (5-20%).
#pragma once

#include <algorithm>
#include <array>
#include <vector>

#include "kernel_common.cuh"

namespace {

// ------------------------------------------------------------ index tables --
// Component pairs of two shells (l1, l2) in order of their number of Hermite
// products (the ket and bra sums' loop lengths, so that the lanes of a warp run
// loops of one length), and the products themselves.
constexpr int PT_MAXCOMP = 100;
constexpr int PT_TERMS = 8192;           // products of all 16 shell pairs
struct PairTab {
  int ncomp, nterm, first;               // first: of its products in d_pt_term
  unsigned char comp[PT_MAXCOMP];        // sorted position -> component (i1 ncart(l2) + i2)
  unsigned short off[PT_MAXCOMP + 1];    // sorted position -> first product
};
__device__ PairTab d_pt[16];             // [l1 * 4 + l2]
// a product E_t E_u E_v: x = t | u << 4 | v << 8, y = offsets of E_t, E_u, E_v in
// the pair's table (three dimensions of n1 each), ten bits each
__device__ uint2 d_pt_term[PT_TERMS];
__device__ unsigned d_htuv[NHMAX];       // Hermite index -> t | u << 4 | v << 8

struct HostPairTabs {
  PairTab pt[16];
  std::vector<uint2> term;
};
static const HostPairTabs &pair_tabs() {
  static const HostPairTabs tabs = [] {
    HostPairTabs h;
    auto cart = [](int l) {
      std::vector<std::array<int, 3>> c;
      for (int i = l; i >= 0; --i)
        for (int j = l - i; j >= 0; --j) c.push_back({i, j, l - i - j});
      return c;
    };
    for (int l1 = 0; l1 <= LSH; ++l1)
      for (int l2 = 0; l2 <= LSH; ++l2) {
        PairTab &p = h.pt[l1 * 4 + l2];
        p = PairTab{};
        const auto c1 = cart(l1), c2 = cart(l2);
        const int nt = l1 + l2 + 1, n1 = (l1 + 1) * (l2 + 1) * nt;
        p.ncomp = (int)(c1.size() * c2.size());
        p.first = (int)h.term.size();
        std::vector<int> order((size_t)p.ncomp);
        auto count = [&](int k) {
          const auto &a = c1[(size_t)k / c2.size()], &b = c2[(size_t)k % c2.size()];
          return (a[0] + b[0] + 1) * (a[1] + b[1] + 1) * (a[2] + b[2] + 1);
        };
        for (int k = 0; k < p.ncomp; ++k) order[(size_t)k] = k;
        std::stable_sort(order.begin(), order.end(), [&](int x, int y) { return count(x) < count(y); });
        for (int s = 0; s < p.ncomp; ++s) {
          const int k = order[(size_t)s];
          p.comp[s] = (unsigned char)k;
          p.off[s] = (unsigned short)p.nterm;
          const auto &a = c1[(size_t)k / c2.size()], &b = c2[(size_t)k % c2.size()];
          unsigned o[3];
          for (int d = 0; d < 3; ++d) o[d] = (unsigned)(d * n1 + (a[d] * (l2 + 1) + b[d]) * nt);
          for (int t = 0; t <= a[0] + b[0]; ++t)
            for (int u = 0; u <= a[1] + b[1]; ++u)
              for (int v = 0; v <= a[2] + b[2]; ++v) {
                uint2 w;
                w.x = (unsigned)(t | u << 4 | v << 8);
                w.y = (o[0] + (unsigned)t) | (o[1] + (unsigned)u) << 10 | (o[2] + (unsigned)v) << 20;
                h.term.push_back(w);
                ++p.nterm;
              }
        }
        p.off[p.ncomp] = (unsigned short)p.nterm;
      }
    return h;
  }();
  return tabs;
}

// largest number of products over ranges of jc consecutive sorted components
static int range_terms(int l1, int l2, int jc) {
  const PairTab &p = pair_tabs().pt[l1 * 4 + l2];
  int best = 0;
  for (int j = 0; j < p.ncomp; j += jc) best = std::max(best, (int)p.off[std::min(p.ncomp, j + jc)] - (int)p.off[j]);
  return best;
}

// ------------------------------------------------------------ Hermite rows --
// The rows of a chunk: the first double of quartet q's lies at off[q] - first
// of p, or (pitch > 0, no table of offsets) its primitive quartets' in order at
// pitch doubles each, `first` of them before p.
struct RowView {
  double *p;
  const int64_t *off;
  int64_t first;
  int pitch;
  __device__ __forceinline__ double *quartet(const QuartetView &QV, int64_t q) const {
    return p + ((pitch ? QV.pq_off[q] * pitch : off[q]) - first);
  }
  __device__ __forceinline__ int stride(int own) const { return pitch ? pitch : own; }
};

__host__ __device__ __forceinline__ int row_pitch(int L) { return (nh_count(L) + 3) & ~3; }   // whole 32-byte sectors

__device__ __forceinline__ void store4(double *p, double a, double b, double c, double d) {
  asm volatile("st.global.v4.f64 [%0], {%1, %2, %3, %4};" ::"l"(p), "d"(a), "d"(b), "d"(c), "d"(d) : "memory");
}

// R^(0)_tuv, t+u+v <= L, from g_n, in the order of hidx, in registers: level n
// replaces level n + 1 in place, highest t+u+v first (its sources t+u+v - 1 and
// - 2 are then still of level n + 1).
template <int L>
__device__ __forceinline__ void hermite_row(const double *g, double X, double Y, double Z, double *out) {
  constexpr int NH = (L + 1) * (L + 2) * (L + 3) / 6, NP = (NH + 3) & ~3;
  double R[NP];
#pragma unroll
  for (int i = 0; i < NP; ++i) R[i] = 0.0;
  R[0] = g[L];
#pragma unroll
  for (int n = L - 1; n >= 0; --n) {
#pragma unroll
    for (int S = L - n; S >= 1; --S)
#pragma unroll
      for (int t = S; t >= 0; --t)
#pragma unroll
        for (int v = 0; v <= S - t; ++v) {
          const int u = S - t - v;
          double val;
          if (t > 0) val = X * R[hidx(t - 1, u, v)] + (t > 1 ? (t - 1) * R[hidx(t > 1 ? t - 2 : 0, u, v)] : 0.0);
          else if (u > 0) val = Y * R[hidx(t, u - 1, v)] + (u > 1 ? (u - 1) * R[hidx(t, u > 1 ? u - 2 : 0, v)] : 0.0);
          else val = Z * R[hidx(t, u, v - 1)] + (v > 1 ? (v - 1) * R[hidx(t, u, v > 1 ? v - 2 : 0)] : 0.0);
          R[hidx(t, u, v)] = val;
        }
    R[0] = g[n];
  }
#pragma unroll
  for (int i = 0; i < NP; i += 4) store4(out + i, R[i], R[i + 1], R[i + 2], R[i + 3]);
}

// The same for any L, in local memory (orders 7 and up: few quartets, whose
// contraction is tens of times the recursion).
__device__ __noinline__ void hermite_row_any(int L, const double *g, double X, double Y, double Z, double *out) {
  double R[NHMAX + 4];
  R[0] = g[L];
  for (int n = L - 1; n >= 0; --n) {
    for (int S = L - n; S >= 1; --S) {
      const int b0 = S * (S + 1) * (S + 2) / 6, b1 = b0 - S * (S + 1) / 2, b2 = b1 - (S - 1) * S / 2;
      // (w = u + v, offset w (w + 1)/2 + v within a level of t + u + v)
      for (int w = S; w >= 0; --w) {
        const int t = S - w;
        for (int v = 0; v <= w; ++v) {
          const int u = w - v, o = w * (w + 1) / 2 + v;
          double val;
          if (t > 0) {
            val = X * R[b1 + o];
            if (t > 1) val += (t - 1) * R[b2 + o];
          } else if (u > 0) {
            val = Y * R[b1 + (w - 1) * w / 2 + v];
            if (u > 1) val += (u - 1) * R[b2 + (w - 2) * (w - 1) / 2 + v];
          } else {
            val = Z * R[b1 + (w - 1) * w / 2 + v - 1];
            if (v > 1) val += (v - 1) * R[b2 + (w - 2) * (w - 1) / 2 + v - 2];
          }
          R[b0 + o] = val;
        }
      }
    }
    R[0] = g[n];
  }
  const int nh = nh_count(L), np = row_pitch(L);
  for (int i = nh; i < np; ++i) R[i] = 0.0;
  for (int i = 0; i < np; i += 2) reinterpret_cast<double2 *>(out)[i >> 1] = make_double2(R[i], R[i + 1]);
}

template <int L>
__device__ __forceinline__ void direct_row(const GridView &G, const PairView &PV, int pab, int pcd, double X, double Y,
                                           double Z, double *out) {
  double g[L + 1];
  aux_direct<L>(G, PV, pab, pcd, X * X + Y * Y + Z * Z, g);
  if constexpr (L <= 6) hermite_row<L>(g, X, Y, Z, out);
  else hermite_row_any(L, g, X, Y, Z, out);
}

// Rows of the primitive quartets pq0 + [0, npq) of a list (npq < 0, in a batch:
// as many as its counts say).  DIRECT: g_n from the
// grid or the Boys table, the primitive screen decided here (keys[r], one int
// per primitive quartet, 0 or the skip key); else g_n is the sum of the
// families' partial rows `part` (nf per primitive quartet, in family order)
// and keys[r nf] says what the screen dropped.
template <bool BATCH, bool DIRECT>
__global__ void __launch_bounds__(BLOCK_AUX)
k_hermite_rows(GridView G, PairView PV0, QuartetView QV, int cls, int nf, int64_t pq0, int64_t npq, int *keys,
               const double *part, RowView rows, unsigned long long *fma_total) {
  // in a batch count_dev[2] is the number of primitive quartets that the
  // general contraction reads (the thin ones follow them in the list)
  const int64_t n = BATCH && npq < 0 ? QV.count_dev[2] : npq;
  const double pi52 = 17.493418327624862846;   // pi^{5/2}
  unsigned long long nfma = 0;
  for (int64_t r0 = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) & ~(int64_t)31; r0 < n;
       r0 += (int64_t)gridDim.x * blockDim.x) {   // warp-uniform
    const int lane = threadIdx.x & 31;
    int64_t lo = lane == 0 ? find_quartet(QV.pq_off, qv_count(QV), pq0 + r0) : 0;
    lo = __shfl_sync(0xffffffffu, lo, 0);
    const int64_t r = r0 + lane, pq = pq0 + r;
    if (r >= n) continue;
    // every quartet holds at least one primitive quartet: the lane's lies within `lane` of the warp's first
    int64_t hi = min(lo + lane, qv_count(QV) - 1);
    while (lo < hi) {
      const int64_t mid = (lo + hi + 1) >> 1;
      if (QV.pq_off[mid] <= pq) lo = mid;
      else hi = mid - 1;
    }
    const PairView &PV = qv_view<BATCH>(PV0, QV, lo);
    const int32_t *s = QV.quartets + 4 * lo;
    const int ns = PV.nshell;
    const int ab = s[0] * ns + s[1], cd = s[2] * ns + s[3];
    const int npcd = PV.pair_start[cd + 1] - PV.pair_start[cd];
    const int k = (int)(pq - QV.pq_off[lo]);
    const int pab = PV.pair_start[ab] + k / npcd, pcd = PV.pair_start[cd] + k % npcd;
    const double X = pair_sep(PV.pp_P, pab, pcd, 0), Y = pair_sep(PV.pp_P, pab, pcd, 1),
                 Z = pair_sep(PV.pp_P, pab, pcd, 2);
    if constexpr (DIRECT) {
      if (prim_negligible(PV, pab, pcd, X * X + Y * Y + Z * Z)) {
        keys[r] = SKIP_KEY;
        continue;
      }
      keys[r] = 0;
    } else if (keys[r * nf] == SKIP_KEY) {
      continue;
    }
    const int L = PV.shell_l[s[0]] + PV.shell_l[s[1]] + PV.shell_l[s[2]] + PV.shell_l[s[3]] + (cls == 5 ? 2 : 0);
    double *o = rows.quartet(QV, lo) + (int64_t)k * rows.stride(row_pitch(L));
    if constexpr (DIRECT) {
      nfma += aux_direct_fmas(G.boys != nullptr, L) + (L + 1) * (L + 2) * (L + 3) * (L + 4) / 24;
      switch (L) {
        case 4: direct_row<4>(G, PV, pab, pcd, X, Y, Z, o); break;
        case 5: direct_row<5>(G, PV, pab, pcd, X, Y, Z, o); break;
        case 6: direct_row<6>(G, PV, pab, pcd, X, Y, Z, o); break;
        case 7: direct_row<7>(G, PV, pab, pcd, X, Y, Z, o); break;
        case 8: direct_row<8>(G, PV, pab, pcd, X, Y, Z, o); break;
        case 9: direct_row<9>(G, PV, pab, pcd, X, Y, Z, o); break;
        case 10: direct_row<10>(G, PV, pab, pcd, X, Y, Z, o); break;
        case 11: direct_row<11>(G, PV, pab, pcd, X, Y, Z, o); break;
        case 12: direct_row<12>(G, PV, pab, pcd, X, Y, Z, o); break;
        case 13: direct_row<13>(G, PV, pab, pcd, X, Y, Z, o); break;
        default: direct_row<14>(G, PV, pab, pcd, X, Y, Z, o); break;
      }
    } else {
      double g[LAUX + 1];
      const double p = PV.pp_p[pab], q = PV.pp_p[pcd];
      const double pref = pi52 / (sqrt(p + q) * p * q);
      for (int l = 0; l <= L; ++l) {
        double acc = 0.0;
        for (int f = 0; f < nf; ++f) acc += part[(r * nf + f) * kPartPitch + l];
        g[l] = pref * acc;
      }
      hermite_row_any(L, g, X, Y, Z, o);
    }
  }
  if (DIRECT && fma_total) {
    for (int o = 16; o > 0; o >>= 1) nfma += __shfl_down_sync(0xffffffffu, nfma, o);
    if ((threadIdx.x & 31) == 0 && nfma) atomicAdd(fma_total, nfma);
  }
}

// ------------------------------------------------------------- contraction --
// One pair of the quartet is the inner one: its Hermite index is summed per
// primitive quartet, for every Hermite index of the outer pair; the outer sum
// follows once per outer primitive pair.  Eq. ii has the ket inner.  Which one
// is cheaper depends on the angular momenta alone up to a factor of ten ((ss|dd)
// with the ket inner sums 336 products per primitive quartet, with the bra inner
// 35), so the plan picks the cheaper (outer_first): a quartet with the bra inner
// is listed as (cd|ab), its task marked, and its block transposed on the way
// out.  For I5, whose operator acts on the bra, the marked task applies it in
// the inner sum.
// Shared memory of a block (T: double, or float on the mixed path):
//   cube   rows of kc inner primitive pairs, each spread over a cube [t][u][v]
//          of pitch L+1, so that R_{t+t',u+u',v+v'} lies at an outer part plus
//          an inner part                                      kc (L+1)^3
//   E3i    products E_t' E_u' E_v' of the same pairs            kc ne3i
//   W      the inner sums of one outer primitive pair           nh(Lo) ni
//   O      the block's elements                                 no ni
//   E3o    products of the outer primitive pair
//   ints   cube offset of each inner product, W row of each outer product, cube
//          offset of each outer Hermite index and of each row element
// (the pair with I5's operator has four products for one: E_t E_u E_v times
// (a-b)/2p, and the three with one factor dE/dAB).
// Every sum is taken by one thread in the order of the primitives, so the
// blocks do not depend on the ranges, kc or the number of threads.
struct ContractShape {
  int la, lb, lc, ld;   // outer (la, lb), inner (lc, ld)
  int ext;              // 2 for I5
  bool op_inner;        // I5's operator acts on the inner pair
  __host__ __device__ int lab() const { return la + lb; }
  __host__ __device__ int L() const { return la + lb + lc + ld + ext; }
  __host__ __device__ int nhB() const { return nh_count(la + lb + (op_inner ? 0 : ext)); }
  __host__ __device__ int nab() const { return ncart(la) * ncart(lb); }
  __host__ __device__ int ncd() const { return ncart(lc) * ncart(ld); }
  __host__ __device__ int outer4() const { return ext && !op_inner ? 4 : 1; }
  __host__ __device__ int inner4() const { return ext && op_inner ? 4 : 1; }
};
// bytes that do not depend on kc, and bytes per staged inner primitive pair, for
// jc inner components with ncd_terms products, nab_terms outer products
__host__ __device__ inline size_t contract_fixed(const ContractShape &s, int jc, int ncd_terms, int nab_terms,
                                                 size_t esz) {
  return esz * ((size_t)s.nhB() * jc + (size_t)s.nab() * jc + (size_t)nab_terms * s.outer4()) +
         4 * ((size_t)ncd_terms + nab_terms + s.nhB() + nh_count(s.L()) + 4);
}
__host__ __device__ inline size_t contract_per_k(const ContractShape &s, int ncd_terms, size_t esz) {
  const size_t P = (size_t)s.L() + 1;
  return esz * (P * P * P + (size_t)ncd_terms * s.inner4());
}
constexpr int KC_MAX = 16;   // staged inner primitive pairs at most

__device__ __forceinline__ double tfma(double a, double b, double c) { return fma(a, b, c); }
__device__ __forceinline__ float tfma(float a, float b, float c) { return fmaf(a, b, c); }

// The rows of the kept primitive quartets of a group, spread over their cubes:
// asynchronous copies, so that the whole group's are in flight at once and the
// products below are formed meanwhile (one load at a time, a block of one warp
// waited about 20,000 cycles for 16 rows: 2000 mixed I4 quartets of one molecule, of up to 4096
// primitive quartets, 22.5 ms, so 20.1; 600,000 I5 quartets 134 and 129 ms).
__device__ __forceinline__ void stage_rows(double *cube, const double *rk, unsigned mask, int nk, int nhL, int pitch,
                                           int P3, const int *cpos, int tid, int nthr) {
  for (int i = tid; i < nhL; i += nthr) {
    const unsigned to = (unsigned)__cvta_generic_to_shared(cube + cpos[i]);
    for (int k = 0; k < nk; ++k)
      if (mask >> k & 1)
        asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(to + 8u * (unsigned)(k * P3)),
                     "l"(rk + (int64_t)k * pitch + i)
                     : "memory");
  }
}
__device__ __forceinline__ void stage_rows(float *cube, const double *rk, unsigned mask, int nk, int nhL, int pitch,
                                           int P3, const int *cpos, int tid, int nthr) {
  for (int i = tid; i < nhL; i += nthr)
    for (int k = 0; k < nk; ++k)
      if (mask >> k & 1) cube[k * P3 + cpos[i]] = (float)rk[(int64_t)k * pitch + i];
}
__device__ __forceinline__ void stage_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// One contraction task (quartet and range of inner components) by the whole
// block; smem_bytes of shared memory.  nsplit < 0: the quartet is listed with
// the bra inner.  iab0, iab1: outer primitive pairs of this launch (a quartet
// whose rows exceed the scratch is done in several launches; the later ones
// continue from the elements written).
template <bool BATCH, class T>
__device__ __forceinline__ void contract_task(const PairView &PV0, const QuartetView &QV, int cls, int kstride,
                                              int64_t pq0, const CTask task, const int *keys, const RowView &rows,
                                              double *out, const int64_t *offsets, unsigned long long *flops_total,
                                              unsigned char *smem_raw, unsigned smem_bytes, int iab0, int iab1) {
  const int64_t q = task.q;
  const PairView &PV = qv_view<BATCH>(PV0, QV, q);
  const int32_t *s = QV.quartets + 4 * q;
  const int ns = PV.nshell;
  const bool swapped = task.nsplit < 0;
  const int nsplit = abs((int)task.nsplit);
  const ContractShape S{PV.shell_l[s[0]], PV.shell_l[s[1]], PV.shell_l[s[2]], PV.shell_l[s[3]], cls == 5 ? 2 : 0,
                        cls == 5 && swapped};
  const PairTab &TB = d_pt[S.la * 4 + S.lb], &TK = d_pt[S.lc * 4 + S.ld];
  const int nab = S.nab(), ncd_all = S.ncd(), nhB = S.nhB(), L = S.L();
  const int jc = (ncd_all + nsplit - 1) / nsplit, j0 = task.split * jc;
  const int ncd = min(jc, ncd_all - j0);   // sorted inner components j0 .. j0 + ncd - 1
  if (ncd <= 0) return;                     // block-uniform
  const int m0 = TK.off[j0], ncdt = TK.off[j0 + ncd] - m0, nabt = TB.nterm;
  const int nhL = nh_count(L), pitch = rows.stride(row_pitch(L)), P = L + 1, P3 = P * P * P;
  const int tid = threadIdx.x, nthr = blockDim.x, lane = tid & 31;   // (whole warps)
  const int ab = s[0] * ns + s[1], cd = s[2] * ns + s[3];
  const int ab0 = PV.pair_start[ab], npab = PV.pair_start[ab + 1] - ab0;
  const int cd0 = PV.pair_start[cd], npcd = PV.pair_start[cd + 1] - cd0;
  const int kc = min(min(npcd, KC_MAX),
                     (int)((smem_bytes - contract_fixed(S, ncd, ncdt, nabt, sizeof(T))) / contract_per_k(S, ncdt, sizeof(T))));
  T *cube = reinterpret_cast<T *>(smem_raw);
  T *E3cd = cube + (size_t)kc * P3;
  T *W = E3cd + (size_t)kc * ncdt * S.inner4();
  T *O = W + (size_t)nhB * ncd;
  T *E3ab = O + (size_t)nab * ncd;
  int *ck = reinterpret_cast<int *>(E3ab + (size_t)nabt * S.outer4());
  int *hb = ck + ncdt, *cb = hb + nabt, *cpos = cb + nhB;
  for (int m = tid; m < ncdt; m += nthr) {
    const unsigned w = d_pt_term[TK.first + m0 + m].x;
    ck[m] = ((int)(w & 15) * P + (int)(w >> 4 & 15)) * P + (int)(w >> 8);
  }
  for (int m = tid; m < nabt; m += nthr) {
    const unsigned w = d_pt_term[TB.first + m].x;
    hb[m] = hidx((int)(w & 15), (int)(w >> 4 & 15), (int)(w >> 8));
  }
  for (int i = tid; i < nhL; i += nthr) {
    const unsigned w = d_htuv[i];
    const int c = ((int)(w & 15) * P + (int)(w >> 4 & 15)) * P + (int)(w >> 8);
    cpos[i] = c;
    if (i < nhB) cb[i] = c;   // (an order below L comes first in the index)
  }
  double *o;
  if constexpr (BATCH) o = QV.slot_out[QV.qslot[q]] + offsets[q];
  else o = out + offsets[q];
  const int i0 = max(iab0, 0), i1 = iab1 < 0 ? npab : min(iab1, npab);
  // an element's place in the block: sorted outer component x sorted inner one
  auto place = [&](int i) -> size_t {
    const int a = i / ncd, j = i - a * ncd;
    const int co = TB.comp[a], ci = TK.comp[j0 + j];
    return swapped ? (size_t)ci * nab + co : (size_t)co * ncd_all + ci;
  };
  for (int i = tid; i < nab * ncd; i += nthr) O[i] = i0 > 0 ? (T)o[place(i)] : (T)0;
  const int n1ab = (S.la + 1) * (S.lb + 1) * (S.lab() + 1), n1cd = (S.lc + 1) * (S.ld + 1) * (S.lc + S.ld + 1);
  const int kE = ncdt * S.inner4();   // products of one staged pair
  // the four products of a term for the pair with I5's operator
  auto products5 = [&](const double *E, const double *Fp, int pair, unsigned w, T *e, int stride) {
    const double a = PV.pp_ab[4 * pair], b = PV.pp_ab[4 * pair + 1];
    const double c5 = (a - b) / (2.0 * (a + b));
    const double ex = E[w & 1023], ey = E[w >> 10 & 1023], ez = E[w >> 20];
    e[0] = (T)(c5 * ex * ey * ez);
    e[stride] = (T)(Fp[w & 1023] * ey * ez);
    e[2 * stride] = (T)(ex * Fp[w >> 10 & 1023] * ez);
    e[3 * stride] = (T)(ex * ey * Fp[w >> 20]);
  };
  const int64_t pqq = QV.pq_off[q] - pq0;
  const double *rq = rows.quartet(QV, q);
  const int nent = nhB * ncd;
  unsigned long long nproc = 0;
  bool have = false;   // the products of every ket pair are staged already
  __syncthreads();
  for (int iab = i0; iab < i1; ++iab) {
    const int pab = ab0 + iab;
    for (int k0 = 0; k0 < npcd; k0 += kc) {
      const int nk = min(kc, npcd - k0);
      const int64_t pqk = pqq + (int64_t)iab * npcd + k0;
      // primitive quartets the screen kept
      const unsigned mask = __ballot_sync(0xffffffffu, lane < nk && keys[(pqk + min(lane, nk - 1)) * kstride] != SKIP_KEY);
      nproc += __popc(mask);
      const bool first = k0 == 0;
      const double *rk = rq + ((int64_t)iab * npcd + k0) * pitch;
      if (mask) {
        stage_rows(cube, rk, mask, nk, nhL, pitch, P3, cpos, tid, nthr);
        if (!have)
          for (int x = tid; x < nk * ncdt; x += nthr) {
            const int k = x / ncdt, m = x - k * ncdt;
            const double *E = PV.epool + PV.pp_eoff[cd0 + k0 + k];
            const unsigned w = d_pt_term[TK.first + m0 + m].y;
            if (!S.op_inner) E3cd[k * kE + m] = (T)(E[w & 1023] * E[w >> 10 & 1023] * E[w >> 20]);
            else products5(E, E + 3 * n1cd, cd0 + k0 + k, w, E3cd + k * kE + m, ncdt);
          }
        have = npcd <= kc;
      }
      if (first) {
        // products of this outer primitive pair
        const double *E = PV.epool + PV.pp_eoff[pab];
        for (int m = tid; m < nabt; m += nthr) {
          const unsigned w = d_pt_term[TB.first + m].y;
          if (S.outer4() == 1) E3ab[m] = (T)(E[w & 1023] * E[w >> 10 & 1023] * E[w >> 20]);
          else products5(E, E + 3 * n1ab, pab, w, E3ab + m, nabt);
        }
      }
      stage_wait();
      __syncthreads();
      // inner sum of Eq. ii: entry (bi, j) = sum over the staged pairs of
      // E_{t'u'v'} R_{t+t',u+u',v+v'}; consecutive threads take consecutive
      // outer indexes of one component
      for (int r = tid; r < nent; r += nthr) {
        const int j = r / nhB, bi = r - j * nhB;
        const int ma = TK.off[j0 + j] - m0, mb = TK.off[j0 + j + 1] - m0;
        T acc = first ? (T)0 : W[bi * ncd + j];
        for (int k = 0; k < nk; ++k) {
          if (!(mask >> k & 1)) continue;   // block-uniform
          const T *R = cube + k * P3 + cb[bi], *e = E3cd + k * kE;
          if (!S.op_inner) {
            for (int m = ma; m < mb; ++m) acc = tfma(e[m], R[ck[m]], acc);
          } else {
            // Eq. I5byI3_ (second coefficient -1, see the derivation note below):
            // R is differentiated by the centre of the inner pair itself
            const int P2 = P * P;
            for (int m = ma; m < mb; ++m) {
              const T *r = R + ck[m];
              acc = tfma(e[m], r[2 * P2] + r[2 * P] + r[2], acc);
              acc = tfma(e[ncdt + m], r[P2], acc);
              acc = tfma(e[2 * ncdt + m], r[P], acc);
              acc = tfma(e[3 * ncdt + m], r[1], acc);
            }
          }
        }
        W[bi * ncd + j] = acc;
      }
      __syncthreads();
    }
    // outer sum, with the sign (-1)^{t+u+v} of Eq. ii
    for (int i = tid; i < nab * ncd; i += nthr) {
      const int a = i / ncd, j = i - a * ncd;
      const int ma = TB.off[a], mb = TB.off[a + 1];
      T acc = O[i];
      for (int m = ma; m < mb; ++m) {
        const unsigned w = d_pt_term[TB.first + m].x;
        const int t = (int)(w & 15), u = (int)(w >> 4 & 15), v = (int)(w >> 8);
        const bool odd = (t + u + v) & 1;
        if (S.outer4() == 1) {
          const T e = E3ab[m];
          acc = tfma(odd ? -e : e, W[hb[m] * ncd + j], acc);
        } else {
          // Eq. I5byI3_ with the second coefficient -1 (see the derivation note
          // below), and the bra sign of t + u + v for both terms
          const T lap = W[hidx(t + 2, u, v) * ncd + j] + W[hidx(t, u + 2, v) * ncd + j] + W[hidx(t, u, v + 2) * ncd + j];
          T d = E3ab[m] * lap;
          d = tfma(-E3ab[nabt + m], W[hidx(t + 1, u, v) * ncd + j], d);
          d = tfma(-E3ab[2 * nabt + m], W[hidx(t, u + 1, v) * ncd + j], d);
          d = tfma(-E3ab[3 * nabt + m], W[hidx(t, u, v + 1) * ncd + j], d);
          acc += odd ? -d : d;
        }
      }
      O[i] = acc;
    }
    __syncthreads();
  }
  for (int i = tid; i < nab * ncd; i += nthr) o[place(i)] = (double)O[i];
  if (flops_total && tid == 0 && nproc) {
    // two flops per product summed, ten (four multiply-adds, two additions) with
    // I5's operator; kept primitive quartets for the inner sum, outer pairs for
    // the outer one
    const unsigned long long in = (S.inner4() == 4 ? 10ull : 2ull) * nhB * ncdt;
    const unsigned long long on = (S.outer4() == 4 ? 10ull : 2ull) * nabt * ncd;
    atomicAdd(flops_total, nproc * in + (unsigned long long)(i1 - i0) * on);
  }
}

// kstride: ints between the keys of consecutive primitive quartets
template <bool BATCH, class T>
__global__ void __launch_bounds__(256)
k_contract(PairView PV0, QuartetView QV, int cls, int kstride, int64_t pq0, const CTask *tasks, int64_t ntask,
           const int64_t *ntask_dev, const int *keys, RowView rows, double *out, const int64_t *offsets, int iab0, int iab1, unsigned long long *flops_total) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  unsigned smem_bytes;
  asm("mov.u32 %0, %%dynamic_smem_size;" : "=r"(smem_bytes));
  if constexpr (BATCH) {
    // ntask_dev = {first, end} of this launch's tasks
    const int64_t te = ntask_dev[1];
    for (int64_t tk = ntask_dev[0] + blockIdx.x; tk < te; tk += gridDim.x) {
      __syncthreads();   // the previous task's shared-memory reads are done
      contract_task<BATCH, T>(PV0, QV, cls, kstride, pq0, tasks[tk], keys, rows, out, offsets,
                              flops_total, smem_raw, smem_bytes, iab0, iab1);
    }
  } else {
    if (blockIdx.x < ntask)
      contract_task<BATCH, T>(PV0, QV, cls, kstride, pq0, tasks[blockIdx.x], keys, rows, out, offsets,
                              flops_total, smem_raw, smem_bytes, iab0, iab1);
  }
}
// Derivation note for I5: with d/dA_x = (a/p) d/dP_x + d/dAB_x and
// d/dB_x = (b/p) d/dP_x - d/dAB_x (E depends on AB only, R on P only),
//   1/2 (lap_A - lap_B) = sum_x [ (a-b)/(2p) d^2/dP_x^2 + d/dP_x d/dAB_x ],
// and d/dP_x = -d/dQ_x on R; hence the coefficient of the gradient term is
// -(a+b)/p = -1 (+1 on the R of a quartet listed with the bra inner, which are
// derivatives by P).

// ----------------------------------------------------------------- planning --
struct ContractPlan {
  int nthr, nsplit;
  size_t smem;
};

// Multiply-adds of a task that owns jc of the inner components, per primitive
// quartet of which npcd share an outer pair.
static double task_fmas(const ContractShape &s, int64_t npcd, int jc) {
  const PairTab &K = pair_tabs().pt[s.lc * 4 + s.ld], &B = pair_tabs().pt[s.la * 4 + s.lb];
  // (a term of the pair with I5's operator takes four multiply-adds and two additions)
  const double ket = (double)s.nhB() * K.nterm * (s.inner4() == 4 ? 6 : 1) * jc / s.ncd();
  const double bra = (double)jc * B.nterm * (s.outer4() == 4 ? 6 : 1) / (double)npcd;
  return nh_count(s.L()) + ket + bra;   // (staging a row costs about a multiply-add per element)
}

// Whether (ab|cd), with npab and npcd primitive pairs, is cheaper with the bra
// inner (listed as (cd|ab)): on the 12-atom s/p/d workload this takes 28% off
// the multiply-adds of the contraction, on f shells up to 44%.  Entries count
// by whole warps (a sum of ten entries costs as much as one of 32).  Past 256
// primitive pairs the smaller side is the inner one: the rows of one outer pair
// are the least that a launch takes, and stay below 1.4 MB at the highest order
// (so that no call is refused for them that its work items fit).
static bool bra_inner(int la, int lb, int lc, int ld, int cls, int64_t npab, int64_t npcd) {
  const ContractShape k{la, lb, lc, ld, cls == 5 ? 2 : 0, false}, b{lc, ld, la, lb, cls == 5 ? 2 : 0, cls == 5};
  auto cost = [](const ContractShape &s, int64_t nin) {
    const int e = s.nhB() * s.ncd(), o = s.nab() * s.ncd();
    const double pe = (double)((e + 31) / 32 * 32) / e, po = (double)((o + 31) / 32 * 32) / o;
    const PairTab &K = pair_tabs().pt[s.lc * 4 + s.ld], &B = pair_tabs().pt[s.la * 4 + s.lb];
    return pe * s.nhB() * K.nterm * (s.inner4() == 4 ? 6 : 1) +
           po * s.ncd() * B.nterm * (s.outer4() == 4 ? 6 : 1) / (double)nin;
  };
  if (std::max(npab, npcd) > 256 && npab != npcd) return npab < npcd;
  return cost(b, npab) < cost(k, npcd);
}
static ContractShape contract_shape(int la, int lb, int lc, int ld, int cls, bool swap) {
  return swap ? ContractShape{lc, ld, la, lb, cls == 5 ? 2 : 0, cls == 5}
              : ContractShape{la, lb, lc, ld, cls == 5 ? 2 : 0, false};
}

static bool valid_split(int ncd, int ns) {
  const int jc = (ncd + ns - 1) / ns;
  return (ncd + jc - 1) / jc == ns;   // no empty ranges
}

// Shared memory that a block of nsplit ranges asks for: up to KC_MAX staged
// inner pairs (no more than the quartet has) while the total stays below `soft`.
static size_t contract_smem(const ContractShape &s, int64_t npcd, int nsplit, size_t esz, size_t soft) {
  const int jc = (s.ncd() + nsplit - 1) / nsplit, ncdt = range_terms(s.lc, s.ld, jc);
  const int nabt = pair_tabs().pt[s.la * 4 + s.lb].nterm;
  const size_t fixed = contract_fixed(s, jc, ncdt, nabt, esz), per = contract_per_k(s, ncdt, esz);
  const size_t most = (size_t)std::min<int64_t>(npcd, KC_MAX);
  size_t k = fixed < soft ? (soft - fixed) / per : 0;
  k = std::min(std::max<size_t>(k, 1), most);
  return (fixed + k * per + 15) & ~(size_t)15;
}

// Soft limit of a block's shared memory, 16 warps an SM: four blocks of 128
// threads, in proportion for fewer (blocks of one warp that staged 54 KB left
// the FP64 pipe idle 80% of the time); and what a block may take when even one
// staged pair does not fit that.
static size_t smem_soft(int nthr) { return (size_t)54 * 1024 * (size_t)std::min(nthr, 128) / 128; }
constexpr size_t kSmemSplit = 72 * 1024, kSmemMax = 200 * 1024;

// Fewest ranges with which a block fits `cap`; 0: none.
static int fit_split(const ContractShape &s, size_t esz, size_t cap) {
  for (int ns = 1; ns <= s.ncd(); ++ns)
    if (valid_split(s.ncd(), ns) && contract_smem(s, 1, ns, esz, 0) <= cap) return ns;
  return 0;
}

// Ranges, threads and shared memory of a quartet of nprimq primitive
// quartets, npcd of them per outer pair: the fewest ranges that fit, more while a
// task exceeds `target` multiply-adds; threads so that the entries of the ket
// sum fill whole warps and rounds.  smem = 0 when nothing fits.
static ContractPlan contract_plan(const ContractShape &s, int64_t nprimq, int64_t npcd, size_t esz, double target,
                                  bool fewest = false) {
  int ns = 0;
  for (size_t cap : {kSmemSplit, 2 * kSmemSplit, kSmemMax})
    if (!ns && (!fewest || cap == kSmemMax)) ns = fit_split(s, esz, cap);
  if (!ns) return ContractPlan{32, 1, 0};
  const int ncd = s.ncd();
  for (int k = ns; k <= ncd; ++k) {
    if (!valid_split(ncd, k)) continue;
    ns = k;
    if ((double)nprimq * task_fmas(s, npcd, (ncd + k - 1) / k) <= target) break;
  }
  const int jc = (ncd + ns - 1) / ns;
  const int e = std::max(s.nhB() * jc, 1);
  int nthr = 32;
  double best = 0.0;
  for (int t : {32, 64, 96, 128, 192, 256}) {
    const double eff = (double)e / ((double)((e + t - 1) / t) * t);
    if (eff >= best - 0.04) {
      nthr = t;
      best = std::max(best, eff);
    }
    if (t >= e) break;
  }
  return ContractPlan{nthr, ns, contract_smem(s, npcd, ns, esz, smem_soft(nthr))};
}

}  // namespace
