// grid_host.cpp -- CPU build of single cells of the auxiliary grid, for tests.
//
// Compiles paper_1412_5070_gb300/csrc/auxgrid.cuh and gridtab.h as plain C++:
// a cell's rows are summed over the builder's own quadrature points, fitted by
// its own conversion, and evaluated as the integral kernels evaluate them, so
// that tests without a GPU can compare the grid with the oracle.  The library
// never loads this file's build.
#include <cstdint>
#include <cstring>
#include <map>
#include <vector>

#include "../paper_1412_5070_gb300/csrc/auxgrid.cuh"
#include "../paper_1412_5070_gb300/csrc/auxtab.h"
#include "../paper_1412_5070_gb300/csrc/gridtab.h"
#include "../paper_1412_5070_gb300/csrc/termlist.h"

using namespace f12dev;

namespace {

constexpr int kCls[4] = {2, 3, 4, 6};

struct Octave {
  GridQuad q;
  std::vector<double> F;   // [point][row]
};

// The grid of one class of a factor pair: its quadrature follows from the
// families of all four classes, as in the library.
struct HostGrid {
  GridClass gc;
  GridClass all[4];
  bool served = false;
  std::map<int, Octave> oct[2];               // the cells' quadrature, the check's
  std::map<int, std::vector<double>> cells;   // [row][coefficient]
  std::vector<double> ztab, node, xt;
  dd conv[GR_NC][GR_NC];
};

void radial(const HostGrid &G, double x, double *F) {
  grid_radial(G.gc.fam.data(), (int)G.gc.fam.size(), G.gc.coef.data(), x, GR_M, F);
}

bool rows_a(HostGrid &G, int cell, double xi, double D, double *V, bool check = false) {
  const int ix = cell / GR_NT, o = grid_octave(ix);
  Octave &O = G.oct[check][o];
  if (O.q.x.empty()) {
    const double lo = std::ldexp(1.0, GR_XLO + o);
    if (!grid_quad(G.all, 4, lo, 2.0 * lo, O.q, check ? GR_CHECK_SCALE : 1.0)) return false;
    O.F.resize(O.q.x.size() * GR_ROWS);
    for (size_t i = 0; i < O.q.x.size(); ++i) radial(G, O.q.x[i], &O.F[i * GR_ROWS]);
  }
  long double acc[GR_ROWS] = {0.0L};   // (the builder's sums carry their rounding)
  double jh[GR_ROWS];
  for (size_t i = 0; i < O.q.x.size(); ++i) {
    const double x = O.q.x[i], e = O.q.w[i] * std::exp(-xi * (x - D) * (x - D));
    if (e == 0.0) continue;
    grid_jhat(G.ztab.data(), 2.0 * xi * D * x, jh);
    for (int m = 0; m <= GR_M; ++m) acc[m] += (long double)(e * jh[m]) * O.F[i * GR_ROWS + m];
  }
  double f = 4.0 * xi * std::sqrt(xi);
  for (int m = 0; m <= GR_M; ++m, f *= 2.0 * xi) V[m] = f * (double)acc[m];
  return true;
}

// Region B, as the library's builder: F_m interpolated for the cell's rows, F_m
// itself and the longer rule for the check.
void rows_b(HostGrid &G, int cell, double xi, double D, double *V, bool check = false) {
  double lo, hi, X[GR_NB], B[GR_NB], F[GR_NB][GR_ROWS];
  grid_cellu(cell, &lo, &hi);
  const double D0 = std::sqrt(0.5 * (lo + hi)), is = 1.0 / std::sqrt(xi);
  for (int j = 0; j < GR_NB; ++j) {
    const double th = M_PI * (j + 0.5) / GR_NB;
    X[j] = D0 * (1.0 + (GR_BW + 0.02) * std::cos(th));
    B[j] = ((j & 1) ? -1.0 : 1.0) * std::sin(th);
    if (!check) radial(G, X[j], F[j]);
  }
  const double b = check ? 0.0 : grid_slope(F[GR_NB - 1], F[0], X[0] - X[GR_NB - 1]);
  const int nh = check ? GR_NHC : GR_NH;
  double hx[GR_NHC], hw[GR_NHC], acc[GR_ROWS] = {0.0}, jh[GR_ROWS], f[GR_ROWS];
  gauss_hermite(nh, hx, hw);
  for (int i = 0; i < nh; ++i) {
    const double x = D + hx[i] * is;
    grid_jhat(G.ztab.data(), 2.0 * xi * D * x, jh);
    if (check) {
      radial(G, x, f);
    } else {
      double den = 0.0;
      for (int j = 0; j < GR_NB; ++j) den += B[j] / (x - X[j]);
      for (int m = 0; m <= GR_M; ++m) {
        f[m] = 0.0;
        for (int j = 0; j < GR_NB; ++j) f[m] += B[j] / (x - X[j]) / den * F[j][m] * std::exp(-b * (X[j] - D0));
        f[m] *= std::exp(b * (x - D0));
      }
    }
    for (int m = 0; m <= GR_M; ++m) acc[m] = std::fma(hw[i] * jh[m], f[m], acc[m]);
  }
  double c = 4.0 * xi;
  for (int m = 0; m <= GR_M; ++m, c *= 2.0 * xi) V[m] = c * acc[m];
}

const std::vector<double> *cell_of(HostGrid &G, int cell) {
  auto it = G.cells.find(cell);
  if (it != G.cells.end()) return &it->second;
  double lo, hi, V[GR_NC][GR_ROWS];
  grid_cellu(cell, &lo, &hi);
  for (int n = 0; n < GR_NC; ++n) {
    const double a = G.node[(size_t)n];
    if (cell < GR_NX * GR_NT) {
      const double *r = &G.xt[(size_t)GR_XT * (size_t)(cell / GR_NT)];
      if (!rows_a(G, cell, grid_xi(r, a), std::sqrt(mul_rn(0.5 * (lo + hi), r[1])), V[n])) return nullptr;
    } else {
      rows_b(G, cell, 2.0 * GR_TB / (hi * (a + 1.0)), std::sqrt(0.5 * (lo + hi)), V[n]);
    }
  }
  std::vector<double> C((size_t)GR_CELL);
  for (int m = 0; m < GR_ROWS; ++m)
    for (int i = 0; i < GR_NC; ++i) {
      dd s{0.0, 0.0};
      for (int n = 0; n < GR_NC; ++n) s = dd_add(s, dd_muld(G.conv[i][n], V[n][m]));
      C[(size_t)(m * GR_NC + i)] = s.h;
    }
  return &(G.cells[cell] = C);
}

template <int L>
void eval(const double *cells, const GridPoint &pt, double *h) {
  grid_eval<L, true>(cells, pt, L, h);
}

}  // namespace

extern "C" {

// The grid of class cls for a factor pair given as terms c, a, b, g; null when
// the grid does not serve it.
void *grid_host_new(const double *t, int nt, const double *tp, int ntp, int cls) {
  f12::TermList T1, T2;
  for (int i = 0; i < nt; ++i) T1.push_back({t[4 * i], t[4 * i + 1], t[4 * i + 2], t[4 * i + 3]});
  for (int i = 0; i < ntp; ++i) T2.push_back({tp[4 * i], tp[4 * i + 1], tp[4 * i + 2], tp[4 * i + 3]});
  f12::simplify(T1);
  f12::simplify(T2);
  HostGrid *G = new HostGrid;
  for (int k = 0; k < 4; ++k) {
    const bool s = grid_families(f12::kernel_terms(kCls[k], T1, T2), G->all[k]);
    if (!s) G->all[k] = GridClass{};
    if (kCls[k] == cls) {
      G->served = s;
      G->gc = G->all[k];
    }
  }
  if (!G->served) {
    delete G;
    return nullptr;
  }
  grid_ztab(G->ztab);
  G->node.resize(GR_NC);
  grid_nodes(G->node.data());
  grid_conversion(G->conv);
  G->xt.assign((size_t)GR_XT * GR_NX, 0.0);
  for (int i = 0; i < GR_NX; ++i) grid_xcell(i, &G->xt[(size_t)GR_XT * (size_t)i]);
  return G;
}

void grid_host_free(void *g) { delete (HostGrid *)g; }

// Whether the library accepts the cell that holds (xi, D); -1: outside the grid.
int grid_host_ok(void *g, double xi, double D) {
  HostGrid &G = *(HostGrid *)g;
  const GridPoint pt = grid_point(G.xt.data(), 1.0 / xi, D * D);
  const std::vector<double> *C = pt.cell < 0 ? nullptr : cell_of(G, pt.cell);
  if (!C) return -1;
  double cxi, cu, V[GR_ROWS];
  grid_check_point(G.xt.data(), pt.cell, &cxi, &cu);
  if (pt.cell < GR_NX * GR_NT) {
    if (!rows_a(G, pt.cell, cxi, std::sqrt(cu), V, true)) return -1;
  } else {
    rows_b(G, pt.cell, cxi, std::sqrt(cu), V, true);
  }
  return grid_cell_ok(G.xt.data(), pt.cell, C->data(), V) ? 1 : 0;
}

// hat g_l, l = 0..L, at (xi, D) as a kernel of highest order L takes it.
// Returns 0, or -1 when the point is outside the grid.
int grid_host_eval(void *g, double xi, double D, int L, double *out) {
  HostGrid &G = *(HostGrid *)g;
  GridPoint pt = grid_point(G.xt.data(), 1.0 / xi, D * D);
  const std::vector<double> *C = pt.cell < 0 ? nullptr : cell_of(G, pt.cell);
  if (!C) return -1;
  pt.cell = 0;
  double h[GR_ROWS];
  switch (L) {
    case 0: eval<0>(C->data(), pt, h); break;
    case 2: eval<2>(C->data(), pt, h); break;
    case 4: eval<4>(C->data(), pt, h); break;
    case 6: eval<6>(C->data(), pt, h); break;
    case 8: eval<8>(C->data(), pt, h); break;
    case 14: eval<14>(C->data(), pt, h); break;
    default: return -1;
  }
  for (int l = 0; l <= L; ++l) out[l] = h[l] / std::sqrt(xi);
  return 0;
}

}  // extern "C"
