// grid.cu -- the builder of the auxiliary grids (auxgrid.cuh) and their
// sharing between contexts.
//
// Four kernels, once per factor: the summed kernel derivatives F_m at the
// quadrature points of every octave of xi (double-double, one thread per
// point), the rows at the Chebyshev points of every cell (one thread per cell
// and point, all classes at once, since e^{-z} j_m is theirs in common), the
// same for the far region, and the polynomial coefficients with the check of
// every cell at one of its corners.  Bound by the FP64 pipe; setting a
// factor pair with four kernels takes 0.17 s with it.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <mutex>

#include "grid.h"
#include "gridtab.h"

using namespace f12dev;

namespace f12grid {

namespace {

constexpr int NCLS = 4;
constexpr int kClass[NCLS] = {2, 3, 4, 6};
constexpr int NODES = GR_NC + 1;              // Chebyshev points and the check point
constexpr int ITB = 16;                       // cells of T' per block of k_rows_a
constexpr int NOCT = GR_XHI - GR_XLO;
constexpr int TILE = 16;                      // quadrature points staged at a time

struct ClassDev {
  const GridFam *fam;
  const dd *coef;
  int nfam;
  double b;   // largest b of its families
};

struct Build {
  int ncls;
  ClassDev cls[NCLS];
  double *cells[NCLS];
  unsigned char *ok[NCLS];
  double *V;                 // [cell][node][class][row]
  // quadrature points, octave after octave
  const double *x, *w;
  const double *F;           // [point][class][row]
  double *Fw;
  int npts;
  const int *pt0;            // [NOCT + 1] first point of an octave
  const double *edge;        // [NOCT][GR_MAXPANEL + 1]
  const int *npanel;         // [NOCT]
  double bpos, bneg;
  const double *xt, *ztab, *node, *ghx, *ghw, *bx, *bw;
  const dd *conv;
};

// Check point of a cell: one of its four corners.
__device__ __forceinline__ double check_a(int cell) { return (cell & 1) ? 1.0 : -1.0; }
__device__ __forceinline__ double check_s(int cell) { return (cell & 2) ? 0.5 : -0.5; }   // in units of the cell's width

__global__ void k_radial(Build B) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x, c = blockIdx.y;
  if (i >= B.npts) return;
  grid_radial(B.cls[c].fam, B.cls[c].nfam, B.cls[c].coef, B.x[i], GR_M, B.Fw + ((size_t)i * B.ncls + c) * GR_ROWS);
}

// Region A.  A block takes one cell of xi and ITB cells of T'; a thread one
// of their (cell, node) pairs.  Bound by the FP64 pipe (e^{-z} j_m and the
// sums); F_m of a tile of points is staged in shared memory for all threads.  A
// tile's sum is added to the total with its rounding kept: some 300 points count,
// and added one by one they left 4 u of noise in every row.
__global__ void __launch_bounds__(NODES *ITB) k_rows_a(Build B) {
  __shared__ double sF[TILE * NCLS * GR_ROWS];
  __shared__ double sx[TILE], sw[TILE];
  const int ix = blockIdx.x, oct = grid_octave(ix);
  const int n = threadIdx.x % NODES, it0 = blockIdx.y * ITB, it = it0 + threadIdx.x / NODES;
  const double c = B.xt[GR_XT * ix], ic = B.xt[GR_XT * ix + 1];
  const bool live = it < GR_NT;
  const int cell = ix * GR_NT + it;
  double lo = 0.0, hi = 0.0;
  if (live) grid_tcell(it, &lo, &hi);
  const double a = n < GR_NC ? B.node[n] : check_a(cell);
  const double xi = grid_xi(B.xt + GR_XT * ix, a);
  double u = mul_rn(0.5 * (lo + hi), ic);
  if (n == GR_NC) u += check_s(cell) * (hi - lo) * ic;
  const double D = sqrt(u);
  const int nrow = B.ncls * GR_ROWS;
  double acc[NCLS * GR_ROWS];
  dd tot[NCLS * GR_ROWS];
  for (int k = 0; k < nrow; ++k) {
    acc[k] = 0.0;
    tot[k] = dd{0.0, 0.0};
  }
  // panels that reach the window of any node of the block: past it e^{-xi (x-D)^2}
  // times the growth of j_m (below D) and of F_m (above) is below double precision
  double clo, chi;   // ends of the cell of xi
  grid_xends(ix, &clo, &chi);
  double tl, th, dummy;
  grid_tcell(it0, &tl, &dummy);
  grid_tcell(min(it0 + ITB, GR_NT) - 1, &dummy, &th);
  const double wl = sqrt(tl / c) - 10.5 / sqrt(clo) - 0.5 * B.bneg / clo;
  const double wh = sqrt(th / c) + 8.5 / sqrt(clo) + 0.5 * B.bpos / clo;
  const double *edge = B.edge + (size_t)oct * (GR_MAXPANEL + 1);
  const int p0 = B.pt0[oct];
  for (int p = 0; p < B.npanel[oct]; ++p) {
    if (edge[p + 1] < wl || edge[p] > wh) continue;
    const int i0 = p0 + (p == 0 ? 0 : GR_NQ0 + (p - 1) * GR_NQ), np = p == 0 ? GR_NQ0 : GR_NQ;
    for (int t0 = 0; t0 < np; t0 += TILE) {
      __syncthreads();
      for (int k = threadIdx.x; k < TILE * nrow; k += blockDim.x) sF[k] = B.F[(size_t)(i0 + t0) * nrow + k];
      if (threadIdx.x < TILE) {
        sx[threadIdx.x] = B.x[i0 + t0 + threadIdx.x];
        sw[threadIdx.x] = B.w[i0 + t0 + threadIdx.x];
      }
      __syncthreads();
      if (!live) continue;
      for (int i = 0; i < TILE; ++i) {
        const double x = sx[i], e = sw[i] * exp(-xi * (x - D) * (x - D));
        double jh[GR_ROWS];
        grid_jhat(B.ztab, 2.0 * xi * D * x, jh);
        const double *f = sF + i * nrow;
        for (int m = 0; m <= GR_M; ++m) {
          const double v = e * jh[m];
          for (int k = 0; k < B.ncls; ++k) acc[k * GR_ROWS + m] = fma(v, f[k * GR_ROWS + m], acc[k * GR_ROWS + m]);
        }
      }
      for (int k = 0; k < nrow; ++k) {
        const dd s = dd_sum(tot[k].h, acc[k]);
        tot[k] = dd{s.h, tot[k].l + s.l};
        acc[k] = 0.0;
      }
    }
  }
  if (!live) return;
  double f = 4.0 * xi * sqrt(xi);
  double *V = B.V + ((size_t)cell * NODES + n) * nrow;
  for (int m = 0; m <= GR_M; ++m) {
    for (int k = 0; k < B.ncls; ++k) V[k * GR_ROWS + m] = f * (tot[k * GR_ROWS + m].h + tot[k * GR_ROWS + m].l);
    f *= 2.0 * xi;
  }
}

// Region B: one block per cell of u.  F_m is evaluated at the Chebyshev points
// of x/D and interpolated at the quadrature nodes.
__global__ void __launch_bounds__(128) k_rows_b(Build B) {
  extern __shared__ double sB[];   // [GR_NB][ncls][row], then a row of rows per node
  const int iu = blockIdx.x, cell = GR_NX * GR_NT + iu, nrow = B.ncls * GR_ROWS;
  double lo, hi;
  grid_ucell(iu, &lo, &hi);
  // the check point has its own u, inside the interpolated range of x
  const double D0 = sqrt(0.5 * (lo + hi));
  for (int t = threadIdx.x; t < GR_NB * B.ncls; t += blockDim.x) {
    const int j = t / B.ncls, k = t % B.ncls;
    const double x = D0 * (1.0 + (GR_BW + 0.02) * B.bx[j]);
    double *F = sB + j * nrow + k * GR_ROWS;
    grid_radial(B.cls[k].fam, B.cls[k].nfam, B.cls[k].coef, x, GR_M, F);
    // interpolated without the growth of e^{bx}, which would cost the small values their digits
    const double e = exp(-B.cls[k].b * (x - D0));
    for (int m = 0; m <= GR_M; ++m) F[m] *= e;
  }
  __syncthreads();
  double *acc = sB + GR_NB * nrow + threadIdx.x * (nrow + 1);
  const int n = threadIdx.x;
  if (n >= NODES) return;
  const double a = n < GR_NC ? B.node[n] : 0.97 * check_a(cell);   // (a = -1 is xi = infinity)
  const double xi = 2.0 * GR_TB / (hi * (a + 1.0)), is = 1.0 / sqrt(xi);
  const double D = n < GR_NC ? D0 : sqrt(0.5 * (lo + hi) + check_s(cell) * (hi - lo));
  for (int k = 0; k < nrow; ++k) acc[k] = 0.0;
  for (int i = 0; i < GR_NH; ++i) {
    const double x = D + B.ghx[i] * is;
    double jh[GR_ROWS], bw[GR_NB], den = 0.0;
    grid_jhat(B.ztab, 2.0 * xi * D * x, jh);
    const double y = (x / D0 - 1.0) / (GR_BW + 0.02);
    int hit = -1;
    for (int j = 0; j < GR_NB; ++j) {
      const double d = y - B.bx[j];
      if (d == 0.0) hit = j;
      bw[j] = d == 0.0 ? 0.0 : B.bw[j] / d;
      den += bw[j];
    }
    for (int j = 0; j < GR_NB; ++j) bw[j] = hit < 0 ? bw[j] / den : (j == hit ? 1.0 : 0.0);
    for (int c = 0; c < B.ncls; ++c) {
      const double e = B.ghw[i] * exp(B.cls[c].b * (x - D0));
      for (int m = 0; m <= GR_M; ++m) {
        const int k = c * GR_ROWS + m;
        double f = 0.0;
        for (int j = 0; j < GR_NB; ++j) f = fma(bw[j], sB[j * nrow + k], f);
        acc[k] = fma(e * jh[m], f, acc[k]);
      }
    }
  }
  double *V = B.V + ((size_t)cell * NODES + n) * nrow;
  double f = 4.0 * xi;
  for (int m = 0; m <= GR_M; ++m) {
    for (int k = 0; k < B.ncls; ++k) V[k * GR_ROWS + m] = f * acc[k * GR_ROWS + m];
    f *= 2.0 * xi;
  }
}

// Coefficients of every row: sum_n conv[i][n] v_n in double-double (the
// entries of conv reach 2^11, which plain sums would lose).
__global__ void k_fit(Build B) {
  const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  const int nrow = B.ncls * GR_ROWS;
  const int64_t cell = t / nrow;
  if (cell >= GR_CELLS) return;
  const int k = (int)(t % nrow), c = k / GR_ROWS, m = k % GR_ROWS;
  double v[GR_NC];
  for (int n = 0; n < GR_NC; ++n) v[n] = B.V[((size_t)cell * NODES + n) * nrow + k];
  double *out = B.cells[c] + (size_t)cell * GR_CELL + m * GR_NC;
  for (int i = 0; i < GR_NC; ++i) {
    dd s{0.0, 0.0};
    for (int n = 0; n < GR_NC; ++n) s = dd_add(s, dd_muld(B.conv[i * GR_NC + n], v[n]));
    out[i] = s.h;
  }
}

// A cell is in order when orders 0..8 at its check point agree with the
// quadrature to kCellTol of the sum of the terms' magnitudes (the scale of the
// result where it passes through zero).
constexpr double kCellTol = 3e-13;
__global__ void k_check(Build B) {
  const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  const int cell = (int)(t / B.ncls), c = (int)(t % B.ncls);
  if (cell >= GR_CELLS) return;
  const int nrow = B.ncls * GR_ROWS;
  const double *V = B.V + ((size_t)cell * NODES + GR_NC) * nrow + c * GR_ROWS;
  const double *C = B.cells[c] + (size_t)cell * GR_CELL;
  double lo, hi, hd, a = check_a(cell);
  if (cell < GR_NX * GR_NT) {
    grid_tcell(cell % GR_NT, &lo, &hi);
    hd = 0.5 * check_s(cell) * (hi - lo) * B.xt[GR_XT * (cell / GR_NT) + 1];
  } else {
    grid_ucell(cell - GR_NX * GR_NT, &lo, &hi);
    hd = 0.5 * check_s(cell) * (hi - lo);
    a *= 0.97;
  }
  constexpr int L = 8, N = grid_terms(L);
  double row[L + N + 1];
  for (int m = 0; m <= L + N; ++m) {
    double r = C[m * GR_NC + GR_NC - 1];
    for (int i = GR_NC - 2; i >= 0; --i) r = fma(r, a, C[m * GR_NC + i]);
    row[m] = r;
  }
  // region B: e^{bx} must vary little enough over a width for the rule's 20 nodes
  bool ok = cell < GR_NX * GR_NT || fmax(B.bpos, B.bneg) * sqrt(hi / GR_TB) <= 3.0;
  for (int l = 0; l <= L; ++l) {
    double s = 0.0, sc = 0.0, w = 1.0;
    for (int k = 0; k <= N; ++k) {
      s = fma(row[l + k], w, s);
      sc += fabs(row[l + k] * w);
      w *= hd / (k + 1);
    }
    ok = ok && fabs(s - V[l]) <= kCellTol * sc;   // false for NaN
  }
  B.ok[c][cell] = ok ? 1 : 0;
}

std::mutex g_mu;
std::vector<std::weak_ptr<const AuxGrid>> g_all;

bool same_terms(const f12::TermList &x, const f12::TermList &y) {
  if (x.size() != y.size()) return false;
  for (size_t i = 0; i < x.size(); ++i)
    if (x[i].c != y[i].c || x[i].a != y[i].a || x[i].b != y[i].b || x[i].g != y[i].g) return false;
  return true;
}

// Device allocations of a build, freed on every way out.
struct Temp {
  std::vector<void *> p;
  ~Temp() {
    for (void *q : p) cudaFree(q);
  }
  template <class T>
  T *up(const std::vector<T> &v, bool &good) {
    T *d = get<T>(v.size(), good);
    if (good && !v.empty() && cudaMemcpy(d, v.data(), sizeof(T) * v.size(), cudaMemcpyHostToDevice) != cudaSuccess)
      good = false;
    return d;
  }
  template <class T>
  T *get(size_t n, bool &good) {
    void *q = nullptr;
    if (!good || cudaMalloc(&q, sizeof(T) * std::max<size_t>(n, 1)) != cudaSuccess) {
      good = false;
      cudaGetLastError();
      return nullptr;
    }
    p.push_back(q);
    return (T *)q;
  }
};

}  // namespace

AuxGrid::~AuxGrid() {
  int cur = 0;
  cudaGetDevice(&cur);
  cudaSetDevice(device);
  for (int c = 1; c <= 6; ++c)
    if (c != 5) {
      cudaFree(cells[c]);
      cudaFree(ok[c]);
    }
  cudaFree(xt);
  cudaSetDevice(cur);
}

std::shared_ptr<const AuxGrid> acquire(int device, const f12::TermList kt[7], const bool want[7], cudaStream_t st) {
  std::lock_guard<std::mutex> lk(g_mu);
  std::vector<f12::TermList> key(7);
  for (int c = 2; c <= 6; ++c)
    if (c != 5 && want[c]) key[(size_t)c] = kt[c];
  for (size_t i = 0; i < g_all.size();) {
    if (std::shared_ptr<const AuxGrid> g = g_all[i].lock()) {
      bool same = g->device == device;
      for (size_t c = 0; c < 7 && same; ++c) same = same_terms(g->key[c], key[c]);
      if (same) return g;
      ++i;
    } else {
      g_all.erase(g_all.begin() + (long)i);
    }
  }
  Build B{};
  GridClass gc[NCLS];
  int cls_of[NCLS];
  double bpos = 0.0, bneg = 0.0;
  for (int k = 0; k < NCLS; ++k)
    if (want[kClass[k]] && grid_families(kt[kClass[k]], gc[B.ncls])) {
      bpos = std::max(bpos, gc[B.ncls].bpos);
      bneg = std::max(bneg, gc[B.ncls].bneg);
      cls_of[B.ncls++] = kClass[k];
    }
  if (!B.ncls) return nullptr;
  std::vector<double> x, w, edge((size_t)NOCT * (GR_MAXPANEL + 1), 0.0);
  std::vector<int> pt0, npanel;
  for (int o = 0; o < NOCT; ++o) {
    GridQuad q;
    const double lo = std::ldexp(1.0, GR_XLO + o);
    if (!grid_quad(gc, B.ncls, lo, 2.0 * lo, q)) return nullptr;
    pt0.push_back((int)x.size());
    npanel.push_back((int)q.edge.size() - 1);
    x.insert(x.end(), q.x.begin(), q.x.end());
    w.insert(w.end(), q.w.begin(), q.w.end());
    std::copy(q.edge.begin(), q.edge.end(), edge.begin() + (size_t)o * (GR_MAXPANEL + 1));
  }
  pt0.push_back((int)x.size());
  static const std::vector<double> ztab = [] {
    std::vector<double> t;
    grid_ztab(t);
    return t;
  }();
  std::vector<dd> conv((size_t)GR_NC * GR_NC);
  {
    dd m[GR_NC][GR_NC];
    grid_conversion(m);
    std::memcpy(conv.data(), m, sizeof(m));
  }
  std::vector<double> node(GR_NC), ghx(GR_NH), ghw(GR_NH), bx(GR_NB), bw(GR_NB), xt((size_t)GR_XT * GR_NX, 0.0);
  grid_nodes(node.data());
  gauss_hermite(GR_NH, ghx.data(), ghw.data());
  for (int j = 0; j < GR_NB; ++j) {   // Chebyshev points of the first kind and their barycentric weights
    const double th = M_PI * (j + 0.5) / GR_NB;
    bx[(size_t)j] = std::cos(th);
    bw[(size_t)j] = ((j & 1) ? -1.0 : 1.0) * std::sin(th);
  }
  for (int i = 0; i < GR_NX; ++i) grid_xcell(i, &xt[(size_t)GR_XT * (size_t)i]);

  std::shared_ptr<AuxGrid> g = std::make_shared<AuxGrid>();
  g->device = device;
  g->key = key;
  Temp tmp;
  bool good = true;
  for (int k = 0; k < B.ncls && good; ++k) {
    B.cls[k] = ClassDev{tmp.up(gc[k].fam, good), tmp.up(gc[k].coef, good), (int)gc[k].fam.size(), gc[k].bmax};
    const int c = cls_of[k];
    good = good && cudaMalloc((void **)&g->cells[c], sizeof(double) * (size_t)GR_CELLS * GR_CELL) == cudaSuccess &&
           cudaMalloc((void **)&g->ok[c], (size_t)GR_CELLS) == cudaSuccess;
    B.cells[k] = g->cells[c];
    B.ok[k] = g->ok[c];
    g->bytes += sizeof(double) * (size_t)GR_CELLS * GR_CELL + (size_t)GR_CELLS;
  }
  good = good && cudaMalloc((void **)&g->xt, sizeof(double) * xt.size()) == cudaSuccess &&
         cudaMemcpy(g->xt, xt.data(), sizeof(double) * xt.size(), cudaMemcpyHostToDevice) == cudaSuccess;
  const int nrow = B.ncls * GR_ROWS;
  B.npts = (int)x.size();
  B.x = tmp.up(x, good);
  B.w = tmp.up(w, good);
  B.pt0 = tmp.up(pt0, good);
  B.npanel = tmp.up(npanel, good);
  B.edge = tmp.up(edge, good);
  B.ztab = tmp.up(ztab, good);
  B.node = tmp.up(node, good);
  B.ghx = tmp.up(ghx, good);
  B.ghw = tmp.up(ghw, good);
  B.bx = tmp.up(bx, good);
  B.bw = tmp.up(bw, good);
  B.conv = tmp.up(conv, good);
  B.Fw = tmp.get<double>((size_t)B.npts * nrow, good);
  B.F = B.Fw;
  B.V = tmp.get<double>((size_t)GR_CELLS * NODES * nrow, good);
  B.xt = g->xt;
  B.bpos = bpos;
  B.bneg = bneg;
  if (!good) {
    cudaGetLastError();
    return nullptr;
  }
  k_radial<<<dim3((unsigned)((B.npts + 63) / 64), (unsigned)B.ncls), 64, 0, st>>>(B);
  k_rows_a<<<dim3(GR_NX, (GR_NT + ITB - 1) / ITB), NODES * ITB, 0, st>>>(B);
  const size_t smb = sizeof(double) * ((size_t)GR_NB * nrow + (size_t)NODES * (nrow + 1));
  cudaFuncSetAttribute(k_rows_b, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smb);
  k_rows_b<<<GR_NU, 128, smb, st>>>(B);
  k_fit<<<(unsigned)(((int64_t)GR_CELLS * nrow + 127) / 128), 128, 0, st>>>(B);
  k_check<<<(unsigned)(((int64_t)GR_CELLS * B.ncls + 127) / 128), 128, 0, st>>>(B);
  if (cudaGetLastError() != cudaSuccess || cudaStreamSynchronize(st) != cudaSuccess) return nullptr;
  for (int k = 0; k < B.ncls; ++k) {
    const int c = cls_of[k];
    g->ok_host[c].resize(GR_CELLS);
    if (cudaMemcpy(g->ok_host[c].data(), g->ok[c], GR_CELLS, cudaMemcpyDeviceToHost) != cudaSuccess) return nullptr;
  }
  g_all.push_back(g);
  return g;
}

bool covers(const AuxGrid &g, int cls, double xi_lo, double xi_hi, double dmax) {
  const int c = cls == 5 ? 3 : cls;
  if (!g.cells[c]) return false;
  // a little room for the rounding of the exponents' sums and distances, and
  // for grid_point's single-precision cell of xi
  const double lo = xi_lo * (1.0 - 1e-6), hi = xi_hi * (1.0 + 1e-6), u = dmax * dmax * (1.0 + 1e-9) + 1e-9;
  const int x0 = grid_xindex(grid_hi(lo)), x1 = grid_xindex(grid_hi(hi));
  if (!(lo > 0.0) || x0 < 0 || x1 < x0) return false;
  const std::vector<unsigned char> &ok = g.ok_host[c];
  for (int ix = x0; ix <= x1; ++ix) {
    double r[GR_XT];
    grid_xcell(ix, r);
    const double cc = r[0];
    for (int it = 0; it < GR_NT; ++it) {
      double tl, th;
      grid_tcell(it, &tl, &th);
      if (tl > cc * u) break;
      if (!ok[(size_t)ix * GR_NT + it]) return false;
    }
  }
  // region B, from the smallest u that reaches it at the largest xi
  double r[GR_XT];
  grid_xcell(x1, r);
  const double cc = r[0];
  if (cc * u >= GR_TMAX) {
    if (u >= std::ldexp(1.0, GR_UHI)) return false;
    for (int iu = 0; iu < GR_NU; ++iu) {
      double ul, uh;
      grid_ucell(iu, &ul, &uh);
      if (uh * cc < GR_TMAX || ul > u) continue;
      if (!ok[(size_t)GR_NX * GR_NT + iu]) return false;
    }
    if (GR_TMAX / cc < std::ldexp(1.0, GR_ULO)) return false;
  }
  return true;
}

}  // namespace f12grid
