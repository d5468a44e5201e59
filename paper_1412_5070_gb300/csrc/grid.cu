// grid.cu -- the builder of the auxiliary grids (auxgrid.cuh) and their
// sharing between contexts.
//
// Five kernels, once per factor: the summed kernel derivatives F_m at the
// quadrature points of every octave of xi (double-double, one thread per
// point), the rows at the Chebyshev points of every cell (one thread per cell
// and point, all classes at once, since e^{-z} j_m is theirs in common), the
// same for the far region, the polynomial coefficients, and the check of every
// cell at one point.  The rows of that point come from a quadrature of its own
// (the first two kernels again, with narrower panels): against the cells' own
// quadrature, what that does not resolve would pass.  Bound by the FP64 pipe;
// setting a factor pair with four kernels takes 0.23 s with it.
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
constexpr int ITB = 16, ITC = 32;             // cells of T' per block of k_rows_a, of its check
constexpr int NOCT = GR_XHI - GR_XLO;
constexpr int TILE = 16;                      // quadrature points staged at a time

struct ClassDev {
  const GridFam *fam;
  const dd *coef;
  int nfam;
};

struct Build {
  int ncls;
  ClassDev cls[NCLS];
  double *cells[NCLS];
  unsigned char *ok[NCLS];
  double *V;                 // [cell][node][class][row]
  double bpos, bneg;
  const double *xt, *ztab, *node, *ghx, *ghw, *ghcx, *ghcw, *bx, *bw;
  const dd *conv;
};

// Quadrature points, octave after octave.
struct Quad {
  const double *x, *w;
  double *F;                 // [point][class][row]
  int npts, rows;            // rows: 0 .. rows - 1
  const int *pt0;            // [NOCT + 1] first point of an octave
  const double *edge;        // [NOCT][GR_MAXPANEL + 1]
  const int *npanel;         // [NOCT]
};

__global__ void k_radial(Build B, Quad Q) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x, c = blockIdx.y;
  if (i >= Q.npts) return;
  grid_radial(B.cls[c].fam, B.cls[c].nfam, B.cls[c].coef, Q.x[i], Q.rows - 1, Q.F + ((size_t)i * B.ncls + c) * Q.rows);
}

// Region A.  A block takes one cell of xi and IT cells of T'; a thread one
// of their (cell, node) pairs, or (CHECK) a cell's check point.  Bound by the
// FP64 pipe (e^{-z} j_m and the sums); F_m of a tile of points is staged in shared
// memory for all threads.  A
// tile's sum is added to the total with its rounding kept: some 300 points count,
// and added one by one they left 4 u of noise in every row.  A check takes the
// rows of the orders that are served only.
template <bool CHECK>
__global__ void __launch_bounds__(CHECK ? ITC : GR_NC *ITB) k_rows_a(Build B, Quad Q) {
  constexpr int NN = CHECK ? 1 : GR_NC, IT = CHECK ? ITC : ITB, R = CHECK ? GR_LMAX + 1 : GR_ROWS;
  __shared__ double sF[TILE * NCLS * R];
  __shared__ double sx[TILE], sw[TILE];
  const int ix = blockIdx.x, oct = grid_octave(ix);
  const int n = CHECK ? GR_NC : threadIdx.x % NN, it0 = blockIdx.y * IT, it = it0 + threadIdx.x / NN;
  const double c = B.xt[GR_XT * ix], ic = B.xt[GR_XT * ix + 1];
  const bool live = it < GR_NT;
  const int cell = ix * GR_NT + min(it, GR_NT - 1);
  double xi, u;
  if (CHECK) {
    grid_check_point(B.xt, cell, &xi, &u);
  } else {
    double lo, hi;
    grid_cellu(cell, &lo, &hi);
    xi = grid_xi(B.xt + GR_XT * ix, B.node[n]);
    u = mul_rn(0.5 * (lo + hi), ic);
  }
  const double D = sqrt(u);
  const int nrow = B.ncls * R;
  double acc[NCLS * R];
  dd tot[NCLS * R];
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
  grid_tcell(min(it0 + IT, GR_NT) - 1, &dummy, &th);
  const double wl = sqrt(tl / c) - 10.5 / sqrt(clo) - 0.5 * B.bneg / clo;
  const double wh = sqrt(th / c) + 8.5 / sqrt(clo) + 0.5 * B.bpos / clo;
  const double *edge = Q.edge + (size_t)oct * (GR_MAXPANEL + 1);
  const int p0 = Q.pt0[oct];
  for (int p = 0; p < Q.npanel[oct]; ++p) {
    if (edge[p + 1] < wl || edge[p] > wh) continue;
    const int i0 = p0 + (p == 0 ? 0 : GR_NQ0 + (p - 1) * GR_NQ), np = p == 0 ? GR_NQ0 : GR_NQ;
    for (int t0 = 0; t0 < np; t0 += TILE) {
      __syncthreads();
      for (int k = threadIdx.x; k < TILE * nrow; k += blockDim.x) sF[k] = Q.F[(size_t)(i0 + t0) * nrow + k];
      if (threadIdx.x < TILE) {
        sx[threadIdx.x] = Q.x[i0 + t0 + threadIdx.x];
        sw[threadIdx.x] = Q.w[i0 + t0 + threadIdx.x];
      }
      __syncthreads();
      if (!live) continue;
      for (int i = 0; i < TILE; ++i) {
        const double x = sx[i], e = sw[i] * exp(-xi * (x - D) * (x - D));
        double jh[GR_ROWS];
        grid_jhat(B.ztab, 2.0 * xi * D * x, jh);
        const double *f = sF + i * nrow;
        for (int m = 0; m < R; ++m) {
          const double v = e * jh[m];
          for (int k = 0; k < B.ncls; ++k) acc[k * R + m] = fma(v, f[k * R + m], acc[k * R + m]);
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
  double *V = B.V + ((size_t)cell * NODES + n) * B.ncls * GR_ROWS;
  for (int m = 0; m < R; ++m) {
    for (int k = 0; k < B.ncls; ++k) V[k * GR_ROWS + m] = f * (tot[k * R + m].h + tot[k * R + m].l);
    f *= 2.0 * xi;
  }
}

// Region B: one block per cell of u.  F_m is evaluated at the Chebyshev points
// of x/D and interpolated at the quadrature nodes; at the nodes of the check
// point's rule it is evaluated itself, for the orders that are served.  A thread
// per evaluation, and the check point in a warp of its own.
constexpr int TRB = 288;
static_assert(TRB >= (GR_NB + GR_NHC) * NCLS && GR_NC <= 32, "a thread each");
__global__ void __launch_bounds__(TRB) k_rows_b(Build B) {
  extern __shared__ double sB[];   // [GR_NB][ncls][row], [GR_NHC][ncls][row], then a row of rows per node
  const int iu = blockIdx.x, cell = GR_NX * GR_NT + iu, nrow = B.ncls * GR_ROWS;
  double *sC = sB + GR_NB * nrow;
  double lo, hi, cxi, cu;
  grid_ucell(iu, &lo, &hi);
  grid_check_point(B.xt, cell, &cxi, &cu);
  const double D0 = sqrt(0.5 * (lo + hi)), cD = sqrt(cu), cis = 1.0 / sqrt(cxi);
  for (int t = threadIdx.x; t < (GR_NB + GR_NHC) * B.ncls; t += blockDim.x) {
    const int j = t / B.ncls, k = t % B.ncls;
    const double x = j < GR_NB ? D0 * (1.0 + (GR_BW + 0.02) * B.bx[j]) : cD + B.ghcx[j - GR_NB] * cis;
    grid_radial(B.cls[k].fam, B.cls[k].nfam, B.cls[k].coef, x, j < GR_NB ? GR_M : GR_LMAX, sB + j * nrow + k * GR_ROWS);
  }
  __syncthreads();
  double b[NCLS];
  const double xlo = D0 * (1.0 + (GR_BW + 0.02) * B.bx[GR_NB - 1]), xhi = D0 * (1.0 + (GR_BW + 0.02) * B.bx[0]);
  for (int k = 0; k < B.ncls; ++k)
    b[k] = grid_slope(sB + (GR_NB - 1) * nrow + k * GR_ROWS, sB + k * GR_ROWS, xhi - xlo);
  __syncthreads();
  for (int t = threadIdx.x; t < GR_NB * B.ncls; t += blockDim.x) {
    const int j = t / B.ncls, k = t % B.ncls;
    const double e = exp(-b[k] * D0 * (GR_BW + 0.02) * B.bx[j]);
    for (int m = 0; m <= GR_M; ++m) sB[j * nrow + k * GR_ROWS + m] *= e;
  }
  __syncthreads();
  const bool check = threadIdx.x == 32;
  const int n = check ? GR_NC : (int)threadIdx.x;
  if (n >= GR_NC && !check) return;
  double *acc = sC + GR_NHC * nrow + n * (nrow + 1);
  const double xi = check ? cxi : 2.0 * GR_TB / (hi * (B.node[n] + 1.0)), is = 1.0 / sqrt(xi);   // (a = -1 is xi = infinity)
  const double D = check ? cD : D0;
  for (int k = 0; k < nrow; ++k) acc[k] = 0.0;
  for (int i = 0; i < (check ? GR_NHC : GR_NH); ++i) {
    const double x = D + (check ? B.ghcx[i] : B.ghx[i]) * is;
    double jh[GR_ROWS];
    grid_jhat(B.ztab, 2.0 * xi * D * x, jh);
    if (check) {
      for (int c = 0; c < B.ncls; ++c)
        for (int m = 0; m <= GR_LMAX; ++m) {
          const int k = c * GR_ROWS + m;
          acc[k] = fma(B.ghcw[i] * jh[m], sC[i * nrow + k], acc[k]);
        }
      continue;
    }
    double bw[GR_NB], den = 0.0;
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
      const double e = B.ghw[i] * exp(b[c] * (x - D0));
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

__global__ void k_check(Build B) {
  const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  const int cell = (int)(t / B.ncls), c = (int)(t % B.ncls);
  if (cell >= GR_CELLS) return;
  const int nrow = B.ncls * GR_ROWS;
  double lo, hi;
  grid_cellu(cell, &lo, &hi);
  // region B: e^{bx} must vary little enough over a width for the rule's 20 nodes
  const bool flat = cell < GR_NX * GR_NT || fmax(B.bpos, B.bneg) * sqrt(hi / GR_TB) <= 3.0;
  const bool ok = flat && grid_cell_ok(B.xt, cell, B.cells[c] + (size_t)cell * GR_CELL,
                                       B.V + ((size_t)cell * NODES + GR_NC) * nrow + c * GR_ROWS);
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

// Device allocations of a build, freed on every way out.  Uploads go to the
// stream of the build's kernels, which reads them in order (the sources live to
// the build's end).
struct Temp {
  std::vector<void *> p;
  cudaStream_t st;
  explicit Temp(cudaStream_t s) : st(s) {}
  ~Temp() {
    for (void *q : p) cudaFree(q);
  }
  template <class T>
  T *up(const std::vector<T> &v, bool &good) {
    T *d = get<T>(v.size(), good);
    if (good && !v.empty() && cudaMemcpyAsync(d, v.data(), sizeof(T) * v.size(), cudaMemcpyHostToDevice, st) != cudaSuccess)
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
  struct HostQuad {   // the cells' quadrature, the check's
    std::vector<double> x, w, edge;
    std::vector<int> pt0, npanel;
  } hq[2];
  for (int k = 0; k < 2; ++k) {
    hq[k].edge.assign((size_t)NOCT * (GR_MAXPANEL + 1), 0.0);
    for (int o = 0; o < NOCT; ++o) {
      GridQuad q;
      const double lo = std::ldexp(1.0, GR_XLO + o);
      if (!grid_quad(gc, B.ncls, lo, 2.0 * lo, q, k ? GR_CHECK_SCALE : 1.0)) return nullptr;
      hq[k].pt0.push_back((int)hq[k].x.size());
      hq[k].npanel.push_back((int)q.edge.size() - 1);
      hq[k].x.insert(hq[k].x.end(), q.x.begin(), q.x.end());
      hq[k].w.insert(hq[k].w.end(), q.w.begin(), q.w.end());
      std::copy(q.edge.begin(), q.edge.end(), hq[k].edge.begin() + (size_t)o * (GR_MAXPANEL + 1));
    }
    hq[k].pt0.push_back((int)hq[k].x.size());
  }
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
  std::vector<double> node(GR_NC), ghx(GR_NH), ghw(GR_NH), ghcx(GR_NHC), ghcw(GR_NHC), bx(GR_NB), bw(GR_NB), xt((size_t)GR_XT * GR_NX, 0.0);
  grid_nodes(node.data());
  gauss_hermite(GR_NH, ghx.data(), ghw.data());
  gauss_hermite(GR_NHC, ghcx.data(), ghcw.data());
  for (int j = 0; j < GR_NB; ++j) {   // Chebyshev points of the first kind and their barycentric weights
    const double th = M_PI * (j + 0.5) / GR_NB;
    bx[(size_t)j] = std::cos(th);
    bw[(size_t)j] = ((j & 1) ? -1.0 : 1.0) * std::sin(th);
  }
  for (int i = 0; i < GR_NX; ++i) grid_xcell(i, &xt[(size_t)GR_XT * (size_t)i]);

  std::shared_ptr<AuxGrid> g = std::make_shared<AuxGrid>();
  g->device = device;
  g->key = key;
  Temp tmp(st);
  bool good = true;
  for (int k = 0; k < B.ncls && good; ++k) {
    B.cls[k] = ClassDev{tmp.up(gc[k].fam, good), tmp.up(gc[k].coef, good), (int)gc[k].fam.size()};
    const int c = cls_of[k];
    good = good && cudaMalloc((void **)&g->cells[c], sizeof(double) * (size_t)GR_CELLS * GR_CELL) == cudaSuccess &&
           cudaMalloc((void **)&g->ok[c], (size_t)GR_CELLS) == cudaSuccess;
    B.cells[k] = g->cells[c];
    B.ok[k] = g->ok[c];
    g->bytes += sizeof(double) * (size_t)GR_CELLS * GR_CELL + (size_t)GR_CELLS;
  }
  good = good && cudaMalloc((void **)&g->xt, sizeof(double) * xt.size()) == cudaSuccess &&
         cudaMemcpyAsync(g->xt, xt.data(), sizeof(double) * xt.size(), cudaMemcpyHostToDevice, st) == cudaSuccess;
  const int nrow = B.ncls * GR_ROWS;
  Quad Q[2];
  for (int k = 0; k < 2; ++k) {
    const int rows = k ? GR_LMAX + 1 : GR_ROWS;
    Q[k] = Quad{tmp.up(hq[k].x, good), tmp.up(hq[k].w, good),
                tmp.get<double>(hq[k].x.size() * (size_t)(B.ncls * rows), good), (int)hq[k].x.size(), rows,
                tmp.up(hq[k].pt0, good), tmp.up(hq[k].edge, good), tmp.up(hq[k].npanel, good)};
  }
  B.ztab = tmp.up(ztab, good);
  B.node = tmp.up(node, good);
  B.ghx = tmp.up(ghx, good);
  B.ghw = tmp.up(ghw, good);
  B.bx = tmp.up(bx, good);
  B.bw = tmp.up(bw, good);
  B.conv = tmp.up(conv, good);
  B.ghcx = tmp.up(ghcx, good);
  B.ghcw = tmp.up(ghcw, good);
  B.V = tmp.get<double>((size_t)GR_CELLS * NODES * nrow, good);
  B.xt = g->xt;
  B.bpos = bpos;
  B.bneg = bneg;
  if (!good) {
    cudaGetLastError();
    return nullptr;
  }
  for (const Quad &q : Q) k_radial<<<dim3((unsigned)((q.npts + 63) / 64), (unsigned)B.ncls), 64, 0, st>>>(B, q);
  k_rows_a<false><<<dim3(GR_NX, (GR_NT + ITB - 1) / ITB), GR_NC * ITB, 0, st>>>(B, Q[0]);
  k_rows_a<true><<<dim3(GR_NX, (GR_NT + ITC - 1) / ITC), ITC, 0, st>>>(B, Q[1]);
  const size_t smb = sizeof(double) * ((size_t)(GR_NB + GR_NHC) * nrow + (size_t)NODES * (nrow + 1));
  cudaFuncSetAttribute(k_rows_b, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smb);
  k_rows_b<<<GR_NU, TRB, smb, st>>>(B);
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
