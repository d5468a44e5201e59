// auxgrid.cuh -- the auxiliary functions from a grid in (xi, D^2).
//
// For one kernel, hat g_l(xi, D) of aux.cuh is a function of two variables,
// and D_Q = D^-1 d/dD is 2 d/du at fixed xi with u = D^2, so that the orders
// above l are the Taylor coefficients of order l about any point u_c:
//
//   hat g_l(xi, u) = sum_k hat g_{l+k}(xi, u_c) w_k,   w_k = ((u - u_c)/2)^k / k!.
//
// The grid holds, per cell, the rows H_m = sqrt(xi) hat g_m(xi, u_c),
// m = 0..GR_M, as polynomials in a local coordinate of xi: a point costs one
// short polynomial per row l..l+N and N multiply-adds per order, whatever the
// kernel's term families are.  (sqrt(xi) hat g_l is, up to sqrt(pi), the l-th
// derivative of the kernel smoothed by a Gaussian of exponent xi, which stays
// finite as xi grows; the sqrt(p+q) of the prefactor of Eq. bfinal cancels
// against it.)
//
// Two regions:
//   A  xi in [2^GR_XLO, 2^GR_XHI), eight cells per octave (sixteen in the
//      lowest, where a kernel that grows like e^{br} makes the functions grow
//      like e^{b^2/(4 xi)}), c the geometric mean of a cell's ends, local
//      coordinate y(c/xi - 1) scaled to [-1, 1], y(d) = d - d^2/2 + d^3/4 (three
//      terms of 2 (c - xi)/(c + xi), on which the singularities, xi = 0 and the
//      negative axis, lie farthest from the cell); T' = c u < GR_TMAX: cells of width 1/4 below 8, then sixteen
//      per octave;
//   B  T' >= GR_TMAX (distant charge distributions): sixteen cells per octave
//      of u in [2^GR_ULO, 2^GR_UHI), local coordinate 1/xi scaled to [-1, 1].
//
// The rows come from the integral of aux.cuh's header with the families
// summed first,
//   hat g_m = 4 xi (2 xi)^m int_0^inf F_m(x) e^{-xi (x - D)^2} jhat_m(2 xi D x) dx,
// F_m(x) = x^{2m+2} (D_r^m k)(x) summed over the families in double-double
// (their terms cancel near r = 0 and at high order), by composite
// Gauss-Legendre quadrature (A) or Gauss-Hermite about x = D (B), where
// e^{-z} j_m(z) > 0.
//
// Measured on 200,000 I4 quartets of s/p/d shells: 160 ms of evaluation and some
// 10 ms of sorting family by family; from the grid the points cost about 6 ms of
// FP64 pipe inside the kernels that use them.
//
// The header also compiles as plain C++ (tests evaluate single cells on the CPU).
#pragma once

#include <cmath>
#include <cstdint>
#include <cstring>

#ifdef __CUDACC__
#define F12_HD __host__ __device__
#ifndef F12_DEV
#define F12_DEV __device__
#endif
#else
#define F12_HD
#ifndef F12_DEV
#define F12_DEV
#endif
#endif

namespace f12dev {

constexpr int GR_M = 28;                 // highest row: LAUX plus the Taylor terms
constexpr int GR_ROWS = GR_M + 1;
constexpr int GR_NC = 12;                // coefficients per row (degree 11)
constexpr int GR_XLO = -7, GR_XHI = 13;
constexpr int GR_XFINE = 4;              // the lowest octaves of xi have 16 cells, the others 8
constexpr int GR_NX = 8 * (GR_XHI - GR_XLO) + 8 * GR_XFINE;
constexpr int GR_TLIN = 32;              // cells of T' in [0, 8)
constexpr int GR_TEXP = 9;               // GR_TMAX = 2^GR_TEXP
constexpr int GR_NT = GR_TLIN + 16 * (GR_TEXP - 3);
constexpr double GR_TMAX = 512.0;
constexpr int GR_ULO = -4, GR_UHI = 14;
constexpr int GR_NU = 16 * (GR_UHI - GR_ULO);
constexpr int GR_CELLS = GR_NX * GR_NT + GR_NU;
constexpr int GR_CELL = GR_ROWS * GR_NC;  // doubles per cell
constexpr double GR_TB = 480.0;           // region B: xi u >= GR_TB (T' >= GR_TMAX and xi >= 0.94 c)

// Taylor terms for orders up to L: the cell's half width in T' (u in region B)
// is at most 3% of it (1/8 below T' = 8), where the k-th term of order l falls
// like C(l + k, k) 0.03^k for a power of D, and like (|b| D/64)^k/k! for
// e^{bD}: 13 terms hold 3e-13 to |b| D of about 40, and full precision to 25.
F12_HD constexpr int grid_terms(int L) { return L <= 8 ? 13 : 14; }

// Coefficients of row L + k that a point of highest order L reads: the k-th
// Taylor term is smaller by some 0.1^k, and so is what its last coefficients
// add (with 15 - k the errors against the oracle stay those of all 12 over
// molecules' exponents and distances; 13 - k costs an order at L = 8).  Takes 52 of 143
// multiply-adds off the rows past L.  Kernels that grow or decay too fast for it are
// found by the cells' check, which evaluates these forms.
F12_HD constexpr int grid_coefs(int L, int k) {
  return k <= 3 || L > 8 ? GR_NC : (k >= 11 ? 4 : 15 - k);
}

// multiply-adds of one point
F12_HD constexpr int grid_fmas(int L) {
  int n = (L + 1) * (GR_NC - 1) + (L + 1) * (grid_terms(L) + 1);
  for (int k = 1; k <= grid_terms(L); ++k) n += grid_coefs(L, k) - 1;
  return n;
}

F12_HD inline int grid_hi(double x) {
#ifdef __CUDA_ARCH__
  return __double2hiint(x);
#else
  long long b;
  std::memcpy(&b, &x, sizeof b);
  return (int)(b >> 32);
#endif
}

F12_HD inline double hi_double(int hi) {
#ifdef __CUDA_ARCH__
  return __hiloint2double(hi, 0);
#else
  long long b = (long long)hi << 32;
  double d;
  std::memcpy(&d, &b, sizeof d);
  return d;
#endif
}

// product rounded on its own (the builder's u_c is that product)
F12_HD inline double mul_rn(double a, double b) {
#ifdef __CUDA_ARCH__
  return __dmul_rn(a, b);
#else
  volatile double p = a * b;
  return p;
#endif
}

// Cell of xi, or -1, from the high word of the double.
F12_HD inline int grid_xindex(int h) {
  if (h < (1023 + GR_XLO) << 20 || h >= (1023 + GR_XHI) << 20) return -1;
  return h < (1023 + GR_XLO + GR_XFINE) << 20 ? (h >> 16) - (1023 + GR_XLO) * 16
                                             : (h >> 17) - (1023 + GR_XLO - GR_XFINE) * 8;
}

// A cell and the local coordinates of a point.
struct GridPoint {
  int cell;       // -1: outside the grid
  double a;       // local coordinate of xi in [-1, 1]
  double hd;      // (u - u_c)/2
};

// GR_XT values per cell of xi in the table that grid_point reads: c, 1/c and the
// scale of y
constexpr int GR_XT = 4;
F12_HD inline double grid_y(double d) { return fma(fma(d, 0.25, -0.5) * d, d, d); }
F12_HD inline void grid_xends(int ix, double *lo, double *hi) {
  if (ix < 16 * GR_XFINE) {
    *lo = hi_double(((1023 + GR_XLO) * 16 + ix) << 16);
    *hi = hi_double(((1023 + GR_XLO) * 16 + ix + 1) << 16);
  } else {
    *lo = hi_double(((1023 + GR_XLO - GR_XFINE) * 8 + ix) << 17);
    *hi = hi_double(((1023 + GR_XLO - GR_XFINE) * 8 + ix + 1) << 17);
  }
}
F12_HD inline void grid_xcell(int ix, double *r) {
  double lo, hi;
  grid_xends(ix, &lo, &hi);
  r[0] = sqrt(lo * hi);
  r[1] = 1.0 / r[0];
  r[2] = 1.0 / fmax(fabs(grid_y(r[0] / lo - 1.0)), fabs(grid_y(r[0] / hi - 1.0)));
  r[3] = 0.0;
}
// xi at local coordinate a of a cell (r: its GR_XT values), by Newton's method
F12_HD inline double grid_xi(const double *r, double a) {
  const double y = a / r[2];
  double d = y / (1.0 - 0.5 * y);
  for (int i = 0; i < 4; ++i) d -= (grid_y(d) - y) / (1.0 - d + 0.75 * d * d);
  return r[0] / (1.0 + d);
}
F12_HD inline int grid_octave(int ix) { return ix < 16 * GR_XFINE ? ix >> 4 : (ix >> 3) - GR_XFINE; }
// ends of a cell of T' (or of u: the same subdivision of an octave)
F12_HD inline void grid_tcell(int it, double *lo, double *hi) {
  if (it < GR_TLIN) {
    *lo = 0.25 * it;
    *hi = 0.25 * (it + 1);
  } else {
    *lo = hi_double(((1023 + 3) * 16 + it - GR_TLIN) << 16);
    *hi = hi_double(((1023 + 3) * 16 + it - GR_TLIN + 1) << 16);
  }
}
F12_HD inline void grid_ucell(int iu, double *lo, double *hi) {
  *lo = hi_double(((1023 + GR_ULO) * 16 + iu) << 16);
  *hi = hi_double(((1023 + GR_ULO) * 16 + iu + 1) << 16);
}

// Local coordinates of (xi, u) with v = 1/xi; xt: GR_XT values per cell of xi.
// The cell of xi comes from a single-precision reciprocal (a cell's polynomials
// hold a little past its ends), the cell and its middle of T' from the bits of
// the double, so that a point costs no FP64 division.
F12_DEV inline GridPoint grid_point(const double *xt, double v, double u) {
  GridPoint g;
  const float xf = 1.0f / (float)v;
  int b;
#ifdef __CUDA_ARCH__
  b = __float_as_int(xf);
#else
  std::memcpy(&b, &xf, sizeof b);
#endif
  const int ix = grid_xindex((b >> 3) + ((1023 - 127) << 20));   // the bits as those of a double's high word
  if (ix < 0) {
    g.cell = -1;
    return g;
  }
  const double *r = xt + GR_XT * ix;
  const double T = r[0] * u;
  const int hT = grid_hi(T);
  if (hT < (1023 + GR_TEXP) << 20) {   // T < GR_TMAX
    double mid;
    int it;
    if (hT < (1023 + 3) << 20) {       // T < 8: the cells of [8, 16) in T + 8
      const int h8 = grid_hi(T + 8.0);
      it = (h8 >> 15) - (1023 + 3) * 32;
      mid = hi_double((h8 & ~0x7FFF) | 0x4000) - 8.0;
    } else {
      it = GR_TLIN + (hT >> 16) - (1023 + 3) * 16;
      mid = hi_double((hT & ~0xFFFF) | 0x8000);
    }
    g.cell = ix * GR_NT + it;
    g.a = grid_y(fma(r[0], v, -1.0)) * r[2];
    g.hd = 0.5 * (u - mul_rn(mid, r[1]));
  } else {
    const int iu = (grid_hi(u) >> 16) - (1023 + GR_ULO) * 16;
    if (iu < 0 || iu >= GR_NU) {
      g.cell = -1;
      return g;
    }
    double lo, hi;
    grid_ucell(iu, &lo, &hi);
    g.cell = GR_NX * GR_NT + iu;
    g.a = 2.0 * GR_TB / hi * v - 1.0;
    g.hd = 0.5 * (u - 0.5 * (lo + hi));
  }
  return g;
}

// ---------------------------------------------------------- double-double --
// (two-sum and two-product of Knuth and Dekker, the latter with a fused multiply-add)
struct dd {
  double h, l;
};
F12_HD inline dd dd_fast(double a, double b) {   // |a| >= |b|
  const double s = a + b;
  return dd{s, b - (s - a)};
}
F12_HD inline dd dd_sum(double a, double b) {
  const double s = a + b, t = s - a;
  return dd{s, (a - (s - t)) + (b - t)};
}
F12_HD inline dd dd_prod(double a, double b) {
  const double p = a * b;
  return dd{p, fma(a, b, -p)};
}
F12_HD inline dd dd_add(dd a, dd b) {
  const dd s = dd_sum(a.h, b.h), t = dd_sum(a.l, b.l);
  const dd v = dd_fast(s.h, s.l + t.h);
  return dd_fast(v.h, v.l + t.l);
}
F12_HD inline dd dd_mul(dd a, dd b) {
  const dd p = dd_prod(a.h, b.h);
  return dd_fast(p.h, p.l + (a.h * b.l + a.l * b.h));
}
F12_HD inline dd dd_muld(dd a, double b) {
  const dd p = dd_prod(a.h, b);
  return dd_fast(p.h, fma(a.l, b, p.l));
}
// e^y: y = k ln 2 + 64 r, Taylor series of e^r (|r| <= ln2/128), six squarings
F12_DEV inline dd dd_exp(dd y) {
  if (y.h < -700.0) return dd{0.0, 0.0};
  const double k = rint(y.h * 1.4426950408889634);
  // ln 2 in three parts (the first with 21 trailing zero bits, so that k times it is exact)
  const double L1 = 0.6931471803691238, L2 = 1.9082149292705877e-10, L3 = 1.1612227229362532e-26;
  dd r = dd_add(y, dd{-k * L1, 0.0});
  r = dd_add(r, dd_prod(-k, L2));
  r = dd_add(r, dd{-k * L3, 0.0});
  r.h *= 0.015625;
  r.l *= 0.015625;
  dd s{0.0, 0.0};   // e^r - 1 by Horner's rule
  for (int n = 11; n >= 1; --n) {
    // s = r/n (1 + s)
    dd t = dd_add(dd{1.0, 0.0}, s);
    t = dd_mul(t, r);
    const double q = t.h / n;
    const double e = fma(-q, (double)n, t.h) + t.l;
    s = dd_fast(q, e / n);
  }
  for (int i = 0; i < 6; ++i) {   // (1 + s)^2 - 1 = 2 s + s^2
    const dd q = dd_mul(s, s);
    s = dd_add(dd{2.0 * s.h, 2.0 * s.l}, q);
  }
  s = dd_add(dd{1.0, 0.0}, s);
  const double f = hi_double((1023 + (int)k) << 20);
  return dd{s.h * f, s.l * f};
}

// --------------------------------------------------------------- builder --
// A term family of the kernel for the grid: F_m's part is
//   x^alpha0 e^{bx - gx^2} sum_j P_mj x^j,  alpha0 = ai + fr.
struct GridFam {
  double b, g, fr;
  int ai;                  // integer part of alpha0
  int lat;                 // index of the power lattice (families of one fr are summed in double-double)
  int deg0;                // length of P_0; P_m has deg0 + 2m coefficients
  int coff;                // offset of P_0 in the double-double coefficient pool; P_m follows P_{m-1}
};
constexpr int GR_MAXLAT = 4;

// F_m(x), m = 0..M.
F12_DEV inline void grid_radial(const GridFam *fam, int nf, const dd *coef, double x, int M, double *F) {
  for (int m = 0; m <= M; ++m) F[m] = 0.0;
  for (int lat = 0; lat < GR_MAXLAT; ++lat) {
    dd acc[GR_ROWS];
    bool any = false;
    double fr = 0.0;
    for (int m = 0; m <= M; ++m) acc[m] = dd{0.0, 0.0};
    for (int f = 0; f < nf; ++f) {
      const GridFam &A = fam[f];
      if (A.lat != lat) continue;
      any = true;
      fr = A.fr;
      const dd arg = dd_add(dd_prod(A.b, x), dd_muld(dd_prod(x, x), -A.g));
      dd e = dd_exp(arg);
      if (e.h == 0.0) continue;
      if (A.ai >= 0) {
        for (int i = 0; i < A.ai; ++i) e = dd_muld(e, x);
      } else {
        for (int i = 0; i < -A.ai; ++i) {   // e / x
          const double q = e.h / x;
          const double r = fma(-q, x, e.h) + e.l;
          e = dd_fast(q, r / x);
        }
      }
      const dd *P = coef + A.coff;
      for (int m = 0; m <= M; ++m) {
        const int n = A.deg0 + 2 * m;
        dd h{0.0, 0.0};
        for (int j = n - 1; j >= 0; --j) {
          h = dd_muld(h, x);
          if (P[j].h != 0.0) h = dd_add(h, P[j]);
        }
        acc[m] = dd_add(acc[m], dd_mul(h, e));
        P += n;
      }
    }
    if (!any) continue;
    const double xf = fr == 0.0 ? 1.0 : (fr == 0.5 ? sqrt(x) : pow(x, fr));
    for (int m = 0; m <= M; ++m) F[m] += xf * acc[m].h;
  }
}

// e^{-z} j_m(z), m = 0..GR_M.  From z = GR_ZMAX by the upward recurrence (its
// loss grows with GR_M^2/(2z)); below, downward recurrence j_{m-1} =
// z^2 j_{m+1} + (2m+1) j_m (every term positive) from the ratio
// j_{GR_M}/j_{GR_M-1}, normalised by e^{-z} j_0 = (1 - e^{-2z})/(2z).  The
// ratio comes from a table in z (cells as those of T', GR_NC coefficients).
constexpr int GR_ZEXP = 12;
constexpr double GR_ZMAX = 4096.0;
constexpr int GR_NZ = GR_TLIN + 16 * (GR_ZEXP - 3);
F12_DEV inline void grid_jhat(const double *ztab, double z, double *jh) {
  if (z >= GR_ZMAX) {
    const double r = 1.0 / z;
    jh[0] = 0.5 * r;
    jh[1] = 0.5 * (1.0 - r) * r * r;
    for (int m = 1; m < GR_M; ++m) jh[m + 1] = (jh[m - 1] - (2 * m + 1) * jh[m]) * r * r;
    return;
  }
  const int iz = z < 8.0 ? (int)(4.0 * z) : GR_TLIN + (grid_hi(z) >> 16) - (1023 + 3) * 16;
  double lo, hi;
  grid_tcell(iz, &lo, &hi);
  const double a = (2.0 * z - (lo + hi)) / (hi - lo);
  const double *c = ztab + iz * GR_NC;
  double q = c[GR_NC - 1];
  for (int i = GR_NC - 2; i >= 0; --i) q = fma(q, a, c[i]);
  const double z2 = z * z;
  // (unnormalised values reach about z^GR_M, within range)
  double up = q, cur = 1.0;
  jh[GR_M] = q;
  jh[GR_M - 1] = 1.0;
  for (int m = GR_M - 1; m >= 1; --m) {
    const double dn = fma(z2, up, (2 * m + 1) * cur);
    up = cur;
    cur = dn;
    jh[m - 1] = dn;
  }
  const double j0 = z > 0.0 ? -0.5 * expm1(-2.0 * z) / z : 1.0;
  const double f = j0 / cur;
  for (int m = 0; m <= GR_M; ++m) jh[m] *= f;
}

// Region B: quadrature nodes, and the Chebyshev points of x/D in
// [1 - GR_BW, 1 + GR_BW] from which F_m is interpolated (barycentric form); the
// rule's outermost node lies within 5.4 widths, a width is at most
// D/sqrt(GR_TB).  The check point's rule has more nodes and takes F_m itself.
constexpr int GR_NH = 20;
constexpr int GR_NHC = 32;
constexpr int GR_NB = 36;
constexpr double GR_BW = 0.25;

// Exponent b of a kernel's lowest rows over the interpolated range (F at its two
// ends, dx apart): F_m e^{-b(x - D)} is interpolated, which varies little whatever
// mixture of decays the kernel has (with one of its families' b instead, a
// kernel like e^{-8x} beside Gaussians lost seven digits).
F12_HD inline double grid_slope(const double *lo, const double *hi, double dx) {
  double a = 0.0, b = 0.0;
  for (int m = 0; m < 3; ++m) {
    const double l = fabs(lo[m]), h = fabs(hi[m]), s = l + h;
    if (s > 0.0) {
      a += l / s;
      b += h / s;
    }
  }
  return a > 0.0 && b > 0.0 ? log(b / a) / dx : 0.0;
}

// ---------------------------------------------------------- check points --
// Every cell is checked at one point: of region A one of its four corners, of
// region B an end of its u at its widest Gaussian (where the rule is at its
// least; a = 1 itself is left a margin).  a: the coordinate of xi, s: of u in
// units of the cell's width, from its middle.
F12_HD inline void grid_check(int cell, double *a, double *s) {
  *a = cell >= GR_NX * GR_NT ? 0.97 : (cell & 1) ? 1.0 : -1.0;
  *s = (cell & 2) ? 0.5 : -0.5;
}
// ends of a cell in T' (region A) or u (B)
F12_HD inline void grid_cellu(int cell, double *lo, double *hi) {
  if (cell < GR_NX * GR_NT) grid_tcell(cell % GR_NT, lo, hi);
  else grid_ucell(cell - GR_NX * GR_NT, lo, hi);
}
// the point itself: its xi and u
F12_HD inline void grid_check_point(const double *xt, int cell, double *xi, double *u) {
  double lo, hi, a, s;
  grid_cellu(cell, &lo, &hi);
  grid_check(cell, &a, &s);
  if (cell < GR_NX * GR_NT) {
    const double *r = xt + GR_XT * (cell / GR_NT);
    *xi = grid_xi(r, a);
    *u = mul_rn(0.5 * (lo + hi), r[1]) + s * (hi - lo) * r[1];
  } else {
    *xi = 2.0 * GR_TB / (hi * (a + 1.0));
    *u = 0.5 * (lo + hi) + s * (hi - lo);
  }
}

// ------------------------------------------------------------ evaluation --
// The Coulomb kernel (I1): sqrt(xi) hat g_l = 2 sqrt(xi) (-2 xi)^l F_l(x), F_l the
// Boys function and x = xi u, xi = 1/v.  tab is the table of e^{-x} M(1, l + 3/2, x) =
// (2l + 1) F_l(x) (aux.cuh: Taylor rows on a grid of x), read for the highest
// order; the others follow by F_{l-1} = (2 x F_l + e^{-x})/(2l - 1), every term
// positive.  Past the table e^{-x} is below double precision of F_l.
constexpr int BY_LSTRIDE = 40 * 201 * 14, BY_NT = 14;   // between orders, per row
constexpr double BY_XMAX = 100.0;
template <int LMAX, bool FIXED>
F12_DEV inline void boys_eval(const double *tab, double v, double u, int L_, double *h) {
  const int L = FIXED ? LMAX : L_;
  const double xi = 1.0 / v, x = xi * u;
  if (x < BY_XMAX) {
    const double r = rint(2.0 * x), d = x - 0.5 * r;
    const double *row = tab + (size_t)L * BY_LSTRIDE + (int)r * BY_NT;
    double t = row[BY_NT - 1];
#pragma unroll
    for (int m = BY_NT - 2; m >= 0; --m) t = fma(t, d, row[m]);
    t *= 1.0 / (2 * L + 1);
    const double e = exp(-x), x2 = 2.0 * x;
#pragma unroll
    for (int l = LMAX; l >= 0; --l) {
      if (!FIXED && l > L) continue;
      h[l] = t;
      if (l > 0) t = fma(x2, t, e) * (1.0 / (2 * l - 1));
    }
  } else {
    const double ix2 = 0.5 / x;
    double t = 0.88622692545275801365 * sqrt(2.0 * ix2);   // sqrt(pi/x)/2
#pragma unroll
    for (int l = 0; l <= LMAX; ++l) {
      if (!FIXED && l > L) continue;
      h[l] = t;
      t *= (2 * l + 1) * ix2;
    }
  }
  double f = 2.0 * sqrt(xi);
#pragma unroll
  for (int l = 0; l <= LMAX; ++l) {
    if (!FIXED && l > L) continue;
    h[l] *= f;
    f *= -2.0 * xi;
  }
}

// Row coefficients of a cell, four at a time (32-byte loads: whole sectors).
F12_DEV inline void grid_load4(const double *p, double *c) {
#ifdef __CUDA_ARCH__
  asm("ld.global.nc.v4.f64 {%0, %1, %2, %3}, [%4];" : "=d"(c[0]), "=d"(c[1]), "=d"(c[2]), "=d"(c[3]) : "l"(p));
#else
  for (int i = 0; i < 4; ++i) c[i] = p[i];
#endif
}

// sqrt(xi) hat g_l for l = 0..L into h[] (L <= LMAX, a compile-time bound of
// the registers; FIXED: L == LMAX).
template <int LMAX, bool FIXED>
F12_DEV inline void grid_eval(const double *cells, const GridPoint &pt, int L, double *h) {
  constexpr int NMAX = grid_terms(LMAX);
  const int N = FIXED ? NMAX : grid_terms(L);
  const double *cell = cells + (size_t)(pt.cell < 0 ? 0 : pt.cell) * GR_CELL;
  // rows, highest first, into the orders' Horner sums
  //   h_l = H_l + t_1 (H_{l+1} + t_2 (H_{l+2} + ..)),  t_k = hd/k
  double t[NMAX + 1];
#pragma unroll
  for (int k = 1; k <= NMAX; ++k) t[k] = pt.hd * (1.0 / k);
#pragma unroll
  for (int l = 0; l <= LMAX; ++l) h[l] = 0.0;
#pragma unroll
  for (int m = LMAX + NMAX; m >= 0; --m) {
    if (!FIXED && m > L + N) continue;
    const double *row = cell + m * GR_NC;
    const int nc = FIXED && m > LMAX ? grid_coefs(LMAX, m - LMAX) : GR_NC;
    double c[GR_NC];
    grid_load4(row, c);
    if (nc > 4) grid_load4(row + 4, c + 4);
    if (nc > 8) grid_load4(row + 8, c + 8);
    double r = 0.0;
#pragma unroll
    for (int i = GR_NC - 1; i >= 0; --i)
      if (i < nc) r = i == nc - 1 ? c[i] : fma(r, pt.a, c[i]);
#pragma unroll
    for (int l = 0; l <= LMAX; ++l) {
      const int k = m - l;   // the row's term of order l
      if (k < 0 || k > NMAX || (!FIXED && (l > L || k > N))) continue;
      h[l] = k == (FIXED ? NMAX : N) ? r : fma(h[l], t[k + 1 <= NMAX ? k + 1 : NMAX], r);
    }
  }
}

// ------------------------------------------------------------ acceptance --
// A cell is in order when every form in which the kernels take it (highest
// orders 0 to 8, each with its shortened rows, and 14, whose rows those of 9 to 13
// are) agrees at its check point with rows V[0..LMAX] from a quadrature of its
// own, to GR_TOL of the sum of the terms' magnitudes (the scale of the result
// where it passes through zero).  Blocks are to hold 1e-10.  Orders past 8 read
// rows to the 28th, which vary like that power of xi and fit their 12 coefficients to
// 1e-9 only: at xi = 0.1..0.6 and small D orders 13 and 14 are within 5e-12,
// 4e-11 where they pass through zero.
constexpr double GR_TOL = 1e-12, GR_TOL_HIGH = 5e-11;
constexpr int GR_LMAX = 14;
template <int L>
F12_DEV inline bool grid_form_ok(const double *cell, const GridPoint &pt, const double *V, const double *sc) {
  double h[L + 1];
  grid_eval<L, true>(cell, pt, L, h);
  bool ok = true;
  for (int l = 0; l <= L; ++l)
    ok = ok && fabs(h[l] - V[l]) <= (L > 8 ? GR_TOL_HIGH : GR_TOL) * sc[l];   // false for NaN
  return ok;
}
F12_DEV inline bool grid_cell_ok(const double *xt, int cell, const double *C, const double *V) {
  double lo, hi, a, s;
  grid_cellu(cell, &lo, &hi);
  grid_check(cell, &a, &s);
  GridPoint pt;
  pt.cell = 0;
  pt.a = a;
  pt.hd = 0.5 * s * (hi - lo) * (cell < GR_NX * GR_NT ? xt[GR_XT * (cell / GR_NT) + 1] : 1.0);
  constexpr int N = grid_terms(GR_LMAX);
  double row[GR_LMAX + N + 1], sc[GR_LMAX + 1];
  for (int m = 0; m <= GR_LMAX + N; ++m) {
    double r = C[m * GR_NC + GR_NC - 1];
    for (int i = GR_NC - 2; i >= 0; --i) r = fma(r, a, C[m * GR_NC + i]);
    row[m] = fabs(r);
  }
  for (int l = 0; l <= GR_LMAX; ++l) {
    double w = 1.0;
    sc[l] = 0.0;
    for (int k = 0; k <= N; ++k) {
      sc[l] = fma(row[l + k], w, sc[l]);
      w *= fabs(pt.hd) / (k + 1);
    }
  }
  return grid_form_ok<0>(C, pt, V, sc) && grid_form_ok<1>(C, pt, V, sc) && grid_form_ok<2>(C, pt, V, sc) &&
         grid_form_ok<3>(C, pt, V, sc) && grid_form_ok<4>(C, pt, V, sc) && grid_form_ok<5>(C, pt, V, sc) &&
         grid_form_ok<6>(C, pt, V, sc) && grid_form_ok<7>(C, pt, V, sc) && grid_form_ok<8>(C, pt, V, sc) &&
         grid_form_ok<14>(C, pt, V, sc);
}

}  // namespace f12dev
