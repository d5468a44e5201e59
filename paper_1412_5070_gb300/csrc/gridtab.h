// gridtab.h -- host-side data of the auxiliary grid (auxgrid.cuh): the term
// families of a kernel with their radial derivatives in double-double, and
// the quadrature points of the grid's rows.
#pragma once

#include <cmath>
#include <vector>

#include "auxgrid.cuh"
#include "auxtab.h"
#include "termlist.h"

namespace f12dev {

struct GridClass {
  std::vector<GridFam> fam;
  std::vector<dd> coef;
  std::vector<double> g, reach;        // the families' g > 0, and how far they count
  double bpos = 0.0, bneg = 0.0;       // largest b > 0, largest |b| of b < 0
};

// Distance past which a family x^alpha e^{bx - gx^2}, alpha <= amax, is below
// double precision of its largest value: t^p e^{-t}, t = g x^2 and p = amax/2, has
// fallen by 2^-58 from its peak at t = p, and e^{bx} moves the peak by b/2g.
inline double grid_reach(double amax, double b, double g) {
  const double p = std::max(0.5 * amax, 1.0);
  double t = p;
  while (p * std::log(t / p) - (t - p) > -40.0) t += 1.0;
  return std::sqrt(t / g) + 0.5 * std::max(b, 0.0) / g;
}

// The families of a kernel, or false when the grid does not serve it: lowest
// powers below -1 (singular groups), a general power so low that the first
// panel's rule would not resolve it, more power lattices than grid_radial
// sums, or a kernel whose every family decays as a Gaussian (it falls by many
// orders of magnitude within one cell).
inline bool grid_families(const f12::TermList &kernel, GridClass &gc) {
  gc = GridClass{};
  std::vector<double> lat;
  bool reach = false;
  for (const f12::Family &f : f12::families(kernel)) {
    GridFam d{};
    const double a = f.a0 + 2.0;
    if (a < -1.0 - 1e-9) return false;
    d.b = f.b;
    d.g = f.g;
    const double fl = std::floor(a + 1e-9);
    d.ai = (int)fl;
    d.fr = std::fabs(a - fl) < 1e-9 ? 0.0 : a - fl;
    const double eighth = 8.0 * a;
    if (a < -0.3 && std::fabs(eighth - std::round(eighth)) > 1e-9) return false;
    d.lat = -1;
    for (size_t i = 0; i < lat.size(); ++i)
      if (std::fabs(lat[i] - d.fr) < 1e-9) d.lat = (int)i;
    if (d.lat < 0) {
      d.lat = (int)lat.size();
      lat.push_back(d.fr);
      if (d.lat >= GR_MAXLAT) return false;
    }
    d.fr = lat[(size_t)d.lat];
    d.deg0 = (int)f.poly.size();
    d.coff = (int)gc.coef.size();
    std::vector<dd> cur;
    for (double c : f.poly) cur.push_back(dd{c, 0.0});
    for (int m = 0; m <= GR_M; ++m) {
      gc.coef.insert(gc.coef.end(), cur.begin(), cur.end());
      // D_r: c x^p e^{bx-gx^2} -> c (p x^{p-2} + b x^{p-1} - 2 g x^p) e^{bx-gx^2}
      std::vector<dd> nxt(cur.size() + 2, dd{0.0, 0.0});
      for (size_t j = 0; j < cur.size(); ++j) {
        const dd p = dd_sum(f.a0, (double)j - 2.0 * m);
        nxt[j] = dd_add(nxt[j], dd_mul(cur[j], p));
        nxt[j + 1] = dd_add(nxt[j + 1], dd_muld(cur[j], f.b));
        nxt[j + 2] = dd_add(nxt[j + 2], dd_muld(cur[j], -2.0 * f.g));
      }
      cur.swap(nxt);
    }
    if (f.g > 0.0) {
      gc.g.push_back(f.g);
      gc.reach.push_back(grid_reach(a + (double)f.poly.size() - 1.0 + 2.0 * GR_M, f.b, f.g));
    }
    gc.bpos = std::max(gc.bpos, f.b);
    gc.bneg = std::max(gc.bneg, -f.b);
    reach = reach || f.g == 0.0;
    gc.fam.push_back(d);
  }
  return reach && !gc.fam.empty();
}

constexpr int GR_NQ = 16;        // Gauss-Legendre nodes per panel
constexpr int GR_NQ0 = 64;       // nodes of the first panel, in x = w u^8
constexpr int GR_MAXPANEL = 512;   // (of the check: a quarter more than the cells take)

// Quadrature points of one octave of xi (all of its cells use them): panels
// of 1.25 widths of the Gaussian -- of the narrowest family's times the
// Gaussian among those that still count -- to the largest D of region A plus 6.6
// widths; 1.25 widths are about the distance over which 16 nodes reach
// double precision.  The first panel is taken in u = (x/w)^{1/8}, which makes
// x^{alpha} du smooth for the powers grid_families admits; the others are at
// most 1.5 times as wide as their distance from r = 0, where the long-range
// families have a branch point: where narrow panels end (a tight Gaussian's
// reach) one of full width would not resolve it.  scale < 1: every panel that
// much narrower (0.8: a thousandth of the error or less), for the cells' check.
struct GridQuad {
  std::vector<double> x, w;
  std::vector<double> edge;   // panel p covers [edge[p], edge[p + 1]]
};
// Gauss-Legendre nodes and weights as double-doubles (long double inside), and for a
// rule of n nodes what rounding its nodes takes: with nodes t + d, exact again up
// to degree n - 1 are the weights w + c d (the changes of the moments of P_k, k < n,
// by the rule's own discrete orthogonality).  Without it the rounding of
// x, up to x sqrt(xi) u of a width, put several u into the rows.
struct GridRule {
  std::vector<dd> t, w;
  std::vector<double> c;   // [n][n]
};
inline GridRule grid_rule(int n, bool corrected) {
  GridRule r;
  std::vector<double> P((size_t)n * n), Q((size_t)n * n);   // P_k(t_i) (2k + 1)/2, P_k'(t_i)
  for (int i = 0; i < n; ++i) {
    long double t = -std::cos(M_PI * (i + 0.75) / (n + 0.5)), dp = 1.0L;
    for (int it = 0; it < 8; ++it) {
      long double p0 = 1.0L, p1 = t;
      for (int k = 2; k <= n; ++k) {
        const long double p2 = ((2 * k - 1) * t * p1 - (k - 1) * p0) / k;
        p0 = p1;
        p1 = p2;
      }
      dp = n * (t * p1 - p0) / (t * t - 1.0L);
      if (it < 7) t -= p1 / dp;
    }
    const long double w = 2.0L / ((1.0L - t * t) * dp * dp);
    r.t.push_back(dd{(double)t, (double)(t - (double)t)});
    r.w.push_back(dd{(double)w, (double)(w - (double)w)});
    double p0 = 1.0, p1 = (double)t, d0 = 0.0, d1 = 1.0;
    for (int k = 0; k < n; ++k) {
      P[(size_t)i * n + k] = (k + 0.5) * p0;
      Q[(size_t)i * n + k] = d0;
      const double p2 = ((2 * k + 3) * (double)t * p1 - (k + 1) * p0) / (k + 2), d2 = d0 + (2 * k + 3) * p1;
      p0 = p1;
      p1 = p2;
      d0 = d1;
      d1 = d2;
    }
  }
  if (!corrected) return r;
  r.c.assign((size_t)n * n, 0.0);
  for (int i = 0; i < n; ++i)
    for (int j = 0; j < n; ++j) {
      double s = 0.0;
      for (int k = 0; k < n; ++k) s += P[(size_t)i * n + k] * Q[(size_t)j * n + k];
      r.c[(size_t)i * n + j] = -r.w[i].h * r.w[j].h * s;
    }
  return r;
}
constexpr double GR_CHECK_SCALE = 0.8;
inline bool grid_quad(const GridClass *gc, int ngc, double xi_lo, double xi_hi, GridQuad &q,
                      double scale = 1.0) {
  q = GridQuad{};
  static const GridRule rule = grid_rule(GR_NQ, true), rule0 = grid_rule(GR_NQ0, false);
  double bpos = 0.0, bneg = 0.0;
  for (int c = 0; c < ngc; ++c) {
    bpos = std::max(bpos, gc[c].bpos);
    bneg = std::max(bneg, gc[c].bneg);
  }
  const double end = std::sqrt((GR_TMAX + 32.0) / xi_lo) + (8.5 + 0.5 * bpos / std::sqrt(xi_lo)) / std::sqrt(xi_lo);
  double a = 0.0;
  q.edge.push_back(0.0);
  while (a < end) {
    double w = 1.25 / std::sqrt(xi_hi);
    for (int c = 0; c < ngc; ++c)
      for (size_t i = 0; i < gc[c].g.size(); ++i)
        if (a < gc[c].reach[i]) w = std::min(w, 1.25 / std::sqrt(xi_hi + gc[c].g[i]));
    if (bneg > 0.0) w = std::min(w, 1.25 * std::sqrt(std::max(1.0, bneg * a)) / bneg);
    if (a > 0.0) w = std::min(w, 1.5 * a);
    w *= scale;
    if (a == 0.0) {
      w *= 0.5;
      for (int i = 0; i < GR_NQ0; ++i) {
        const double u = 0.5 * (rule0.t[i].h + 1.0) + 0.5 * rule0.t[i].l, u2 = u * u, u4 = u2 * u2;
        q.x.push_back(w * u4 * u4);
        q.w.push_back(0.5 * rule0.w[i].h * w * 8.0 * u4 * u2 * u);
      }
      a = w;
    } else {
      const double e = a + w;
      dd h = dd_sum(e, -a);
      h = dd{0.5 * h.h, 0.5 * h.l};
      double d[GR_NQ];
      for (int i = 0; i < GR_NQ; ++i) {
        const dd x = dd_add(dd{a, 0.0}, dd_mul(h, dd_add(dd{1.0, 0.0}, rule.t[i])));
        q.x.push_back(x.h);
        d[i] = -x.l / h.h;
      }
      for (int i = 0; i < GR_NQ; ++i) {
        double c = rule.w[i].l;
        for (int j = 0; j < GR_NQ; ++j) c += rule.c[(size_t)i * GR_NQ + j] * d[j];
        const dd wi = dd_mul(h, dd_fast(rule.w[i].h, c));
        q.w.push_back(wi.h);
      }
      a = e;
    }
    q.edge.push_back(a);
    if (q.edge.size() > GR_MAXPANEL) return false;
  }
  return true;
}

// Monomial coefficients of the polynomial through values at the GR_NC
// Chebyshev points a_n = cos(pi (n + 1/2)/GR_NC): coefficient i is
// sum_n conv[i][n] v_n (long double, split in two doubles).
inline void grid_nodes(double *a) {
  for (int n = 0; n < GR_NC; ++n) a[n] = std::cos(M_PI * (n + 0.5) / GR_NC);
}
inline void grid_conversion(dd conv[GR_NC][GR_NC]) {
  // the Lagrange basis polynomials of the rounded nodes, expanded in double-double
  double a[GR_NC];
  grid_nodes(a);
  for (int n = 0; n < GR_NC; ++n) {
    std::vector<dd> p{dd{1.0, 0.0}};
    dd den{1.0, 0.0};
    for (int k = 0; k < GR_NC; ++k) {
      if (k == n) continue;
      p.push_back(dd{0.0, 0.0});
      for (size_t i = p.size(); i-- > 0;)
        p[i] = dd_add(i > 0 ? p[i - 1] : dd{0.0, 0.0}, dd_muld(p[i], -a[k]));
      den = dd_mul(den, dd_sum(a[n], -a[k]));
    }
    for (int i = 0; i < GR_NC; ++i) {
      // p_i / den
      const double q1 = p[i].h / den.h;
      const dd r = dd_add(p[i], dd_muld(den, -q1));
      conv[i][n] = dd_fast(q1, r.h / den.h);
    }
  }
}

// The table of grid_jhat: j_{GR_M}/j_{GR_M-1} = rho_{GR_M} with
// rho_m = 1/(z^2 rho_{m+1} + 2m + 1), from an order where rho is below double
// precision of its effect (the recursion damps errors).
inline void grid_ztab(std::vector<double> &tab) {
  dd conv[GR_NC][GR_NC];
  grid_conversion(conv);
  double nd[GR_NC];
  grid_nodes(nd);
  tab.assign((size_t)GR_NZ * GR_NC, 0.0);
  for (int iz = 0; iz < GR_NZ; ++iz) {
    double lo, hi, v[GR_NC];
    grid_tcell(iz, &lo, &hi);
    for (int n = 0; n < GR_NC; ++n) {
      const double z = 0.5 * (lo + hi) + 0.5 * (hi - lo) * nd[n], z2 = z * z;
      double r = 0.0;
      for (int m = (int)std::sqrt((double)GR_M * GR_M + 80.0 * z) + 12; m >= GR_M; --m)
        r = 1.0 / (z2 * r + 2.0 * m + 1.0);
      v[n] = r;
    }
    for (int i = 0; i < GR_NC; ++i) {
      dd s{0.0, 0.0};
      for (int n = 0; n < GR_NC; ++n) s = dd_add(s, dd_muld(conv[i][n], v[n]));
      tab[(size_t)iz * GR_NC + i] = s.h;
    }
  }
}

}  // namespace f12dev
