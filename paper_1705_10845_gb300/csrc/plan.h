// Host-side plan of the inverses Y_k = (I + T_k^2)^-1 of the recursive expansion.
//
// A level's inverse starts from a combination of matrices that are already there and is finished by
// residual corrections of order 2, 3 or 5:
//   W = I - Y,  W0 = g0 I + g1 W_{k-1} + g2 S_k + g3 S_{k-1},  S_k = T_k^2,
//   Q = S_k - W - W S_k (= -R, R = I - Y B),  W <- W + P - P W,  P = Q - Q^2 + ... +- Q^(order-1).
// All of these are functions of one scalar: with w the eigenvalue of W_{k-1},
//   s_k = 4 w (1 - w),  s_{k-1} = w / (1 - w),
// (t = tan(x/2) gives T_k = sin x, I - 2 W_{k-1} = cos x), so the best g is the solution of a scalar
// minimax problem on [0, w_max] and the residual after the corrections is known beforehand.
// At the late levels (w_max = 1/2) the start c Y_{k-1} alone leaves |R| <= 0.136 and takes four Newton
// steps to 1e-8; with S_k and S_{k-1}, which cost one pass over memory, |R| <= 0.017 and one correction of
// order 5 (four products) gives 1.4e-9.  Every factor is a function of one matrix, so all products run in
// symmetric-output mode (half the tiles); the residual Q used to be a dense product.  An expansion of
// 10 levels takes 25-30 dense-equivalent products instead of 59-64 (corrected to 1e-8; 34-40 to the FP64
// path's 1e-16): charges and forces of 4096 atoms in FP16x3 1349 -> 732 ms, of 100 atoms in FP64 254.8 ->
// 198.1 ms, their errors against 64 bits no larger.
#pragma once
#include <algorithm>
#include <cmath>
#include <vector>

namespace xl {

// Corrections of one inverse: orders (2, 3 or 5), each round costing order_products() products.
struct InvOrders {
  int n = 0;
  int order[12] = {0};
};

inline int order_products(int o) { return o == 2 ? 2 : o == 3 ? 3 : 4; }

// Fewest products that bring a residual e0 < 1 below tol (the residual's power is the product of
// the orders); of equal plans the one with the smallest final residual.
inline InvOrders plan_orders(double e0, double tol) {
  InvOrders p;
  double e = e0;
  // far from the end order 5 is the cheapest per digit (5^(1/4) > 3^(1/3) > 2^(1/2))
  while (p.n < 8 && e < 1.0 && std::pow(e, 125.0) > tol) {
    p.order[p.n++] = 5;
    e = std::pow(e, 5.0);
  }
  int best_cost = 1 << 30;
  double best_pow = 0.0;
  int best[3] = {0, 0, 0};
  const int opt[4] = {1, 2, 3, 5};
  // larger orders first: the last round works on the smallest residual
  for (int a = 3; a >= 0; --a)
    for (int b = a; b >= 0; --b)
      for (int c = b; c >= 0; --c) {
        const double pw = (double)opt[a] * opt[b] * opt[c];
        if (std::pow(e, pw) > tol) continue;
        const int cost = (a ? order_products(opt[a]) : 0) + (b ? order_products(opt[b]) : 0) +
                         (c ? order_products(opt[c]) : 0);
        if (cost < best_cost || (cost == best_cost && pw > best_pow)) {
          best_cost = cost;
          best_pow = pw;
          best[0] = opt[a];
          best[1] = opt[b];
          best[2] = opt[c];
        }
      }
  for (int i = 0; i < 3; ++i)
    if (best[i] > 1) p.order[p.n++] = best[i];
  return p;
}

inline int orders_cost(const InvOrders& p) {
  int c = 0;
  for (int i = 0; i < p.n; ++i) c += order_products(p.order[i]);
  return c;
}

// Minimax of |1 - f(x) sum_j c_j phi_j(x)| over nb <= 4 functions on a grid of kPlanGrid points
// (exchange algorithm).  Returns the maximum over the grid that the returned c has; 1 when it fails
// (c then is all zero).
constexpr int kPlanGrid = 129;
inline double plan_minimax(const std::vector<double>& f, const std::vector<double> (&phi)[4], int nb, double (&c)[4]) {
  const int G = (int)f.size(), m = nb + 1;
  int pt[5];
  for (int i = 0; i < m; ++i) pt[i] = (int)std::lround(0.5 * (1.0 - std::cos(3.14159265358979323846 * i / nb)) * (G - 1));
  double best = 1.0;
  for (int j = 0; j < 4; ++j) c[j] = 0.0;
  std::vector<double> r(G);
  for (int it = 0; it < 8; ++it) {
    double A[5][6];
    for (int i = 0; i < m; ++i) {
      for (int j = 0; j < nb; ++j) A[i][j] = f[pt[i]] * phi[j][pt[i]];
      A[i][nb] = (i & 1) ? -1.0 : 1.0;
      A[i][m] = 1.0;
    }
    bool ok = true;
    for (int k = 0; k < m && ok; ++k) {
      int p = k;
      for (int i = k + 1; i < m; ++i)
        if (std::fabs(A[i][k]) > std::fabs(A[p][k])) p = i;
      if (!(std::fabs(A[p][k]) > 1e-14)) ok = false;
      for (int j = 0; j <= m; ++j) std::swap(A[k][j], A[p][j]);
      for (int i = 0; i < m && ok; ++i) {
        if (i == k) continue;
        const double q = A[i][k] / A[k][k];
        for (int j = k; j <= m; ++j) A[i][j] -= q * A[k][j];
      }
    }
    if (!ok) break;
    double x[4] = {0, 0, 0, 0};
    for (int j = 0; j < nb; ++j) x[j] = A[j][m] / A[j][j];
    double e = 0.0;
    for (int i = 0; i < G; ++i) {
      double y = 0.0;
      for (int j = 0; j < nb; ++j) y += x[j] * phi[j][i];
      r[i] = 1.0 - f[i] * y;
      e = std::max(e, std::fabs(r[i]));
    }
    if (!(e < best)) break;   // no longer improving
    best = e;
    for (int j = 0; j < 4; ++j) c[j] = x[j];
    // exchange: the extremum of each run of one sign
    int np = 0, q[8];
    for (int i = 0; i < G;) {
      int b = i, j = i;
      while (j < G && (r[j] >= 0) == (r[i] >= 0)) {
        if (std::fabs(r[j]) > std::fabs(r[b])) b = j;
        ++j;
      }
      if (np < 8) q[np] = b;
      ++np;
      i = j;
    }
    if (np < m || np > 8) break;
    const int off = (np > m && std::fabs(r[q[0]]) < std::fabs(r[q[np - 1]])) ? np - m : 0;
    bool same = true;
    for (int i = 0; i < m; ++i) {
      same = same && pt[i] == q[off + i];
      pt[i] = q[off + i];
    }
    if (same) break;
  }
  return best;
}

// One level: W0 = g[0] I + g[1] W_{k-1} + g[2] S_k + g[3] S_{k-1} (nb of them in use) and the corrections.
struct LevelPlan {
  int nb = 0;
  double g[4] = {0, 0, 0, 0};
  double e0 = 0.0;      // max |R| of the start over the spectrum
  InvOrders inv;
};

// Level k > 0 with eigenvalues of W_{k-1} in [0, wmax]: the smallest set of functions that needs
// the fewest products.  A set whose coefficients would magnify the rounding errors of the matrices
// (sum |g_j| > 16; the functions are nearly dependent for small wmax) is passed over.
inline LevelPlan plan_level(double wmax, double tol) {
  std::vector<double> f(kPlanGrid), phi[4];
  for (auto& p : phi) p.resize(kPlanGrid);
  // the functions are scaled to order one, so that narrow spectra stay well conditioned
  const double scale[4] = {1.0, wmax, 4.0 * wmax, wmax};
  for (int i = 0; i < kPlanGrid; ++i) {
    const double w = wmax * i / (kPlanGrid - 1), s = 4.0 * w * (1.0 - w);
    f[i] = 1.0 + s;
    phi[0][i] = 1.0;
    phi[1][i] = w / scale[1];
    phi[2][i] = s / scale[2];
    phi[3][i] = w / (1.0 - w) / scale[3];
  }
  LevelPlan best;
  int cost = 1 << 30;
  for (int nb = 2; nb <= 4; ++nb) {
    double c[4];
    // the grid resolves the maximum of these low-order residuals to well under 1 %
    const double e = 1.01 * plan_minimax(f, phi, nb, c);
    for (int j = 0; j < 4; ++j) c[j] /= scale[j];
    if (!(e < 0.5) || std::fabs(c[1]) + std::fabs(c[2]) + std::fabs(c[3]) > 16.0) continue;
    const InvOrders o = plan_orders(e, tol);
    if (orders_cost(o) >= cost) continue;
    cost = orders_cost(o);
    best.nb = nb;
    best.g[0] = 1.0 - c[0];
    for (int j = 1; j < 4; ++j) best.g[j] = -c[j];
    best.e0 = e;
    best.inv = o;
  }
  if (best.nb == 0) {   // cannot happen for wmax <= 1/2; the start c Y_{k-1} always converges
    best.nb = 2;
    best.g[0] = -0.2;
    best.g[1] = 1.2;
    best.e0 = 0.5;
    best.inv = plan_orders(0.5, tol);
  }
  return best;
}

// Level 0 from S_0 alone: minimax line of 1/(1 + s) on [0, smax] (Chebyshev polynomial of degree 2).
inline LevelPlan plan_level0(double smax, double tol) {
  LevelPlan p;
  p.nb = 3;
  // 1 - (1 + s)(a + b s) = T_2(y)/T_2(y0), y the map of [0, smax] to [-1, 1] and y0 that of s = -1
  const double y0 = -1.0 - 2.0 / std::max(smax, 1e-12);
  const double d = 2.0 * y0 * y0 - 1.0, h = 2.0 / std::max(smax, 1e-12);
  // T_2(h s - 1) = 2 h^2 s^2 - 4 h s + 1; divide 1 - T_2/d by (1 + s)
  const double b = -2.0 * h * h / d, a = 1.0 - 1.0 / d;
  p.g[0] = 1.0 - a;
  p.g[2] = -b;
  p.e0 = std::min(0.5, 1.01 / d);
  p.inv = plan_orders(p.e0, tol);
  return p;
}

// Inverse of I - S for eigenvalues of S in [0, smax], smax < 1: Z0 = z0 I + z1 S and its corrections.
struct ResolventPlan {
  double z0 = 1.0, z1 = 1.0;
  InvOrders inv;
};

inline ResolventPlan plan_resolvent(double smax, double tol) {
  ResolventPlan p;
  const double sm = std::max(smax, 1e-12), h = 2.0 / sm, y0 = h - 1.0;   // s = 1
  const double d = 2.0 * y0 * y0 - 1.0;
  // 1 - (1 - s)(a + b s) = T_2(h s - 1)/d
  p.z0 = 1.0 - 1.0 / d;
  p.z1 = 2.0 * h * h / d;
  p.inv = plan_orders(std::min(1.01 / d, 1.0 - 1e-9), tol);
  return p;
}

// Plans of the levels, kept per start interval: wmax is rounded up to the next of 16 steps per
// octave, so a search or a trajectory meets the same few intervals again and again.
class PlanCache {
 public:
  const LevelPlan& level(double wmax, double tol) {
    const double lg = std::max(-60.0, std::log2(std::max(wmax, 1e-18)));
    int key = (int)std::ceil(lg * 16.0 - 1e-9);
    key = std::min(key, -16);   // wmax <= 1/2
    for (auto& e : v_)
      if (e.key == key && e.tol == tol) return e.p;
    v_.push_back({key, tol, plan_level(std::exp2(key / 16.0), tol)});
    return v_.back().p;
  }

 private:
  struct E {
    int key;
    double tol;
    LevelPlan p;
  };
  std::vector<E> v_;   // at most 16 x 60 entries
};

// The unit probes of the exact kernel in parts of one size that run side by side: 96 probes on 64 slots as
// 48 + 48 and not as 64 + 32, which is one wave of tiles less.  side is the size of a part when memory sets no
// limit: the form of a chain level (and with it the rounding) is chosen by it, so that K does not
// depend on how much memory was free when the slots were made.
constexpr int kMaxSlots = 64;
struct ProbeParts {
  int size, side;
};
inline ProbeParts probe_parts(int nat, int slots) {
  auto even = [nat](int s) {
    const int parts = (nat + s - 1) / s;
    return (nat + parts - 1) / parts;
  };
  return {even(std::max(1, std::min(slots, nat))), even(std::min(nat, kMaxSlots))};
}

// The whole expansion: level 0 on |t| <= t0max, then t <- 2 t / (1 + t^2).
inline void plan_expansion(PlanCache& cache, double t0max, int n, double tol, std::vector<LevelPlan>& out) {
  out.resize(n);
  double t = t0max;
  for (int k = 0; k < n; ++k) {
    const double s = t * t;
    if (k == 0)
      out[0] = plan_level0(s, tol);
    else
      // eigenvalues of W_{k-1}: w = s/(1+s) of the level before; s here is 4 w (1 - w)
      out[k] = cache.level(std::min(0.5, 0.5 * (1.0 - std::sqrt(std::max(0.0, 1.0 - s)))), tol);
    t = 2.0 * t / (1.0 + s);
  }
}

}  // namespace xl
