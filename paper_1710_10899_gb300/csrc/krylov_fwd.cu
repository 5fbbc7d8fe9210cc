// Host side of the Krylov forward: its instances' launchers, the quadrature tables and the size classes.
#include <algorithm>
#include <cmath>
#include <mutex>

#include "krylov.cuh"

namespace submat {
namespace kry {

cudaError_t launch_fwd(const Args& a, const Class& c, int grid, cudaStream_t s) {
  if (a.p == 1 && a.sign < 0) return a.fp64 ? launch_inverse_fp64(a, c, grid, s) : launch_inverse_df(a, c, grid, s);
  return a.fp64 ? launch_roots_fp64(a, c, grid, s) : launch_roots_df(a, c, grid, s);
}

cudaError_t set_attr_fwd(int p, int sign, bool fp64) {
  if (p == 1 && sign < 0) return fp64 ? set_attr_inverse_fp64() : set_attr_inverse_df();
  return fp64 ? set_attr_roots_fp64() : set_attr_roots_df();
}

// Gauss-Jacobi nodes for the weight (1-s)^(-a) (1+s)^(a-1): Newton's method on the Jacobi
// polynomial P_N^(-a, a-1) from the asymptotic zeros; a weight is proportional to
// 1 / ((1 - s^2) P'(s)^2), and the weights are scaled to the sum 1, which makes the rule
// exact at x = tau.
template <class F>
static F jacobi_step(int N, F a, F b, F x, F* dp) {         // P_N(x) / P_N'(x)
  const F ab = a + b;
  F p0 = 1, p1 = ((a - b) + (ab + 2) * x) / 2;              // P_0, P_1
  for (int k = 2; k <= N; ++k) {
    const F c = 2 * k + ab;
    const F p2 = ((c - 1) * (c * (c - 2) * x + a * a - b * b) * p1 -
                  2 * (k + a - 1) * (k + b - 1) * c * p0) /
                 (2 * k * (k + ab) * (c - 2));
    p0 = p1;
    p1 = p2;
  }
  const F c = 2 * N + ab;
  *dp = (N * (a - b - c * x) * p1 + 2 * (N + a) * (N + b) * p0) / (c * (1 - x * x));
  return p1 / *dp;
}
static bool gauss_jacobi(int N, double al, double* theta, double* weight) {
  typedef long double ld;
  const ld a = -(ld)al, b = (ld)al - 1.0L;                  // a + b = -1
  ld sum = 0.0L, s[kNodesWide], w[kNodesWide];
  for (int q = 0; q < N; ++q) {
    double xd = std::cos(3.14159265358979323846 * (q + 0.75 - al / 2) / N), dpd = 0.0;   // ab = -1
    for (int it = 0; it < 30; ++it) {
      const double dx = jacobi_step<double>(N, -al, al - 1.0, xd, &dpd);
      xd -= dx;
      if (!(std::fabs(dx) > 1e-15)) break;
    }
    ld x = xd, dp = 0.0L;                                   // polished in extended precision
    x -= jacobi_step<ld>(N, a, b, x, &dp);
    jacobi_step<ld>(N, a, b, x, &dp);
    if (!(x > -1.0L && x < 1.0L)) return false;
    s[q] = x;
    w[q] = 1.0L / ((1 - x * x) * dp * dp);
    sum += w[q];
  }
  for (int q = 0; q < N; ++q) {
    if (q > 0 && !(s[q] < s[q - 1])) return false;          // two starts met in one zero
    theta[q] = (double)((1 - s[q]) / (1 + s[q]));
    weight[q] = (double)(w[q] / sum * 2 / (1 + s[q]));
  }
  return true;
}

static bool make_nodes(int p, int sign, Nodes* out) {
  *out = Nodes{};
  if (p == 1) return true;                                  // x^(-1) needs no quadrature
  const double al = sign < 0 ? 1.0 / p : 1.0 - 1.0 / p;
  return gauss_jacobi(kNodes, al, out->theta, out->w) &&
         gauss_jacobi(kNodesWide, al, out->theta + kNodes, out->w + kNodes) &&
         gauss_jacobi(kNodesGrad, al, out->theta + kNodes + kNodesWide, out->w + kNodes + kNodesWide);
}

bool cached_nodes(int p, int sign, Nodes* out) {     // a constant table per (p, sign)
  static std::mutex lock;
  static Nodes table[2][SUBMAT_MIXED_MAX_P + 1];
  static bool have[2][SUBMAT_MIXED_MAX_P + 1] = {};
  if (p < 1 || p > SUBMAT_MIXED_MAX_P) return false;
  const int s = sign < 0 ? 0 : 1;
  std::lock_guard<std::mutex> hold(lock);
  if (!have[s][p]) have[s][p] = make_nodes(p, sign, &table[s][p]);
  *out = table[s][p];
  return have[s][p];
}

// Classes by order: warps per CTA and CTAs per SM.  S's blocks fill what shared memory the
// CTAs per SM leave; a class whose blocks do not all fit streams the rest from scratch (L2).
constexpr int kClassMax[] = {32, 64, 96, 128, 192, SUBMAT_MAX_M};
constexpr int kClassWarps[] = {1, 3, 3, 5, 15, 15};    // matrix warps (and one for the nodes)
constexpr int kClassCtas[] = {8, 4, 3, 2, 1, 1};

int class_of(int m) {
  int i = 0;
  while (m > kClassMax[i]) ++i;
  return i;
}

Class make_class(int index, int m_max, int rows, int n_sm, bool bwd) {
  Class c;
  c.max_m = std::min(kClassMax[index], (m_max + kB - 1) / kB * kB);
  c.nw = kClassWarps[index];
  c.nb = c.max_m / kB;
  c.ctas = kClassCtas[index];
  if (index == 0) {
    // Two warps a row while the rows are at most about two waves of them, then one warp and twice
    // the rows per SM (as far as the adjoint's factors, 16 KB a CTA, leave room): n = 200, 98 -> 78 us with two;
    // n = 2000, FP64, 343 -> 260; n = 4000, double-float, 263 -> 205 with one; adjoint n = 700, 351 -> 338
    // with two, n = 2000, 430 -> 388 with one.
    c.lone = rows > n_sm * (bwd ? 8 : 16);
    if (c.lone && !bwd) c.ctas = 16;
  }
  c.part_smem = c.max_m <= 480;
  const bool all = index + 1 < (int)(sizeof(kClassMax) / sizeof(kClassMax[0]));   // holds every block
  for (;; --c.ctas) {
    const size_t room = 233472 / c.ctas - 1024;      // 228 KB an SM, 1 KB reserved per CTA
    c.ns = nblocks(c.nb);
    while (c.ns > 0 && layout(c.nb, c.ns, c.nw, c.part_smem, bwd).total > room) --c.ns;
    if (c.ns > 0 && (!all || c.ns == nblocks(c.nb))) break;
    if (c.ctas == 1) break;                          // refused by the launch
  }
  return c;
}

}  // namespace kry
}  // namespace submat
