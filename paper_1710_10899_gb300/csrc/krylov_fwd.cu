// Forward by the Krylov engine (krylov.cuh): one persistent launch per size class, one CTA per
// submatrix, FP64 or double-float arithmetic.  The mixed mode's inverse (p = 1) is refined to FP64
// accuracy, as the coupled iteration's is: n = 12288, orders 36..244, 59.5 -> 17.8 ms at the same
// error (2.5e-15), of which the FP64 residual and the correction take 4.
#include <algorithm>
#include <cmath>
#include <mutex>

#include "krylov.cuh"

namespace submat {
namespace kry {
namespace {

// Relative bound at which the recurrence stops.  FP64: its rounding.  Double-float serves the
// mixed mode, whose tensor-core rows are off by 1e-10 to 1e-9 at these orders; the bound
// overestimates the error about tenfold, and two digits more would cost four steps in thirty.
template <class T> struct Tol;
template <> struct Tol<df> { static constexpr float value = 1e-11f; };
template <> struct Tol<double> { static constexpr float value = 2e-16f; };
// The correction of the double-float inverse: four digits of a residual near 1e-12.
constexpr float kTolFix = 3e-4f;

// What became of a row: left to the general path, written, or to be computed again in FP64.
enum RowState { kLeft, kWritten, kAgain };

// Row r.j's column (r bound, its flag 1 zero).  The same on every thread.
template <int NE, class T, int NW, bool GP, bool ALL>
__device__ __forceinline__ RowState column(Row<T, NW, GP, ALL, false>& r, const Args& a) {
  constexpr int NT = threads_of<NW, ALL>();
  constexpr int NM = NW * 32;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const bool mat = warp < NW, node = kLone<NW, ALL> || warp == NW;
  double* scale_s = reinterpret_cast<double*>(r.flag() + 4);
  const int p = a.p;
  const bool direct = p == 1 && a.sign > 0;          // A itself, once it is found definite
  bool ok = gather(r, a);
  int K = 0, nc = 0;
  double fix[NE];
  double res1 = 0.0;                               // p = 1: the column's residual, in FP64
  float est = 0.f, lo = 1.f;
  if (ok) {
    stats(r);
    if (!direct) {
      for (int i = tid; i < r.mp; i += NT) r.set_v(i, i == r.pos ? one<T>() : zero<T>());
      sync_all<NW, ALL>();
      K = lanczos<NE>(r, p, a.sign, Tol<T>::value, &est, &lo);
      // the recurrence's bound not met (NaN is not): nothing more is spent on the row
      if (node && lane == 0)
        r.flag()[6] = !(lo > 0.f && est <= Tol<T>::value) ? 0 : lo * a.kappa_max < 1.f ? 2 : 1;
      sync_all<NW, ALL>();
      ok = r.flag()[6] != 0;
      if constexpr (kDf<T>) {
        // rows whose condition estimate exceeds kappa_max are FP64's on every engine of the mixed
        // mode (p = 1 is refined to that below).  The recurrence's own bracket says which rows to
        // estimate at all; it is the sharper one, and rows above kappa_max by it alone (2 in 1000
        // of the small overlap matrices) are within 2e-11 here, within 1e-8 on the other engines.
        if (p > 1 && r.flag()[6] == 2 && condition_estimate<NW, GP, ALL>(a, r.m, r.lam) > a.kappa_max) return kAgain;
      }
    }
  }
  if (ok) {
    if constexpr (kDf<T>) {
      if (p == 1 && !direct) {
        // The inverse's column to FP64 accuracy (as the coupled iteration's): x from the
        // double-float recurrence, its residual in FP64, and a single-precision recurrence
        // for the correction, which needs few digits.  x stays in registers.
        if (node) {
          nc = root_coefs(r, K, p, lo, false, lane);
          if (lane == 0) r.flag()[3] = K + 1;
        }
        sync_all<NW, ALL>();
        nc = r.flag()[3] - 1;
        const double unit = exp2((double)(1023 - r.e0));
        double* xd = reinterpret_cast<double*>(r.part());
        double* rd = reinterpret_cast<double*>(r.X);
        if (mat)
#pragma unroll
          for (int e = 0; e < NE; ++e) {
            const int i = tid + e * NM;
            fix[e] = 0.0;
            if (i < r.m) {
              T s = zero<T>();
              for (int k = 0; k < nc; ++k) s = add(s, mul(r.coef()[k], r.V[(size_t)k * r.mp + i]));
              fix[e] = join(s) * unit;
              xd[i] = fix[e];
            }
          }
        sync_all<NW, ALL>();
        residual(r, a, xd, rd);
        sync_all<NW, ALL>();
        Row<float, NW, GP, ALL, false> q;
        q.m = r.m, q.nb = r.nb, q.mp = r.mp, q.ns = r.ns, q.pos = r.pos, q.j = r.j;
        q.o_part = r.o_part, q.o_t = 0;
        q.gblk = r.gblk;
        q.gpart = reinterpret_cast<float*>(r.gpart);
        q.V = reinterpret_cast<float*>(r.V);
        q.X = reinterpret_cast<float*>(r.X);
        q.AB = nullptr;
        q.e0 = r.e0, q.lam = r.lam, q.C = r.C, q.sigma = r.sigma;
        float n2 = 0.f;
        for (int i = tid; i < r.mp; i += NT) {
          const float x = i < r.m ? (float)rd[i] : 0.f;
          q.set_v(i, x);
          n2 = fmaf(x, x, n2);
        }
        n2 = warp_total(n2);
        if (lane == 0) q.red()[warp] = n2;
        sync_all<NW, ALL>();
        n2 = total_of<NT / 32>(q.red(), lane, NT / 32);
        res1 = sqrt((double)n2);
        const float inv = n2 > 1e-36f ? rsqrtf(n2) : 0.f;
        for (int i = tid; i < r.mp; i += NT) q.set_v(i, q.v_at(i) * inv);
        sync_all<NW, ALL>();
        if (inv > 0.f) {                            // (the residual may vanish: m = 1)
          float est2 = 0.f, lo2 = 0.f;
          const int K2 = lanczos<NE>(q, 1, -1, kTolFix, &est2, &lo2);
          if (node) {
            root_coefs(q, K2, 1, lo2, false, lane);
            if (lane == 0 && !(lo2 > 0.f && est2 <= kTolFix)) r.flag()[3] = 0;
          }
          sync_all<NW, ALL>();
          if (mat)
#pragma unroll
            for (int e = 0; e < NE; ++e) {
              const int i = tid + e * NM;
              float s = 0.f;
              if (i < r.m)
                for (int k = 0; k < K2; ++k) s = fmaf(q.coef()[k], q.V[(size_t)k * r.mp + i], s);
              fix[e] = fma((double)(s * (n2 * inv)), unit, fix[e]);
            }
          sync_all<NW, ALL>();
        }
      }
    }
    if (node) {
      const float tau_f = tau_of(r.lam, lo);
      const bool fixed_up = kDf<T> && p == 1 && !direct;        // done above
      if (!direct && !fixed_up) nc = root_coefs(r, K, p, lo, a.sign > 0, lane);
      if (lane == 0) {
        const double E = (double)(r.e0 - 1023), ex = (double)a.sign / (double)p;
        const double tau = (double)tau_f;
        const double al = a.sign < 0 ? 1.0 / (double)p : 1.0 - 1.0 / (double)p;
        *scale_s = exp2(E * ex) * (p > 1 ? pow(tau, -al) : 1.0);
        // for p = 1 the residual of the column (before its correction) is what is compared, as in
        // refine_column
        if (!fixed_up) r.flag()[3] = direct || (double)est <= a.resid_tol ? nc + 1 : 0;
        else if (!(res1 <= a.resid_tol)) r.flag()[3] = 0;
      }
    }
    if (mat) cholesky(r);
    sync_all<NW, ALL>();
    nc = r.flag()[3] - 1;
    ok = nc >= 0 && r.flag()[1] == 0;
    if constexpr (!kDf<T>) {
      if (ok && p == 1 && !direct) {                // the residual of the FP64 inverse's column
        double* xd = r.part();
        double* rd = r.X;
        const double unit = exp2((double)(1023 - r.e0));
        for (int i = tid; i < r.m; i += NT) {
          double s = 0.0;
          for (int k = 0; k < nc; ++k) s += r.coef()[k] * r.V[(size_t)k * r.mp + i];
          xd[i] = s * unit;
        }
        sync_all<NW, ALL>();
        residual(r, a, xd, rd);
        sync_all<NW, ALL>();
        double n2 = 0.0;
        for (int i = tid; i < r.m; i += NT) n2 = fma(rd[i], rd[i], n2);
        n2 = warp_total(n2);
        if (lane == 0) r.red()[warp] = n2;
        sync_all<NW, ALL>();
        res1 = sqrt(total_of<NT / 32>(r.red(), lane, NT / 32));
        ok = res1 <= a.resid_tol;
        if (ok)
          for (int i = tid; i < r.m; i += NT) a.out[a.rowptr[r.j] + i] = xd[i];
      }
    }
  }
  if (ok) {
    const double scale = *scale_s;
    double* out = a.out + a.rowptr[r.j];
    if (direct) {
      for (int i = tid; i < r.m; i += NT) out[i] = a.vals[a.rowptr[r.j] + i];
    } else if (!kDf<T> && p == 1) {
      // written above
    } else if (kDf<T> && p == 1) {
      if (mat)
#pragma unroll
        for (int e = 0; e < NE; ++e) {
          const int i = tid + e * NM;
          if (i < r.m) out[i] = fix[e];
        }
    } else if (mat) {
      for (int i = tid; i < r.m; i += NM) {
        T s = zero<T>();
        for (int k = 0; k < nc; ++k) s = add(s, mul(r.coef()[k], r.V[(size_t)k * r.mp + i]));
        out[i] = join(s) * scale;
      }
    }
  }
  if (node && lane == 0) {
    if (!ok) {
      leave(r, a);
    } else {
      // (without a recurrence: on the certified interval)
      const int iters = coupled_steps(direct ? r.sigma / r.lam : lo, p, r.m, !kDf<T>);
      const double m2 = (double)r.m * r.m;
      atomicMax(&a.ctr->iters_max, iters);
      atomicAdd(&a.ctr->iters_sum, (unsigned long long)iters);
      atomic_max_nonneg(&a.ctr->resid_max_bits, p == 1 && !direct ? res1 : (double)est);
      if (!kDf<T>) atomicAdd(&a.ctr->flops_fp64, 2.0 * m2 * (double)K);
      else atomicAdd(&a.ctr->products_df, m2 * (double)K);
      atomicAdd(&a.ctr->flops_alg, ((double)iters * (p + 1) + (p == 1 ? 1.0 : 0.0)) * 2.0 * m2 * r.m);
    }
  }
  return ok ? kWritten : kLeft;
}

// A double-float row over again in FP64 (the storage of both has 8 bytes an element).
template <int NE, int NW, bool GP, bool ALL>
__device__ __noinline__ void column_fp64(const Args& a, int j) {
  Row<double, NW, GP, ALL, false> r;
  bind_storage(r, a);
  take_row(r, a, j);
  sync_all<NW, ALL>();                               // the flags of the first attempt have been read
  column<NE>(r, a);
}

template <class T, int NW, bool GP, bool ALL, int NE, int MINB>
__global__ void __launch_bounds__(threads_of<NW, ALL>(), MINB) fwd_kernel(const __grid_constant__ Args a) {
  Row<T, NW, GP, ALL, false> r;
  bind_storage(r, a);
  load_nodes(r, a);
  for (;;) {
    if (threadIdx.x == 0) {
      r.flag()[2] = atomicAdd(a.queue, 1);
      r.flag()[1] = 0;
    }
    sync_all<NW, ALL>();
    const int idx = r.flag()[2];
    if (idx >= a.n) break;
    take_row(r, a, a.order[idx]);
    const RowState st = column<NE>(r, a);
    if constexpr (kDf<T>)
      if (st == kAgain) column_fp64<NE, NW, GP, ALL>(a, r.j);
    sync_all<NW, ALL>();
  }
}

template <class T, int NW, bool GP, bool ALL, int NE, int MINB>
cudaError_t run(const Args& a, int grid, cudaStream_t s) {
  const Layout L = layout(a.nb, a.ns, NW, !GP, false);
  if (((ALL || NW == 1) && a.ns < nblocks(a.nb)) || L.total > kMaxSmem) return cudaErrorInvalidValue;
  fwd_kernel<T, NW, GP, ALL, NE, MINB><<<grid, threads_of<NW, ALL>(), L.total, s>>>(a);
  return cudaGetLastError();
}
template <class T, int NW, bool GP, bool ALL, int NE, int MINB>
cudaError_t attr() {
  return cudaFuncSetAttribute(fwd_kernel<T, NW, GP, ALL, NE, MINB>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              kMaxSmem);
}

template <class T>
cudaError_t dispatch(const Args& a, const Class& c, int grid, cudaStream_t s) {
  switch (c.nw) {
    case 1: return c.lone ? run<T, 1, false, false, 1, 16>(a, grid, s) : run<T, 1, false, true, 1, 8>(a, grid, s);
    case 3: return run<T, 3, false, true, 1, 4>(a, grid, s);
    case 5: return run<T, 5, false, true, 1, 2>(a, grid, s);
  }
  if (c.nb <= 6) return run<T, 15, false, true, 1, 1>(a, grid, s);
  return c.part_smem ? run<T, 15, false, false, 1, 1>(a, grid, s) : run<T, 15, true, false, 4, 1>(a, grid, s);
}

template <class T>
cudaError_t attrs() {
  cudaError_t e;
  if ((e = attr<T, 1, false, true, 1, 8>()) != cudaSuccess) return e;
  if ((e = attr<T, 1, false, false, 1, 16>()) != cudaSuccess) return e;
  if ((e = attr<T, 3, false, true, 1, 4>()) != cudaSuccess) return e;
  if ((e = attr<T, 5, false, true, 1, 2>()) != cudaSuccess) return e;
  if ((e = attr<T, 15, false, true, 1, 1>()) != cudaSuccess) return e;
  if ((e = attr<T, 15, false, false, 1, 1>()) != cudaSuccess) return e;
  return attr<T, 15, true, false, 4, 1>();
}

}  // namespace

cudaError_t launch_fwd(const Args& a, const Class& c, int grid, cudaStream_t s) {
  return a.fp64 ? dispatch<double>(a, c, grid, s) : dispatch<df>(a, c, grid, s);
}

cudaError_t set_attr_fwd() {
  const cudaError_t e = attrs<df>();
  return e != cudaSuccess ? e : attrs<double>();
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
