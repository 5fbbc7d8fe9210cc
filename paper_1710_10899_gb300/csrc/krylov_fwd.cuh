// Forward by the Krylov engine (krylov.cuh): one persistent launch per size class, one CTA per
// submatrix, FP64 or double-float arithmetic.  The kernel; the roots and the inverse are instances of
// their own (what only one of them needs costs the other up to 5 % at orders up to 32: registers),
// compiled in files of their own.
// The mixed mode's inverse (p = 1) is refined to FP64 accuracy, as the coupled iteration's is: n =
// 12288, orders 36..244, 59.5 -> 17.9 ms at the same error (2.5e-15), of which the FP64 residual and the
// correction take 4.
#pragma once
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

// Row r.j's column (r bound, its flag 1 zero).  The same on every thread.  INV: the inverse (p = 1).
template <bool INV, int NE, class T, int NW, bool GP, bool ALL>
__device__ __forceinline__ RowState column(Row<T, NW, GP, ALL, false>& r, const Args& a) {
  constexpr int NT = threads_of<NW, ALL>();
  constexpr int NM = NW * 32;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const bool mat = warp < NW, node = kLone<NW, ALL> || warp == NW;
  double* scale_s = reinterpret_cast<double*>(r.flag() + 4);
  const int p = INV ? 1 : a.p;
  const bool direct = !INV && p == 1;                // A itself, once it is found definite
  bool ok = gather(r, a);
  int K = 0, nc = 0;
  double fix[NE];
  double res1 = 0.0;                                 // p = 1: the column's residual, in FP64
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
    }
  }
  if (ok) {
    if constexpr (kDf<T> && INV) {
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
    if constexpr (!kDf<T> && INV) {
      // The inverse's column in FP64 (in registers) and its residual, by one more product.  It needs S,
      // so the node solve is not hidden behind the factorisation: n = 2048, orders 28..239, 6.66 ->
      // 6.96 ms (from the pattern rows instead, after the factorisation: 7.04; n = 2000, orders up to
      // 28: 248 us, 281 from the rows).
      if (node) {
        nc = root_coefs(r, K, p, lo, false, lane);
        if (lane == 0) r.flag()[3] = nc + 1;
      }
      sync_all<NW, ALL>();
      if (mat) {
        nc = r.flag()[3] - 1;
#pragma unroll
        for (int e = 0; e < NE; ++e) {
          const int i = tid + e * NM;
          fix[e] = 0.0;
          if (i < r.mp) {
            for (int k = 0; k < nc; ++k) fix[e] += r.coef()[k] * r.V[(size_t)k * r.mp + i];
            r.set_v(i, fix[e]);
          }
        }
        sync_mat<NW>();
        double dot = 0.0;
        for_blocks(r, warp, [&](int t, int I, int J) {
          auto go = [&](const float4* x) {
            if (I == J) block_mul<false>(x, r.v(), I, J, 0.f, r.part(), r.mp, lane, dot);
            else block_mul<true>(x, r.v(), I, J, 0.f, r.part(), r.mp, lane, dot);
          };
          if (ALL || t < r.ns) go(r.sblk(t)); else go(r.gblk_at(t));
        });
        sync_mat<NW>();
        double n2 = 0.0;
#pragma unroll
        for (int e = 0; e < NE; ++e) {
          const int i = tid + e * NM;
          if (i < r.m) {
            const double d = (i == r.pos ? 1.0 : 0.0) - row_sum<NW>(r.part(), i, r.mp, r.nb);
            n2 = fma(d, d, n2);
          }
        }
        n2 = warp_total(n2);
        if (lane == 0) r.red()[warp] = n2;
      }
    }
    if (node) {
      const float tau_f = tau_of(r.lam, lo);
      constexpr bool fixed_up = INV;                            // done above
      if (!direct && !fixed_up) nc = root_coefs(r, K, p, lo, a.sign > 0, lane);
      if (lane == 0) {
        const double E = (double)(r.e0 - 1023), ex = (double)a.sign / (double)p;
        const double tau = (double)tau_f;
        const double al = a.sign < 0 ? 1.0 / (double)p : 1.0 - 1.0 / (double)p;
        *scale_s = exp2(E * ex) * (p > 1 ? pow(tau, -al) : 1.0);
        // for p = 1 the residual of the column (before its correction) is what is compared, as in
        // refine_column
        if (!fixed_up) r.flag()[3] = direct || (double)est <= a.resid_tol ? nc + 1 : 0;
        else if (kDf<T> && !(res1 <= a.resid_tol)) r.flag()[3] = 0;
      }
    }
    // Rows whose condition estimate exceeds kappa_max are FP64's on every engine of the mixed mode
    // (p = 1 is refined to that above).  The recurrence's own bracket says which rows to estimate
    // at all; it is the sharper one, and rows above kappa_max by it alone (2 in 1000 of the small
    // overlap matrices) are within 2e-11 here, within 1e-8 on the other engines.
    const bool wide = kDf<T> && !INV && !direct && r.flag()[6] == 2;
    if (mat) {
      bool again = false;
      if constexpr (kDf<T> && !INV) {
        if (wide) {
          again = condition_estimate<NW, GP, ALL>(a, r.m, r.lam) > a.kappa_max;
          if (tid == 0) r.flag()[7] = again;
        }
      }
      if (!again) cholesky(r);
    }
    sync_all<NW, ALL>();
    if (wide && r.flag()[7]) return kAgain;
    nc = r.flag()[3] - 1;
    ok = nc >= 0 && r.flag()[1] == 0;
    if constexpr (!kDf<T> && INV) {
      res1 = sqrt(total_of<NW>(r.red(), lane, NW));
      ok = ok && res1 <= a.resid_tol;
    }
  }
  if (ok) {
    const double scale = *scale_s;
    double* out = a.out + a.rowptr[r.j];
    if (direct) {
      for (int i = tid; i < r.m; i += NT) out[i] = a.vals[a.rowptr[r.j] + i];
    } else if constexpr (INV) {
      const double unit = kDf<T> ? 1.0 : exp2((double)(1023 - r.e0));
      if (mat)
#pragma unroll
        for (int e = 0; e < NE; ++e) {
          const int i = tid + e * NM;
          if (i < r.m) out[i] = fix[e] * unit;
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
      atomic_max_nonneg(&a.ctr->resid_max_bits, INV ? res1 : (double)est);
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
  column<false, NE>(r, a);
}

template <bool INV, class T, int NW, bool GP, bool ALL, int NE, int MINB>
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
    const RowState st = column<INV, NE>(r, a);
    if constexpr (kDf<T> && !INV)
      if (st == kAgain) column_fp64<NE, NW, GP, ALL>(a, r.j);
    sync_all<NW, ALL>();
  }
}

template <bool INV, class T, int NW, bool GP, bool ALL, int NE, int MINB>
cudaError_t run(const Args& a, int grid, cudaStream_t s) {
  const Layout L = layout(a.nb, a.ns, NW, !GP, false);
  if (((ALL || NW == 1) && a.ns < nblocks(a.nb)) || L.total > kMaxSmem) return cudaErrorInvalidValue;
  fwd_kernel<INV, T, NW, GP, ALL, NE, MINB><<<grid, threads_of<NW, ALL>(), L.total, s>>>(a);
  return cudaGetLastError();
}
template <bool INV, class T, int NW, bool GP, bool ALL, int NE, int MINB>
cudaError_t attr() {
  return cudaFuncSetAttribute(fwd_kernel<INV, T, NW, GP, ALL, NE, MINB>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              kMaxSmem);
}

template <bool INV, class T>
cudaError_t dispatch(const Args& a, const Class& c, int grid, cudaStream_t s) {
  switch (c.nw) {
    case 1: return c.lone ? run<INV, T, 1, false, false, 1, 16>(a, grid, s) : run<INV, T, 1, false, true, 1, 8>(a, grid, s);
    case 3: return run<INV, T, 3, false, true, 1, 4>(a, grid, s);
    case 5: return run<INV, T, 5, false, true, 1, 2>(a, grid, s);
  }
  if (c.nb <= 6) return run<INV, T, 15, false, true, 1, 1>(a, grid, s);
  return c.part_smem ? run<INV, T, 15, false, false, 1, 1>(a, grid, s) : run<INV, T, 15, true, false, 4, 1>(a, grid, s);
}

template <bool INV, class T>
cudaError_t attrs() {
  cudaError_t e;
  if ((e = attr<INV, T, 1, false, true, 1, 8>()) != cudaSuccess) return e;
  if ((e = attr<INV, T, 1, false, false, 1, 16>()) != cudaSuccess) return e;
  if ((e = attr<INV, T, 3, false, true, 1, 4>()) != cudaSuccess) return e;
  if ((e = attr<INV, T, 5, false, true, 1, 2>()) != cudaSuccess) return e;
  if ((e = attr<INV, T, 15, false, true, 1, 1>()) != cudaSuccess) return e;
  if ((e = attr<INV, T, 15, false, false, 1, 1>()) != cudaSuccess) return e;
  return attr<INV, T, 15, true, false, 4, 1>();
}

}  // namespace
}  // namespace kry
}  // namespace submat
