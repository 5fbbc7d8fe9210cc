// Adjoint by the Krylov engine (krylov.cuh): for L = <g, f(S) e_pos> and f as a sum of simple
// fractions, f(S) = sum_q w_q (S + t_q)^(-1),
//     dL/dS = - sum_q w_q (x_q y_q^T + y_q x_q^T) / 2,   x_q = (S + t_q)^(-1) g,
//                                                        y_q = (S + t_q)^(-1) e_pos,
// the Daleckii-Krein form of that f (for f(x) = x^(1/p) = sum_q w_q (1 - t_q (x + t_q)^(-1)) the
// weights are + w_q t_q).  Two Lanczos processes (from e_pos and from g) give all x_q and y_q, so
// the gradient of a submatrix is a sum of kNodesGrad (or kNodes) rank-two terms instead of a full
// eigendecomposition: O((k + q) m^2) against the ~9 sweeps of m^3 rotations of a Jacobi method.
// In double-float arithmetic, wide spectra in FP64 (krylov.cuh).  Only stored entries are formed:
// the pattern rows are scanned as in the gather, upper triangle only, and an entry's mirror image is
// found by the transposed map.  Rows that the engine refuses are left to the Jacobi kernel (eig.cu), and so is the
// inverse, where the Jacobi's error is the smaller one (5e-13 against 1.5e-12 of the gradient).
// Measured on GB300, one backward, Jacobi -> this: n = 6144, orders 27..183, p = 2: 514 -> 9.5 ms;
// n = 2501, orders 10..88, deterministic: 24.5 -> 1.6 ms; n = 400, orders up to 300 (which the
// Jacobi kernel keeps in global memory): 2180 -> 2.3 ms; error of the gradient no larger
// (4.2e-12 -> 3.7e-12 on the first).  Bound by the latency of the Lanczos steps, as the forward.
#include "krylov.cuh"

namespace submat {
namespace kry {
namespace {

// Relative bound at which the recurrences stop.
template <class T> constexpr float kTolGrad = kDf<T> ? 1e-13f : 1e-15f;

// f 2^e as a double, by integer operations.
__device__ __forceinline__ double widen(float f, int e) {
  const unsigned b = __float_as_uint(f);
  const int ex = (int)((b >> 23) & 0xFF), ne = ex + 896 + e;
  if (ex == 0 || ne <= 0) return 0.0;
  if (ex == 0xFF || ne >= 0x7FF) return __longlong_as_double(0x7ff8000000000000ll);
  return __hiloint2double((int)((b & 0x80000000u) | ((unsigned)ne << 20) | ((b & 0x7FFFFFu) >> 3)),
                          (int)(b << 29));
}

// Node solutions of both processes (one warp): g's in X0, e_pos's, weighted, in X1.  Every
// factor of the row goes into the weights, their power of two into flag 5.  r is bound to g's
// process (al, be).
template <class T, int NW, bool GP, bool ALL>
__device__ void solve_nodes(Row<T, NW, GP, ALL, true>& r, const Args& a, int K0, int K1, T* X0, T* X1, int t_bytes,
                            T gnorm, int eg, int pass) {
  const int lane = threadIdx.x & 31, p = a.p, Q = r.flag()[3];
  const float lo = __int_as_float(r.flag()[4]);
  const float tau = r.lam * sqrtf(lo);
  const int q0 = lo >= 0.02f ? kNodes + kNodesWide : (lo >= kLoWide ? 0 : kNodes + 32 * pass);
  const int q = q0 + min(lane, Q - 1);
  const double al = a.sign < 0 ? 1.0 / (double)p : 1.0 - 1.0 / (double)p;
  double f = pow((double)tau, -al) * 0.5 * join(gnorm);
  const double E = (double)(r.e0 - 1023) * ((double)a.sign / (double)p - 1.0);
  const double fl = floor(E);
  f *= exp2(E - fl);
  const int ef = ((__double2hiint(f) >> 20) & 0x7FF) - 1023;
  f *= exp2((double)-ef);                            // in [1, 2)
  T wt0 = as(a.sign < 0 ? -f : f, (T*)nullptr);
  if (lane >= Q) wt0 = zero<T>();
  r.X = X0;
  node_solve(r, K1, tau, q, false, false, one<T>());
  r.X = X1;
  r.o_t -= t_bytes;
  node_solve(r, K0, tau, q, true, a.sign > 0, wt0);
  r.o_t += t_bytes;
  r.X = X0;
  if (lane == 0) r.flag()[5] = ef + (int)fl + (eg - 1023);
}

// Row r.j's gradient (r bound, its flag 1 zero), the same on every thread; true: to be computed
// again in FP64, nothing is written.
template <int NE, class T, int NW, bool GP, bool ALL>
__device__ __forceinline__ bool row_gradient(Row<T, NW, GP, ALL, true>& r, const Args& a) {
  constexpr int NT = threads_of<NW, ALL>();
  constexpr int NM = NW * 32;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const bool mat = warp < NW, node = kLone<NW, ALL> || warp == NW;
  const Layout L = layout(a.nb, a.ns, NW, !GP, true);
  constexpr int t_bytes = Row<T, NW, GP, ALL, true>::kF.t_bytes;
  T* const V0 = r.V;
  T* const X0 = r.X;
  T* const V1 = reinterpret_cast<T*>(reinterpret_cast<char*>(V0) + L.v_bytes);
  T* const X1 = reinterpret_cast<T*>(reinterpret_cast<char*>(X0) + L.x_bytes);
  const int p = a.p;
  const bool direct = p == 1 && a.sign > 0;          // f(x) = x: one term, x = g, y = e_pos
  const int base = a.rowptr[r.j];
  bool ok = gather(r, a);
  // g 2^-eg, eg the exponent of its largest entry
  int eg = 0;
  for (int i = tid; i < r.m; i += NT)
    eg = max(eg, __double2hiint(a.grad_out[base + i]) & 0x7FFFFFFF);
  eg = __reduce_max_sync(0xffffffffu, eg);
  int* ired = reinterpret_cast<int*>(r.red());
  sync_all<NW, ALL>();
  if (lane == 0) ired[warp] = eg;
  sync_all<NW, ALL>();
#pragma unroll
  for (int w = 0; w < NT / 32; ++w) eg = max(eg, ired[w]);
  eg >>= 20;
  sync_all<NW, ALL>();
  const bool none = eg == 0;                       // g = 0: no contribution
  ok = ok && eg < 0x7FF - 64 && (none || eg >= 64);
  int K0 = 0, K1 = 0, Q = 1, passes = 1;
  float lo = 1.f;
  T gnorm = one<T>();
  if (ok) {
    stats(r);
    if (!direct && !none) {
      float est0 = 0.f, est1 = 0.f, lo0 = 0.f, lo1 = 0.f;
      for (int i = tid; i < r.mp; i += NT) r.set_v(i, i == r.pos ? one<T>() : zero<T>());
      sync_all<NW, ALL>();
      K0 = lanczos<NE>(r, p, a.sign, kTolGrad<T>, &est0, &lo0);
      if (node && lane == 0) r.flag()[8] = est0 <= kTolGrad<T> && lo0 > 0.f;
      T n2 = zero<T>();
      for (int i = tid; i < r.mp; i += NT) {
        const T x = i < r.m ? scaled(a.grad_out[base + i], eg, (T*)nullptr) : zero<T>();
        r.set_v(i, x);
        n2 = add(n2, mul(x, x));
      }
      n2 = warp_total(n2);
      if (lane == 0) r.red()[warp] = n2;
      sync_all<NW, ALL>();
      n2 = total_of<NT / 32>(r.red(), lane, NT / 32);
      const T inv = inv_sqrt(n2);
      gnorm = mul(n2, inv);
      for (int i = tid; i < r.mp; i += NT) r.set_v(i, mul(r.v_at(i), inv));
      r.V = V1;
      r.o_t += t_bytes;
      sync_all<NW, ALL>();
      // (a row that the first process refuses needs no second)
      if (r.flag()[8]) K1 = lanczos<NE>(r, p, a.sign, kTolGrad<T>, &est1, &lo1);
      if (node) {
        lo = fminf(lo0, lo1);
        // the divided differences need the quadrature over both spectra; a double-float row with
        // a wide one is FP64's (-1)
        const bool good = est0 <= kTolGrad<T> && est1 <= kTolGrad<T> && lo > 0.f;
        const bool again = kDf<T> && lo < kLoWide;
        if (lane == 0) {
          r.flag()[3] = !good ? 0 : again ? -1 : lo >= 0.02f ? kNodesGrad : kNodes;
          r.flag()[4] = __float_as_int(lo);
          r.flag()[6] = lo >= kLoWide ? 1 : kNodesWide / 32;
        }
        __syncwarp();
        if (good && !again) solve_nodes(r, a, K0, K1, X0, X1, t_bytes, gnorm, eg, 0);
      }
      r.V = V0;
      r.o_t -= t_bytes;
    } else if (tid == 0) {
      r.flag()[3] = 1;
      r.flag()[5] = eg - 1023;
      r.flag()[6] = 1;
    }
    if (mat) cholesky(r);
    sync_all<NW, ALL>();
    Q = r.flag()[3];
    lo = __int_as_float(r.flag()[4]);
    passes = r.flag()[6];
    ok = Q != 0 && r.flag()[1] == 0;
    if (ok && Q < 0) return true;
  }
  if (!ok) {
    if (tid == 0) leave(r, a);
    return false;
  }
  if (none) {
    if (a.gbuf) {
      double* gj = a.gbuf + (a.gofs[r.j] - a.gofs[a.j0]);
      for (int e = tid; e < r.m * r.m; e += NT) gj[e] = 0.0;
    }
    return false;
  }
  const Buckets bk = make_buckets(r);
  double* gj = a.gbuf ? a.gbuf + (a.gofs[r.j] - a.gofs[a.j0]) : nullptr;
  for (int pass = 0; pass < passes; ++pass) {
  if (pass > 0) {                                  // the wide rule's next 32 nodes
    if (node) {
      r.V = V1;
      r.o_t += t_bytes;
      solve_nodes(r, a, K0, K1, X0, X1, t_bytes, gnorm, eg, pass);
      r.V = V0;
      r.o_t -= t_bytes;
    }
    sync_all<NW, ALL>();
  }
  const int shift = r.flag()[5];
  // factors of row i at (q mp + i): component 0 (leading) / 2 (trailing) x_q, 1 / 3 y_q; or two
  // doubles x_q, y_q
  if (direct) {
    for (int i = tid; i < r.mp; i += NT) {
      const T x = i < r.m ? scaled(a.grad_out[base + i], eg, (T*)nullptr) : zero<T>();
      if constexpr (kDf<T>) r.AB[i] = make_float4(x.h, i == r.pos ? 0.5f : 0.f, x.l, 0.f);
      else reinterpret_cast<double2*>(r.AB)[i] = make_double2(x, i == r.pos ? 0.5 : 0.0);
    }
  } else if constexpr (!kDf<T>) {
    for (int it = tid; it < 2 * Q * r.mp; it += NT) {   // (process, node, row)
      const int i = it % r.mp, c = it / r.mp, q = c % Q, which = c / Q;   // 0: y, 1: x
      const int K = which ? K1 : K0;
      const double *V = (which ? V1 : V0) + i, *X = (which ? X0 : X1) + q;
      double s = 0.0;
      for (int k = 0; k < K; ++k) s = fma(V[(size_t)k * r.mp], X[(size_t)k * kNodes], s);
      reinterpret_cast<double*>(r.AB)[2 * ((size_t)q * r.mp + i) + (which ? 0 : 1)] = s;
    }
  } else if (mat) {
    float* AB = reinterpret_cast<float*>(r.AB);
    const int nch = (Q + 7) / 8, items = 2 * nch * r.mp;
    for (int it = tid; it < items; it += NM) {      // (process, 8 nodes, row): uniform in a warp
      const int i = it % r.mp, c = it / r.mp, h = c % nch, which = c / nch;   // 0: y, 1: x
      const int K = which ? K1 : K0;
      const T* V = (which ? V1 : V0) + i;
      const float* X = reinterpret_cast<const float*>(which ? X0 : X1) + 8 * h;
      const f2 minus1 = pack(-1.f, -1.f);
      float C[8];
      f2 s[4], cc[4];
      // |sum_k V_k(i) X_k| <= |X_k|, and |X| <= |X_0| (the first component) (lam / lo) scale:
      // bound by the vector's own norm
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        float n2 = 0.f;
        for (int k = 0; k < K; ++k) {
          const float x = X[(size_t)k * 64 + q];
          n2 = fmaf(x, x, n2);
        }
        const int ex = (int)((__float_as_uint(n2) >> 23) & 0xFF) - 127;
        C[q] = 3.f * __int_as_float(min(max(((ex + 2) >> 1) + 1 + 127, 1), 250) << 23);
      }
#pragma unroll
      for (int u = 0; u < 4; ++u) s[u] = pack(C[2 * u], C[2 * u + 1]), cc[u] = 0;
      for (int k = 0; k < K; ++k) {
        const T v = V[(size_t)k * r.mp];
        const f2 vh = pack(v.h, v.h), vl = pack(v.l, v.l);
        const ulonglong2* xh = reinterpret_cast<const ulonglong2*>(X + (size_t)k * 64);
        const ulonglong2* xl = reinterpret_cast<const ulonglong2*>(X + (size_t)k * 64 + 32);
        const ulonglong2 h0 = xh[0], h1 = xh[1], l0 = xl[0], l1 = xl[1];
        madd2(h0.x, l0.x, vh, vl, minus1, s[0], cc[0]);
        madd2(h0.y, l0.y, vh, vl, minus1, s[1], cc[1]);
        madd2(h1.x, l1.x, vh, vl, minus1, s[2], cc[2]);
        madd2(h1.y, l1.y, vh, vl, minus1, s[3], cc[3]);
      }
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        if (8 * h + q >= Q) break;
        const float sv = (q & 1) ? hi32(s[q / 2]) : lo32(s[q / 2]);
        const float cv = (q & 1) ? hi32(cc[q / 2]) : lo32(cc[q / 2]);
        const T x = quick(__fsub_rn(sv, C[q]), cv);
        float* d = AB + 4 * ((size_t)(8 * h + q) * r.mp + i) + (which ? 0 : 1);
        d[0] = x.h;
        d[2] = x.l;
      }
    }
  }
  sync_all<NW, ALL>();
  // G(k, l) over the stored entries of the upper triangle
  for (int k = warp; k < r.m; k += NT / 32) {
    const int e1 = r.ext()[k].y;
    for (int e0 = r.ext()[k].x; e0 < e1; e0 += 32) {
      const int e = e0 + lane;
      int col[1] = {e < e1 ? a.colind[e] : -1}, l[1];
      find_cols<1>(r, bk, col, l);
      if (!__any_sync(0xffffffffu, l[0] >= 0)) continue;
      const int li = l[0] < 0 ? k : l[0];
      double val = 0.0;
      if constexpr (kDf<T>) {
        // a_k b_l and b_k a_l side by side
        float s0 = 0.f, s1 = 0.f, c0 = 0.f;
        for (int q = 0; q < Q; ++q) {
          const float4 x = r.AB[(size_t)q * r.mp + k];
          const float4 y = r.AB[(size_t)q * r.mp + li];
          const float p0 = __fmul_rn(x.x, y.y), p1 = __fmul_rn(x.y, y.x);
          float t = __fadd_rn(__fmaf_rn(x.x, y.y, -p0), __fmaf_rn(x.y, y.x, -p1));
          t = __fmaf_rn(x.x, y.w, t);
          t = __fmaf_rn(x.z, y.y, t);
          t = __fmaf_rn(x.y, y.z, t);
          t = __fmaf_rn(x.w, y.x, t);
          float u, v;
          two_sum(s0, p0, u, v);
          s0 = u;
          t = __fadd_rn(t, v);
          two_sum(s1, p1, u, v);
          s1 = u;
          c0 = __fadd_rn(c0, __fadd_rn(t, v));
        }
        float s, err;
        two_sum(s0, s1, s, err);
        const df g = quick(s, __fadd_rn(err, c0));
        val = widen(g.h, shift) + widen(g.l, shift);
      } else {
        const double2* AB = reinterpret_cast<const double2*>(r.AB);
        for (int q = 0; q < Q; ++q) {
          const double2 x = AB[(size_t)q * r.mp + k], y = AB[(size_t)q * r.mp + li];
          val = fma(x.x, y.y, fma(x.y, y.x, val));
        }
        val = ldexp(val, shift);
      }
      if (l[0] >= 0) {
        if (gj) {
          const double sum = pass > 0 ? gj[(size_t)k * r.m + li] + val : val;
          gj[(size_t)k * r.m + li] = sum;
          gj[(size_t)li * r.m + k] = sum;
        } else {
          atomicAdd(a.out + e, val);
          if (li != k) atomicAdd(a.out + r.start()[li] + a.tpos[e], val);
        }
      }
    }
  }
  sync_all<NW, ALL>();
  }
  if (tid == 0) {
    // products with S and of the Lanczos vectors with the node solutions
    const double done = (double)r.m * (r.m + Q * passes) * (double)(K0 + K1);
    if (kDf<T>) atomicAdd(&a.ctr->products_df, done);
    else atomicAdd(&a.ctr->flops_fp64, 2.0 * done);
  }
  return false;
}

// A double-float row over again in FP64 (the storage of both has 8 bytes an element).
template <int NE, int NW, bool GP, bool ALL>
__device__ __noinline__ void row_gradient_fp64(const Args& a, int j) {
  Row<double, NW, GP, ALL, true> r;
  bind_storage(r, a);
  take_row(r, a, j);
  sync_all<NW, ALL>();                               // the flags of the first attempt have been read
  row_gradient<NE>(r, a);
}

template <int NW, bool GP, bool ALL, int NE, int MINB>
__global__ void __launch_bounds__(threads_of<NW, ALL>(), MINB) bwd_kernel(const __grid_constant__ Args a) {
  Row<df, NW, GP, ALL, true> r;
  bind_storage(r, a);
  load_nodes(r, a);
  for (;;) {
    if (threadIdx.x == 0) {
      r.flag()[2] = atomicAdd(a.queue, 1);
      r.flag()[1] = 0;
    }
    sync_all<NW, ALL>();
    const int idx = r.flag()[2];
    sync_all<NW, ALL>();
    if (idx >= a.n) break;
    const int j = a.order[idx];
    if (a.gbuf && (j < a.j0 || j >= a.j1)) continue;         // another wave's row
    take_row(r, a, j);
    if (row_gradient<NE>(r, a)) row_gradient_fp64<NE, NW, GP, ALL>(a, j);
    sync_all<NW, ALL>();
  }
}

template <int NW, bool GP, bool ALL, int NE, int MINB>
cudaError_t run(const Args& a, int grid, cudaStream_t s) {
  const Layout L = layout(a.nb, a.ns, NW, !GP, true);
  if (((ALL || NW == 1) && a.ns < nblocks(a.nb)) || L.total > kMaxSmem) return cudaErrorInvalidValue;
  bwd_kernel<NW, GP, ALL, NE, MINB><<<grid, threads_of<NW, ALL>(), L.total, s>>>(a);
  return cudaGetLastError();
}
template <int NW, bool GP, bool ALL, int NE, int MINB>
cudaError_t attr() {
  return cudaFuncSetAttribute(bwd_kernel<NW, GP, ALL, NE, MINB>,
                              cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxSmem);
}

}  // namespace

cudaError_t launch_bwd(const Args& a, const Class& c, int grid, cudaStream_t s) {
  switch (c.nw) {
    case 1: return c.lone ? run<1, false, false, 1, 8>(a, grid, s) : run<1, false, true, 1, 8>(a, grid, s);
    case 3: return run<3, false, true, 1, 4>(a, grid, s);
    case 5: return run<5, false, true, 1, 2>(a, grid, s);
  }
  if (c.nb <= 6) return run<15, false, true, 1, 1>(a, grid, s);
  return c.part_smem ? run<15, false, false, 1, 1>(a, grid, s) : run<15, true, false, 4, 1>(a, grid, s);
}

cudaError_t set_attr_bwd() {
  cudaError_t e;
  if ((e = attr<1, false, true, 1, 8>()) != cudaSuccess) return e;
  if ((e = attr<1, false, false, 1, 8>()) != cudaSuccess) return e;
  if ((e = attr<3, false, true, 1, 4>()) != cudaSuccess) return e;
  if ((e = attr<5, false, true, 1, 2>()) != cudaSuccess) return e;
  if ((e = attr<15, false, true, 1, 1>()) != cudaSuccess) return e;
  if ((e = attr<15, false, false, 1, 1>()) != cudaSuccess) return e;
  return attr<15, true, false, 4, 1>();
}

}  // namespace kry
}  // namespace submat
