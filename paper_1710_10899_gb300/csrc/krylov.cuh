// One column of a root of a symmetric positive definite submatrix by a Krylov method
// (internal header; kernels in krylov_fwd.cuh and krylov_bwd.cu).
//
// The method keeps one column of F = f(S), f(x) = x^(-1/p) or x^(1/p).  From the Lanczos
// recurrence S V = V T + beta v e^T started at e_pos (or at a cotangent), f(S) e_pos is
// V f(T) e_1, which takes k products with S (O(k m^2)) instead of the O(m^3) products of an
// iteration on the whole matrix; k is 15..45 for submatrices of condition 10..60.  Without
// reorthogonalisation the recurrence in finite precision still gives f(S) e_pos to the
// working precision, some steps later (Druskin & Knizhnerman 1991).
//
// f(T) e_1: x^(-a), 0 < a < 1, as a sum of simple fractions, x^(-a) = sin(pi a)/pi times
// the integral of t^(-a) / (x + t) over t > 0, with t = tau (1-s)/(1+s) and the Gauss-Jacobi
// rule of kNodes nodes for the weight (1-s)^(-a) (1+s)^(a-1): the error falls by
// ((r^(1/4) + 1) / (r^(1/4) - 1))^2 per node, r^(1/2) the ratio between tau and the ends of the
// spectrum: below 1e-16 over [lam / 100, lam] with tau = lam / 10, and with kNodesWide nodes and
// tau at the geometric mean over [lam / kKappa, lam].  So f(T) e_1 is a sum of
// tridiagonal solves, one per lane of a warp.  x^(-1) is the node t = 0; x^(1/p) is x times
// x^(-(1-1/p)).
//
// Stopping: the residual of (S + t) x = e_pos after k steps is beta_k |e_k^T (T + t)^(-1) e_1|,
// from a two-term recurrence per node, so the error bound sum_q w_q resid_q / (lo + t_q) is known
// at every step (lo: the smallest Ritz value's bracket); lam / kKappa is certified as a lower
// bound of the whole spectrum at the end by an FP32 Cholesky factorisation of
// S - lam / kKappa I (a Krylov space from e_pos alone need not see every eigenvalue: a submatrix that is
// not positive definite in a part that e_pos does not reach has to be found all the same).
// A row whose factorisation or bound fails is left to the coupled iteration.
//
// Storage: S's upper block triangle in 32 x 32 blocks, an element a double-float (FP32 pair)
// or a double (8 bytes either way), the elements of a lane's 4 x 8 tile 16 bytes apart in
// pairs so that a warp reads a block with 16 conflict-free 16-byte loads; the first blocks in
// shared memory, the rest (if any) in global scratch.  Every element is read once per product
// and used twice (S_ij v_j and S_ij v_i).
//
// Double-float products: acc s starts at C, larger than any partial sum (|sum| <= the row's
// 2-norm as |v| = 1), so s' = fma(a, b, s), z = s' - s and fma(a, b, -z) split a product into
// a part on s's grid, summed exactly, and an exact remainder: 6 FP32 operations for a product
// of two double-floats and its addition, with an absolute error near 2^-45 of the row's norm.
//
// Why: the coupled iteration spends p m^3 products (ten FP16 slice products each on the mixed
// path, FP64 at 2 FMA per clock and SM on the FP64 path) per step for a matrix of which one
// column is kept.  Measured on GB300, whole forward, coupled -> Krylov: FP64 n = 2048, orders
// 28..239, 301 -> 6.4 ms (bound: the FP64 pipe, 30 products of m^2 a row); FP64 n = 2000,
// orders 1..28, 11.6 -> 0.26 ms; double-float n = 8192, orders 19..119, 11.1 -> 2.6 ms and
// n = 9973, orders 25..169, 23.0 -> 4.7 ms.  By the counters (classes of 64 to 250): FP64 keeps its
// pipe 60..82 % busy; double-float issues in 27..43 % of the slots (adjoint 33..50 %) and waits at
// the step's two barriers first.
//
// Wide spectra.  Double-float errors grow as kappa 2^-45, so rows beyond lam / 100 are FP64's where
// the coupled iteration and the Jacobi adjoint gave them that accuracy: the kernel repeats such a
// row with its FP64 instance.  7200 rows of order 24 / 1800 of order 150 at kappa = 300, forward
// p = 2: 45 / 1929 ms (fallback), 0.39 / 1.26 (double-float, 2e-12..1e-11 off), 1.37 / 5.4 (2e-14);
// adjoint 19 / 217 ms (Jacobi), 1.8 / 4.4 (double-float, up to 1e-10 off), 5.0 / 17.2 (1e-14..1e-13).
#pragma once
#include "common.cuh"
#include "scaled_step.cuh"

namespace submat {
namespace kry {

constexpr int kB = 32;                     // block edge
constexpr int kBlkBytes = kB * kB * 8;
constexpr int kBuckets = 256;              // column buckets of the gather
constexpr int kNodes = 32;                 // quadrature nodes (one per lane)
constexpr int kNodesWide = 64;             // nodes for spectra wider than [lam / 100, lam]
constexpr int kNodesGrad = 20;             // nodes of the adjoint for spectra within [lam / 50, lam]
constexpr int kNodesAll = kNodes + kNodesWide + kNodesGrad;
constexpr float kKappa = 2000.f;           // largest lam / lambda_min taken here
constexpr float kTau = 0.1f;               // tau / lam for spectra in [lam / 100, lam]
constexpr float kLoWide = 0.01f;            // lo / lam from which kNodes nodes do
constexpr float kSturm = 0.36f;            // log2 spacing of the Sturm shifts (31 of them: 2^-11.2)

__host__ __device__ constexpr int cap_of(int nw) { return nw == 1 ? 64 : 128; }
__host__ __device__ inline int nblocks(int nb) { return nb * (nb + 1) / 2; }

// Quadrature of one exponent a: nodes theta = (1-s)/(1+s), weights omega 2/(1+s) (sum of omega
// 1), so x^(-a) = tau^(-a) sum_q w_q tau / (x + tau theta_q).
struct Nodes {
  double theta[kNodesAll], w[kNodesAll];   // the rules of kNodes, kNodesWide and kNodesGrad nodes
};

// One size class: a persistent launch over rows of order <= 32 nb.
struct Args {
  const int32_t* rowptr;
  const int32_t* colind;
  const int32_t* m;
  const int32_t* pos;
  const int32_t* order;                    // rows of this launch
  int32_t n;
  int32_t p, sign;
  const double* vals;
  double* out;                             // forward: vals_out; backward: grad_in
  DevCounters* ctr;
  int32_t* queue;
  int32_t *redo_list, *redo_small;         // rows left to the general path; of order <= small_max
  int32_t small_max;
  const int32_t* nonfinite;                // nonzero: some value is infinite or NaN
  char* scratch;
  size_t stride;                           // bytes per CTA
  int32_t nb;                              // blocks per edge of the class
  int32_t ns;                              // blocks of S held in shared memory
  double resid_tol;
  float kappa_max;
  int32_t fp64;                            // every row in FP64 (else double-float first)
  Nodes nodes;
  // backward
  const double* grad_out;
  const int32_t* tpos;
  double* gbuf;
  const int64_t* gofs;
  int32_t j0, j1;
};

// Shared-memory and scratch layout (bytes), host and device.  What a kernel instance needs is
// sized for its largest order, so that the offsets are constants of the code (kept in
// registers they cost ten of them); S's blocks follow, then the partial sums.
struct Fixed {
  int t_bytes;                             // one Lanczos process's share of al and be
  int al, be, coef, red, nodes, bk, v, ext, R, start, blocks;
};
// Largest order of an instance in blocks: by its warps, or for kBigWarps by where S and the
// partial sums lie.
constexpr int kBigWarps = 15;
__host__ __device__ constexpr int nb_cap(int nw, bool part_smem, bool all) {
  return nw == 1 ? 1 : nw == 3 ? 3 : nw == 5 ? 4 : all ? 6 : part_smem ? 15 : SUBMAT_MAX_M / kB;
}
__host__ __device__ constexpr int up16(int b) { return (b + 15) / 16 * 16; }
__host__ __device__ constexpr Fixed fixed(int nw, int nb, bool bwd) {
  const int mp = nb * kB, cap = cap_of(nw), proc = bwd ? 2 : 1;
  Fixed f{};
  f.t_bytes = up16((cap + 1) * 8);
  f.al = 0;
  f.be = f.al + proc * f.t_bytes;
  f.coef = f.be + proc * f.t_bytes;
  f.red = f.coef + up16((cap + 2) * 8);
  f.nodes = f.red + 32 * 8 + 64;           // two sums of 16 warps, then flags
  f.bk = f.nodes + 2 * kNodesAll * 8;
  f.v = f.bk + up16((kBuckets + 2) * 2);
  f.ext = f.v + mp * 8;
  f.R = f.ext + mp * 8;
  f.start = f.R + mp * 4;
  f.blocks = f.start + (bwd ? mp * 4 : 0);
  return f;
}
struct Layout {
  size_t part, total;
  size_t g_blocks, g_v, g_x, g_part, g_ab, g_total;
  size_t v_bytes, x_bytes;                 // one process's share of g_v and g_x
};
__host__ __device__ inline Layout layout(int nb, int ns, int nw, bool part_smem, bool bwd) {
  Layout L{};
  const size_t mp = (size_t)nb * kB, cap = cap_of(nw);
  const bool all = nw != kBigWarps || nb <= 6;
  const size_t proc = bwd ? 2 : 1;         // Lanczos processes (the adjoint runs two)
  L.v_bytes = (cap + 2) * mp * 8;
  L.x_bytes = (cap + 1) * (size_t)kNodes * 8;
  // the adjoint's factors take S's place when all of S lies in shared memory
  const size_t ab = bwd && all ? (size_t)kNodes * mp * 16 : 0;
  const size_t blocks = (size_t)ns * kBlkBytes;
  L.part = fixed(nw, nb_cap(nw, part_smem, all), bwd).blocks + (blocks > ab ? blocks : ab);
  L.total = L.part + (part_smem ? (size_t)nb * mp * 8 : 0);
  size_t o = 0;
  auto take = [&](size_t b) { const size_t at = o; o += (b + 15) / 16 * 16; return at; };
  L.g_blocks = take((size_t)(nblocks(nb) - ns) * kBlkBytes);
  L.g_v = take(proc * L.v_bytes);
  L.g_x = take(proc * L.x_bytes);
  L.g_part = take(part_smem ? 0 : (size_t)nb * mp * 8);
  L.g_ab = take(bwd && !ab ? (size_t)kNodes * mp * 16 : 0);
  L.g_total = (o + 1023) / 1024 * 1024;
  return L;
}

// Host side: quadrature tables, size classes and launchers.
bool cached_nodes(int p, int sign, Nodes* out);
struct Class {
  int max_m = 0, nw = 0, nb = 0, ns = 0, ctas = 0;
  bool part_smem = true, lone = false;     // lone: one warp in both roles
};
int class_of(int m);                       // class index of a row of order m
Class make_class(int index, int m_max, int rows, int n_sm, bool bwd);
cudaError_t launch_fwd(const Args& a, const Class& c, int grid, cudaStream_t s);
cudaError_t launch_bwd(const Args& a, const Class& c, int grid, cudaStream_t s);
cudaError_t set_attr_fwd(int p, int sign, bool fp64);
cudaError_t set_attr_bwd();
// the forward's instances (krylov_fwd.cuh)
cudaError_t launch_roots_df(const Args& a, const Class& c, int grid, cudaStream_t s);
cudaError_t launch_roots_fp64(const Args& a, const Class& c, int grid, cudaStream_t s);
cudaError_t launch_inverse_df(const Args& a, const Class& c, int grid, cudaStream_t s);
cudaError_t launch_inverse_fp64(const Args& a, const Class& c, int grid, cudaStream_t s);
cudaError_t set_attr_roots_df();
cudaError_t set_attr_roots_fp64();
cudaError_t set_attr_inverse_df();
cudaError_t set_attr_inverse_fp64();

}  // namespace kry
}  // namespace submat

#ifdef __CUDACC__
namespace submat {
namespace kry {

// ---- scalars: double-float (df) and double ---------------------------------------------
struct __align__(8) df {
  float h, l;
};
__device__ __forceinline__ void two_sum(float a, float b, float& s, float& e) {
  s = __fadd_rn(a, b);
  const float bb = __fsub_rn(s, a);
  e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
}
__device__ __forceinline__ df quick(float s, float e) {
  const float h = __fadd_rn(s, e);
  return df{h, __fsub_rn(e, __fsub_rn(h, s))};
}
__device__ __forceinline__ df add(df a, df b) {
  float s, e;
  two_sum(a.h, b.h, s, e);
  return quick(s, __fadd_rn(e, __fadd_rn(a.l, b.l)));
}
__device__ __forceinline__ df neg(df a) { return df{-a.h, -a.l}; }
__device__ __forceinline__ df sub(df a, df b) { return add(a, neg(b)); }
__device__ __forceinline__ df mul(df a, df b) {
  const float p = __fmul_rn(a.h, b.h);
  float e = __fmaf_rn(a.h, b.h, -p);
  e = __fmaf_rn(a.h, b.l, e);
  e = __fmaf_rn(a.l, b.h, e);
  return quick(p, e);
}
__device__ __forceinline__ df rcp(df d) {
  const float r = __frcp_rn(d.h);
  const float e = __fmaf_rn(-d.l, r, __fmaf_rn(-d.h, r, 1.f));
  return quick(r, __fmul_rn(r, e));
}
__device__ __forceinline__ df inv_sqrt(df a) {
  const float r = rsqrtf(a.h);
  const df q = mul(mul(a, df{r, 0.f}), df{r, 0.f});       // a r^2, near 1
  const float e = __fsub_rn(__fsub_rn(1.f, q.h), q.l);
  return quick(r, r * e * fmaf(0.375f, e, 0.5f));
}
__device__ __forceinline__ df shfl_xor(df a, int o) {
  return df{__shfl_xor_sync(0xffffffffu, a.h, o), __shfl_xor_sync(0xffffffffu, a.l, o)};
}
__device__ __forceinline__ float hi(df a) { return a.h; }
__device__ __forceinline__ double join(df a) { return (double)a.h + (double)a.l; }
__device__ __forceinline__ df as(float x, df*) { return df{x, 0.f}; }
__device__ __forceinline__ df as(double x, df*) {
  const float h = (float)x;
  return df{h, (float)(x - (double)h)};
}

__device__ __forceinline__ double add(double a, double b) { return a + b; }
__device__ __forceinline__ double sub(double a, double b) { return a - b; }
__device__ __forceinline__ double neg(double a) { return -a; }
__device__ __forceinline__ double mul(double a, double b) { return a * b; }
__device__ __forceinline__ double rcp(double a) { return 1.0 / a; }
__device__ __forceinline__ double inv_sqrt(double a) { return rsqrt(a); }
__device__ __forceinline__ double shfl_xor(double a, int o) {
  return __shfl_xor_sync(0xffffffffu, a, o);
}
__device__ __forceinline__ float hi(double a) { return (float)a; }
__device__ __forceinline__ double join(double a) { return a; }
__device__ __forceinline__ double as(float x, double*) { return (double)x; }
__device__ __forceinline__ double as(double x, double*) { return x; }

// Single precision: the correction of a refined column.
__device__ __forceinline__ float add(float a, float b) { return a + b; }
__device__ __forceinline__ float sub(float a, float b) { return a - b; }
__device__ __forceinline__ float neg(float a) { return -a; }
__device__ __forceinline__ float mul(float a, float b) { return a * b; }
__device__ __forceinline__ float rcp(float a) { return __frcp_rn(a); }
__device__ __forceinline__ float inv_sqrt(float a) { return rsqrtf(a); }
__device__ __forceinline__ float shfl_xor(float a, int o) { return __shfl_xor_sync(0xffffffffu, a, o); }
__device__ __forceinline__ float hi(float a) { return a; }
__device__ __forceinline__ double join(float a) { return (double)a; }
__device__ __forceinline__ float as(float x, float*) { return x; }
__device__ __forceinline__ float as(double x, float*) { return (float)x; }

template <class T> constexpr bool kDf = false;
template <> constexpr bool kDf<df> = true;

template <class T> __device__ __forceinline__ T zero() { return as(0.f, (T*)nullptr); }
template <class T> __device__ __forceinline__ T one() { return as(1.f, (T*)nullptr); }

// v 2^-E (E = e0 - 1023, e0 the exponent field of the largest diagonal entry) by integer
// operations (the FP64 pipe has 2 lanes); results below the normal range become 0, Inf and NaN
// become NaN.
__device__ __forceinline__ double scaled(double v, int e0, double*) {
  const int h = __double2hiint(v), ex = (h >> 20) & 0x7FF;
  if (ex == 0x7FF) return __longlong_as_double(0x7ff8000000000000ll);
  const int ne = ex - e0 + 1023;
  if (ex == 0 || ne <= 0) return 0.0;
  if (ne >= 0x7FF) return __longlong_as_double(0x7ff8000000000000ll);
  return __hiloint2double((h & ~0x7FF00000) | (ne << 20), __double2loint(v));
}
__device__ __forceinline__ df scaled(double v, int e0, df*) {
  const int h = __double2hiint(v), ex = (h >> 20) & 0x7FF;
  if (ex == 0x7FF) return df{__int_as_float(0x7FC00000), 0.f};
  const int ne = ex - e0 + 127;                      // FP32 exponent field of the leading part
  if (ex == 0 || ne <= 60) return df{0.f, 0.f};      // below 2^-66 of the largest diagonal entry
  if (ne >= 0xFF) return df{__int_as_float(0x7FC00000), 0.f};
  const unsigned lo = (unsigned)__double2loint(v);
  const unsigned sgn = (unsigned)h & 0x80000000u;
  const float fh = __uint_as_float(sgn | ((unsigned)ne << 23) | (((unsigned)h & 0xFFFFFu) << 3) |
                                   (lo >> 29));
  const float sc = __uint_as_float(sgn | ((unsigned)(ne - 52) << 23));     // 2^(ne - 127 - 52)
  return df{fh, (float)(lo & 0x1FFFFFFFu) * sc};
}

// ---- barriers ---------------------------------------------------------------------------
// One matrix warp comes in two forms: with a node warp beside it (lower latency of a row), or, as
// ALL = false, alone with both roles (more rows per SM).
template <int NW, bool ALL> constexpr bool kLone = NW == 1 && !ALL;
template <int NW, bool ALL> __device__ __forceinline__ void sync_all() {
  if constexpr (kLone<NW, ALL>) __syncwarp(); else __syncthreads();
}
template <int NW> __device__ __forceinline__ void sync_mat() {   // the NW matrix warps only
  if constexpr (NW == 1) __syncwarp();
  else asm volatile("bar.sync 1, %0;" ::"n"(NW * 32) : "memory");
}
template <int NW, bool ALL> __host__ __device__ constexpr int threads_of() {
  return NW * 32 + (NW == 1 && !ALL ? 0 : 32);
}

// Sum over a warp (every lane gets it); double-floats as unnormalised pairs between levels.
__device__ __forceinline__ df warp_total(df a) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const df b = shfl_xor(a, o);
    float s, e;
    two_sum(a.h, b.h, s, e);
    a = df{s, __fadd_rn(e, __fadd_rn(a.l, b.l))};
  }
  return a;
}
__device__ __forceinline__ double warp_total(double a) { return warp_sum(a); }
__device__ __forceinline__ float warp_total(float a) { return warp_sum_f(a); }

// Sum of the first n warps' totals in red, the same on every thread (lane w reads warp w's).
template <int NW, class T> __device__ __forceinline__ T total_of(const T* red, int lane, int n) {
  if constexpr (NW == 1) {
    return red[0];
  } else {
    constexpr int P2 = NW <= 4 ? 4 : (NW <= 8 ? 8 : 16);
    const int w = lane & (P2 - 1);
    T a = w < n ? red[w] : zero<T>();
#pragma unroll
    for (int o = P2 / 2; o > 0; o >>= 1) a = add(a, shfl_xor(a, o));
    return a;
  }
}

// ---- products with one block --------------------------------------------------------------
// lane (a, b) = (lane / 4, lane % 4) holds rows 4a..4a+3 and columns 8b..8b+7 of a block.
__device__ __forceinline__ int pair_at(int r, int c) {       // 16-byte unit of a block's element
  return ((r & 3) * 4 + ((c & 7) >> 1)) * 32 + (r >> 2) * 4 + (c >> 3);
}
// A pair of neighbouring columns: two doubles, or (h0, h1, l0, l1) for packed FP32 operations.
__device__ __forceinline__ void put(float4* blk, int r, int c, double x) {
  reinterpret_cast<double*>(blk + pair_at(r, c))[c & 1] = x;
}
__device__ __forceinline__ void put(float4* blk, int r, int c, df x) {
  float* u = reinterpret_cast<float*>(blk + pair_at(r, c)) + (c & 1);
  u[0] = x.h;
  u[2] = x.l;
}

// Sums rs[4] over the 4 lanes of a row group and cs[8] over the 8 lanes of a column group; the
// lane's row sum is row `lane` of the block, its column sum column 8b + a.
template <class S> __device__ __forceinline__ S lane_rows(S* rs, int lane) {
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    const S keep = (lane & 2) ? rs[i + 2] : rs[i], send = (lane & 2) ? rs[i] : rs[i + 2];
    rs[i] = keep + __shfl_xor_sync(0xffffffffu, send, 2);
  }
  const S keep = (lane & 1) ? rs[1] : rs[0], send = (lane & 1) ? rs[0] : rs[1];
  return keep + __shfl_xor_sync(0xffffffffu, send, 1);
}
template <class S> __device__ __forceinline__ S lane_cols(S* cs, int lane) {
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const S keep = (lane & 16) ? cs[i + 4] : cs[i], send = (lane & 16) ? cs[i] : cs[i + 4];
    cs[i] = keep + __shfl_xor_sync(0xffffffffu, send, 16);
  }
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    const S keep = (lane & 8) ? cs[i + 2] : cs[i], send = (lane & 8) ? cs[i] : cs[i + 2];
    cs[i] = keep + __shfl_xor_sync(0xffffffffu, send, 8);
  }
  const S keep = (lane & 4) ? cs[1] : cs[0], send = (lane & 4) ? cs[0] : cs[1];
  return keep + __shfl_xor_sync(0xffffffffu, send, 4);
}

// Packed FP32: two operations on neighbouring columns per instruction.
typedef unsigned long long f2;
__device__ __forceinline__ f2 fma2(f2 a, f2 b, f2 c) {
  f2 d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
__device__ __forceinline__ f2 add2(f2 a, f2 b) {
  f2 d;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ f2 pack(float x, float y) {
  return ((f2)__float_as_uint(y) << 32) | __float_as_uint(x);
}
__device__ __forceinline__ float lo32(f2 a) { return __uint_as_float((unsigned)a); }
__device__ __forceinline__ float hi32(f2 a) { return __uint_as_float((unsigned)(a >> 32)); }

__device__ __forceinline__ void madd2(f2 sh, f2 sl, f2 vh, f2 vl, f2 minus1, f2& s, f2& c) {
  const f2 s1 = fma2(sh, vh, s);
  const f2 nz = fma2(s1, minus1, s);                 // s - s1, exact
  f2 t = fma2(sh, vh, nz);                           // exact; the small terms meet before c
  t = fma2(sl, vh, t);
  t = fma2(sh, vl, t);
  c = add2(c, t);
  s = s1;
}

// part[J][32 I + r] = (S_IJ v_J)_r and, off the diagonal, part[I][32 J + c] = (S_IJ^T v_I)_c.
// dot += the block's (and its mirror image's) share of v^T S v in row `lane`.  A double-float
// vector is held as mp leading parts followed by mp trailing parts.
template <bool OFF>
__device__ __forceinline__ void block_mul(const float4* blk, const df* v, int I, int J, float C,
                                          df* part, int mp, int lane, df& dot) {
  const int a = lane >> 2, b = lane & 3;
  const float* vh = reinterpret_cast<const float*>(v);
  const float* vl = vh + mp;
  const ulonglong2* ch = reinterpret_cast<const ulonglong2*>(vh + J * kB + b * 8);
  const ulonglong2* cl = reinterpret_cast<const ulonglong2*>(vl + J * kB + b * 8);
  const ulonglong2 h0 = ch[0], h1 = ch[1], l0 = cl[0], l1 = cl[1];
  const f2 vch[4] = {h0.x, h0.y, h1.x, h1.y}, vcl[4] = {l0.x, l0.y, l1.x, l1.y};
  const f2 minus1 = pack(-1.f, -1.f), C2 = pack(C, C);
  f2 rs[4], rc[4], cs[4], cc[4], vrh[4], vrl[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) rs[i] = cs[i] = C2, rc[i] = cc[i] = 0;
  if (OFF) {
    const float4 xh = *reinterpret_cast<const float4*>(vh + I * kB + a * 4);
    const float4 xl = *reinterpret_cast<const float4*>(vl + I * kB + a * 4);
    vrh[0] = pack(xh.x, xh.x), vrh[1] = pack(xh.y, xh.y), vrh[2] = pack(xh.z, xh.z), vrh[3] = pack(xh.w, xh.w);
    vrl[0] = pack(xl.x, xl.x), vrl[1] = pack(xl.y, xl.y), vrl[2] = pack(xl.z, xl.z), vrl[3] = pack(xl.w, xl.w);
  }
  const ulonglong2* e = reinterpret_cast<const ulonglong2*>(blk) + lane;
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    ulonglong2 x[4];                                 // a column pair's four rows
#pragma unroll
    for (int i = 0; i < 4; ++i) x[i] = e[(i * 4 + j) * 32];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      madd2(x[i].x, x[i].y, vch[j], vcl[j], minus1, rs[i], rc[i]);
      if (OFF) madd2(x[i].x, x[i].y, vrh[i], vrl[i], minus1, cs[j], cc[j]);
    }
  }
  float s4[4], c4[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {                      // grid parts add exactly
    s4[i] = __fadd_rn(__fsub_rn(lo32(rs[i]), C), __fsub_rn(hi32(rs[i]), C));
    c4[i] = __fadd_rn(lo32(rc[i]), hi32(rc[i]));
  }
  const float s = lane_rows(s4, lane), c = lane_rows(c4, lane);
  part[J * mp + I * kB + lane] = df{s, c};
  const float f = OFF ? 2.f : 1.f;
  dot = add(dot, mul(quick(f * s, f * c), df{vh[I * kB + lane], vl[I * kB + lane]}));
  if (OFF) {
    float s8[8], c8[8];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      s8[2 * j] = __fsub_rn(lo32(cs[j]), C);
      s8[2 * j + 1] = __fsub_rn(hi32(cs[j]), C);
      c8[2 * j] = lo32(cc[j]);
      c8[2 * j + 1] = hi32(cc[j]);
    }
    const float t = lane_cols(s8, lane), u = lane_cols(c8, lane);
    part[I * mp + J * kB + b * 8 + a] = df{t, u};
  }
}
template <bool OFF>
__device__ __forceinline__ void block_mul(const float4* blk4, const double* v, int I,
                                          int J, float, double* part, int mp, int lane, double& dot) {
  const int a = lane >> 2, b = lane & 3;
  const double2* blk = reinterpret_cast<const double2*>(blk4);
  double vr[4], vc[8], rs[4], cs[8];
#pragma unroll
  for (int i = 0; i < 4; ++i) vr[i] = v[I * kB + a * 4 + i], rs[i] = 0.0;
#pragma unroll
  for (int i = 0; i < 8; ++i) vc[i] = v[J * kB + b * 8 + i], cs[i] = 0.0;
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const double2 x = blk[(i * 4 + j) * 32 + lane];
      rs[i] = fma(x.x, vc[2 * j], rs[i]);
      rs[i] = fma(x.y, vc[2 * j + 1], rs[i]);
      if (OFF) {
        cs[2 * j] = fma(x.x, vr[i], cs[2 * j]);
        cs[2 * j + 1] = fma(x.y, vr[i], cs[2 * j + 1]);
      }
    }
  const double s = lane_rows(rs, lane);
  part[J * mp + I * kB + lane] = s;
  dot = fma(OFF ? 2.0 * s : s, v[I * kB + lane], dot);
  if (OFF) {
    const double t = lane_cols(cs, lane);
    part[I * mp + J * kB + b * 8 + a] = t;
  }
}

// Single precision, from the leading parts of a double-float block.
template <bool OFF>
__device__ __forceinline__ void block_mul(const float4* blk, const float* v, int I, int J, float, float* part,
                                          int mp, int lane, float& dot) {
  const int a = lane >> 2, b = lane & 3;
  const ulonglong2* ch = reinterpret_cast<const ulonglong2*>(v + J * kB + b * 8);
  const ulonglong2 h0 = ch[0], h1 = ch[1];
  const f2 vc[4] = {h0.x, h0.y, h1.x, h1.y};
  f2 rs[4] = {}, cs[4] = {}, vr[4];
  const float4 xr = *reinterpret_cast<const float4*>(v + I * kB + a * 4);
  vr[0] = pack(xr.x, xr.x), vr[1] = pack(xr.y, xr.y), vr[2] = pack(xr.z, xr.z), vr[3] = pack(xr.w, xr.w);
  const ulonglong2* e = reinterpret_cast<const ulonglong2*>(blk) + lane;
#pragma unroll
  for (int j = 0; j < 4; ++j)
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const f2 x = e[(i * 4 + j) * 32].x;
      rs[i] = fma2(x, vc[j], rs[i]);
      if (OFF) cs[j] = fma2(x, vr[i], cs[j]);
    }
  float s4[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) s4[i] = lo32(rs[i]) + hi32(rs[i]);
  const float s = lane_rows(s4, lane);
  part[J * mp + I * kB + lane] = s;
  dot = fmaf(OFF ? 2.f * s : s, v[I * kB + lane], dot);
  if (OFF) {
    float s8[8];
#pragma unroll
    for (int j = 0; j < 4; ++j) s8[2 * j] = lo32(cs[j]), s8[2 * j + 1] = hi32(cs[j]);
    const float t = lane_cols(s8, lane);
    part[I * mp + J * kB + b * 8 + a] = t;
  }
}

__device__ __forceinline__ void elem_hi(const float4& x, float& a, float& b, df*) { a = x.x; b = x.y; }
__device__ __forceinline__ void elem_hi(const float4& x, float& a, float& b, double*) {
  const double2 d = *reinterpret_cast<const double2*>(&x);
  a = (float)d.x;
  b = (float)d.y;
}

// As block_mul with |S| 1 and S^2 1 in FP32 (row sums and squared row norms).
template <class T>
__device__ __forceinline__ void block_stats(const float4* blk, int I, int J,
                                            float2* part, int mp, int lane) {
  const int a = lane >> 2, b = lane & 3;
  float rs[4] = {}, rc[4] = {}, cs[8] = {}, cc[8] = {};
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      float x, y;
      elem_hi(blk[(i * 4 + j) * 32 + lane], x, y, (T*)nullptr);
      rs[i] += fabsf(x) + fabsf(y);
      rc[i] = fmaf(x, x, fmaf(y, y, rc[i]));
      cs[2 * j] += fabsf(x);
      cs[2 * j + 1] += fabsf(y);
      cc[2 * j] = fmaf(x, x, cc[2 * j]);
      cc[2 * j + 1] = fmaf(y, y, cc[2 * j + 1]);
    }
  const float s = lane_rows(rs, lane), c = lane_rows(rc, lane);
  part[J * mp + I * kB + lane] = make_float2(s, c);
  if (I != J) {
    const float t = lane_cols(cs, lane), u = lane_cols(cc, lane);
    part[I * mp + J * kB + b * 8 + a] = make_float2(t, u);
  }
}

// ---- one row's working set ---------------------------------------------------------------
// Shared memory is addressed by byte offsets from the dynamic array itself, so that the
// accesses compile to shared-memory instructions with 32-bit addresses; pointers kept in a
// struct become generic ones (a block's product measured 1.9x slower).
extern __shared__ __align__(16) unsigned char kry_smem[];

// GP: partial sums in scratch instead of shared memory; ALL: every block in shared memory
template <class T, int NW, bool GP, bool ALL, bool BWD>
struct Row {
  static constexpr int kNb = nb_cap(NW, !GP, ALL);
  static constexpr Fixed kF = fixed(NW, kNb, BWD);
  int m, nb, mp, ns, pos, j;
  int o_part, o_t;              // partial sums; current Lanczos process in al and be
  float4* gblk;                 // blocks t >= ns, in scratch
  T* gpart;                     // partial sums (GP)
  T *V, *X;                     // scratch: Lanczos vectors [k][mp], node solutions [k][32]
  float4* AB;                   // adjoint: factors (a, b) per node and row
  int e0;                       // exponent field of the largest diagonal entry
  float lam, C, sigma;          // of the scaled submatrix: Gershgorin bound, accumulator start,
                                // certified lower end
  __device__ __forceinline__ T* v() const { return reinterpret_cast<T*>(kry_smem + kF.v); }
  __device__ __forceinline__ T v_at(int i) const {
    if constexpr (!kDf<T>) {
      return v()[i];
    } else {
      const float* h = reinterpret_cast<const float*>(kry_smem + kF.v);
      return df{h[i], h[mp + i]};
    }
  }
  __device__ __forceinline__ void set_v(int i, T x) const {
    if constexpr (!kDf<T>) {
      v()[i] = x;
    } else {
      float* h = reinterpret_cast<float*>(kry_smem + kF.v);
      h[i] = x.h;
      h[mp + i] = x.l;
    }
  }
  // node solution k of node q (a double-float row: 32 leading, then 32 trailing parts)
  __device__ __forceinline__ T x_at(int k, int q) const {
    if constexpr (!kDf<T>) {
      return X[(size_t)k * kNodes + q];
    } else {
      const float* h = reinterpret_cast<const float*>(X + (size_t)k * kNodes);
      return df{h[q], h[kNodes + q]};
    }
  }
  __device__ __forceinline__ void set_x(int k, int q, T x) const {
    if constexpr (!kDf<T>) {
      X[(size_t)k * kNodes + q] = x;
    } else {
      float* h = reinterpret_cast<float*>(X + (size_t)k * kNodes);
      h[q] = x.h;
      h[kNodes + q] = x.l;
    }
  }
  __device__ __forceinline__ T* part() const {
    if constexpr (GP) return gpart; else return reinterpret_cast<T*>(kry_smem + o_part);
  }
  __device__ __forceinline__ T* al() const { return reinterpret_cast<T*>(kry_smem + kF.al + o_t); }
  __device__ __forceinline__ T* be() const { return reinterpret_cast<T*>(kry_smem + kF.be + o_t); }
  __device__ __forceinline__ T* coef() const { return reinterpret_cast<T*>(kry_smem + kF.coef); }
  __device__ __forceinline__ T* red() const { return reinterpret_cast<T*>(kry_smem + kF.red); }
  __device__ __forceinline__ int* flag() const { return reinterpret_cast<int*>(kry_smem + kF.red + 256); }
  __device__ __forceinline__ double* nodes() const { return reinterpret_cast<double*>(kry_smem + kF.nodes); }
  __device__ __forceinline__ int2* ext() const { return reinterpret_cast<int2*>(kry_smem + kF.ext); }
  __device__ __forceinline__ int32_t* R() const { return reinterpret_cast<int32_t*>(kry_smem + kF.R); }
  // first position of each column bucket (kBuckets + 1 entries)
  __device__ __forceinline__ uint16_t* bk() const { return reinterpret_cast<uint16_t*>(kry_smem + kF.bk); }
  __device__ __forceinline__ int32_t* start() const { return reinterpret_cast<int32_t*>(kry_smem + kF.start); }
  __device__ __forceinline__ float4* sblk() const { return reinterpret_cast<float4*>(kry_smem + kF.blocks); }
  __device__ __forceinline__ float4* sblk(int t) const { return sblk() + t * (kBlkBytes / 16); }
  __device__ __forceinline__ float4* gblk_at(int t) const { return gblk + (size_t)(t - ns) * (kBlkBytes / 16); }
  __device__ __forceinline__ float4* blk(int t) const {
    if constexpr (ALL) return sblk(t);
    else return t < ns ? sblk(t) : gblk_at(t);
  }
  __device__ __forceinline__ int tri(int I, int J) const { return I * nb - I * (I - 1) / 2 + J - I; }
};

template <class T, int NW, bool GP, bool ALL, bool BWD>
__device__ __forceinline__ void bind_storage(Row<T, NW, GP, ALL, BWD>& r, const Args& a) {
  const Layout L = layout(a.nb, a.ns, NW, !GP, BWD);
  char* scr = a.scratch + (size_t)blockIdx.x * a.stride;
  r.o_part = (int)L.part;
  r.o_t = 0;
  r.ns = a.ns;
  r.gblk = reinterpret_cast<float4*>(scr + L.g_blocks);
  r.gpart = reinterpret_cast<T*>(scr + L.g_part);
  r.V = reinterpret_cast<T*>(scr + L.g_v);
  r.X = reinterpret_cast<T*>(scr + L.g_x);
  r.AB = ALL || NW == 1 ? r.sblk() : reinterpret_cast<float4*>(scr + L.g_ab);
}
template <class T, int NW, bool GP, bool ALL, bool BWD>
__device__ __forceinline__ void take_row(Row<T, NW, GP, ALL, BWD>& r, const Args& a, int j) {
  r.j = j;
  r.m = a.m[j];
  r.pos = a.pos[j];
  r.nb = (r.m + kB - 1) / kB;
  r.mp = r.nb * kB;
}
template <class T, int NW, bool GP, bool ALL, bool BWD>
__device__ __forceinline__ void load_nodes(const Row<T, NW, GP, ALL, BWD>& r, const Args& a) {
  for (int q = threadIdx.x; q < kNodesAll; q += threads_of<NW, ALL>()) {
    r.nodes()[q] = a.nodes.theta[q];
    r.nodes()[kNodesAll + q] = a.nodes.w[q];
  }
}

// Column -> bucket of its position in R: kBuckets equal parts of [R_0, R_last], so a bucket
// holds a position or two of a scattered pattern and a search is one bucket read and a short
// bisection instead of log2(m) dependent shared-memory reads.
struct Buckets {
  unsigned first, range, mul;
  __device__ __forceinline__ unsigned of(int col) const {       // col in [R_0, R_last]
    const unsigned d = (unsigned)col - first;
    return range <= (unsigned)kBuckets ? d : __umulhi(d, mul);
  }
};
template <class T, int NW, bool GP, bool ALL, bool BWD>
__device__ __forceinline__ Buckets make_buckets(const Row<T, NW, GP, ALL, BWD>& r) {
  Buckets k;
  k.first = (unsigned)r.R()[0];
  k.range = (unsigned)r.R()[r.m - 1] - k.first + 1;
  k.mul = k.range <= (unsigned)kBuckets ? 0u : (unsigned)(((unsigned long long)kBuckets << 32) / k.range);
  return k;
}
// r.bk()[b] = first position whose bucket is at least b (b <= kBuckets).
template <class T, int NW, bool GP, bool ALL, bool BWD>
__device__ __forceinline__ void fill_buckets(const Row<T, NW, GP, ALL, BWD>& r, const Buckets& k) {
  for (int i = threadIdx.x; i <= r.m; i += threads_of<NW, ALL>()) {
    const int b0 = i == 0 ? 0 : (int)k.of(r.R()[i - 1]) + 1;
    const int b1 = i == r.m ? kBuckets : (int)k.of(r.R()[i]);
    for (int b = b0; b <= b1; ++b) r.bk()[b] = (uint16_t)i;
  }
}
// Positions of U columns in R (-1 where absent; col < 0 gives -1).
template <int U, class T, int NW, bool GP, bool ALL, bool BWD>
__device__ __forceinline__ void find_cols(const Row<T, NW, GP, ALL, BWD>& r, const Buckets& k, const int* col, int* pos) {
  int lo[U], n[U];
  int most = 0;
#pragma unroll
  for (int u = 0; u < U; ++u) {
    const bool in = col[u] >= 0 && (unsigned)col[u] - k.first < k.range;
    const unsigned b = in ? k.of(col[u]) : 0u;
    lo[u] = r.bk()[b];
    n[u] = in ? (int)r.bk()[b + 1] - lo[u] : 0;
    most = max(most, n[u]);
  }
  for (most = __reduce_max_sync(0xffffffffu, most); most > 1; most -= most >> 1) {
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int half = n[u] >> 1;
      if (half > 0 && r.R()[lo[u] + half] <= col[u]) lo[u] += half;
      n[u] -= half;
    }
  }
#pragma unroll
  for (int u = 0; u < U; ++u) pos[u] = n[u] > 0 && r.R()[lo[u]] == col[u] ? lo[u] : -1;
}

// Gather (Alg. 1): the stored entries (k, l), l >= k, of S into the blocks.  A pattern row is
// read from its diagonal on (plan's pos), so half of it; a warp takes one row, its next row's
// first entries already requested.  Returns false (to every thread) when some diagonal entry
// is not a positive normal number, or an entry below the diagonal is not finite (those are looked
// at only when A holds such a value at all; above it, they reach the row sums of stats()).
template <class T, int NW, bool GP, bool ALL, bool BWD>
__device__ bool gather(Row<T, NW, GP, ALL, BWD>& r, const Args& a) {
  constexpr int NT = threads_of<NW, ALL>();
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int base = a.rowptr[r.j], m = r.m;
  const bool look = *a.nonfinite != 0;
  int mx = 0, mn = 0x7fffffff;                       // high words of the diagonal entries
  for (int k = tid; k < m; k += NT) {
    const int c = a.colind[base + k];
    r.R()[k] = c;
    const int first = a.rowptr[c];
    const int2 x = make_int2(first + a.pos[c], a.rowptr[c + 1]);
    r.ext()[k] = x;
    if (BWD) r.start()[k] = first;
    const int h = __double2hiint(a.vals[x.x]);
    mx = max(mx, h);
    mn = min(mn, h);
  }
  const int nblk = nblocks(r.nb), in_s = min(nblk, r.ns) * (kBlkBytes / 16);
  for (int e = tid; e < in_s; e += NT) r.sblk()[e] = make_float4(0.f, 0.f, 0.f, 0.f);
  for (int e = tid; e < nblk * (kBlkBytes / 16) - in_s; e += NT) r.gblk[e] = make_float4(0.f, 0.f, 0.f, 0.f);
  mx = __reduce_max_sync(0xffffffffu, mx);
  mn = __reduce_min_sync(0xffffffffu, mn);
  int* ired = reinterpret_cast<int*>(r.red());
  if (lane == 0) {
    ired[2 * warp] = mx;
    ired[2 * warp + 1] = mn;
  }
  sync_all<NW, ALL>();
  const Buckets bk = make_buckets(r);
  fill_buckets(r, bk);
#pragma unroll
  for (int w = 0; w < NT / 32; ++w) {
    mx = max(mx, ired[2 * w]);
    mn = min(mn, ired[2 * w + 1]);
  }
  r.e0 = mx >> 20;
  sync_all<NW, ALL>();
  if (mn <= 0x00100000 || r.e0 < 64 || r.e0 >= 0x7FF - 64) return false;
  constexpr int U = 4;                               // 128 entries of a pattern row in flight
  int ncol[U];
  double nv[U];
  auto load = [&](int e0, int e1, int* col, double* v) {
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int e = e0 + u * 32 + lane;
      col[u] = e < e1 ? a.colind[e] : -1;
      v[u] = e < e1 ? a.vals[e] : 0.0;
    }
  };
  constexpr int NWALL = NT / 32;
  if (warp < m) load(r.ext()[warp].x, r.ext()[warp].y, ncol, nv);
  for (int k = warp; k < m; k += NWALL) {
    const int b = r.ext()[k].x, e1 = r.ext()[k].y;
    int col[U];
    double v[U];
#pragma unroll
    for (int u = 0; u < U; ++u) col[u] = ncol[u], v[u] = nv[u];
    if (k + NWALL < m) load(r.ext()[k + NWALL].x, r.ext()[k + NWALL].y, ncol, nv);
    const int I = k >> 5, rr = k & 31, t0 = r.tri(I, I) - I;
    for (int e0 = b;;) {
      int l[U];
      find_cols<U>(r, bk, col, l);
#pragma unroll
      for (int u = 0; u < U; ++u) {
        if (l[u] >= 0) {
          const int q = l[u], J = q >> 5, cc = q & 31;
          const T x = scaled(v[u], r.e0, (T*)nullptr);
          float4* blk = r.blk(t0 + J);
          put(blk, rr, cc, x);
          if (I == J) put(blk, cc, rr, x);
        }
      }
      e0 += 32 * U;
      if (e0 >= e1) break;
      load(e0, e1, col, v);
    }
  }
  if (look) {
    for (int k = warp; k < m; k += NWALL) {
      const int e1 = r.ext()[k].x;
      for (int e0 = a.rowptr[r.R()[k]]; e0 < e1; e0 += 32 * U) {
        int col[U], l[U];
        double v[U];
        load(e0, e1, col, v);
        find_cols<U>(r, bk, col, l);
#pragma unroll
        for (int u = 0; u < U; ++u)
          if (l[u] >= 0 && (__double2hiint(v[u]) & 0x7FF00000) == 0x7FF00000) r.flag()[1] = 1;
      }
    }
  }
  sync_all<NW, ALL>();
  return !look || r.flag()[1] == 0;
}

template <class T, int NW, bool GP, bool ALL, bool BWD, class F>
__device__ __forceinline__ void for_blocks(const Row<T, NW, GP, ALL, BWD>& r, int warp, F f) {
  int I = 0, J = 0;
  auto step = [&](int s) {
    J += s;
    while (I < r.nb && J >= r.nb) {
      ++I;
      J = J - r.nb + I;
    }
  };
  step(warp);
  for (int t = warp; I < r.nb; t += NW, step(NW)) f(t, I, J);
}

// Gershgorin bound, accumulator start and certified lower end.
template <class T, int NW, bool GP, bool ALL, bool BWD>
__device__ void stats(Row<T, NW, GP, ALL, BWD>& r) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  float2* p2 = reinterpret_cast<float2*>(r.part());
  if (warp < NW)
    for_blocks(r, warp, [&](int t, int I, int J) {
      if (ALL || t < r.ns) block_stats<T>(r.sblk(t), I, J, p2, r.mp, lane);
      else block_stats<T>(r.gblk_at(t), I, J, p2, r.mp, lane);
    });
  sync_all<NW, ALL>();
  float lam = 0.f, nu = 0.f;
  if (warp < NW)
    for (int i = tid; i < r.mp; i += NW * 32) {
      float s = 0.f, c = 0.f;
      for (int x = 0; x < r.nb; ++x) {
        const float2 q = p2[x * r.mp + i];
        s += q.x;
        c += q.y;
      }
      lam = (s != s || lam != lam) ? s + lam : fmaxf(lam, s);
      nu = fmaxf(nu, c);
    }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const float s = __shfl_xor_sync(0xffffffffu, lam, o);
    lam = (s != s || lam != lam) ? s + lam : fmaxf(lam, s);
    nu = fmaxf(nu, __shfl_xor_sync(0xffffffffu, nu, o));
  }
  float* fred = reinterpret_cast<float*>(r.red());
  if (lane == 0) {
    fred[2 * warp] = lam;
    fred[2 * warp + 1] = nu;
  }
  sync_all<NW, ALL>();
  constexpr int NWALL = threads_of<NW, ALL>() / 32;
#pragma unroll
  for (int w = 0; w < NWALL; ++w) {
    const float s = fred[2 * w];
    lam = (s != s || lam != lam) ? s + lam : fmaxf(lam, s);
    nu = fmaxf(nu, fred[2 * w + 1]);
  }
  r.lam = lam * (1.f + 1e-4f);                       // covers the FP32 sums' rounding
  const float norm = sqrtf(nu) * (1.f + 1e-4f);
  int ex = ((__float_as_int(norm) >> 23) & 0xFF) + 1;      // 2^(ex - 127) > norm
  ex = min(max(ex, 1), 250);
  r.C = 3.f * __int_as_float(ex << 23);
  r.sigma = r.lam / kKappa;
  sync_all<NW, ALL>();
}

// Node state of the stopping bound (node warp: lane = node) and a Sturm sequence at the
// lane's shift, which brackets T's smallest eigenvalue.
struct NodeState {
  float t, wt;            // shift, weight
  float d, u;             // last pivot of T + t, |e_k^T (T + t)^(-1) e_1|
  float shift, ds;        // Sturm shift, last pivot of T - shift
  bool above;             // T - shift positive definite so far
  float b2;               // beta^2 of the last step
  float lam;
  bool first;
};
__device__ __forceinline__ float sturm_shift(int lane) {      // over lam
  return lane == 31 ? 0.985f : exp2f(-kSturm * (float)(lane + 1));
}
__device__ __forceinline__ void node_init(NodeState& s, float theta, float w, float lam, float sigma,
                                          int p, int sign, int lane) {
  const float tau = kTau * lam;
  if (p == 1) {           // x^(-1): the node t = 0 alone
    s.t = 0.f;
    s.wt = lane == 0 ? lam : 0.f;
  } else {
    s.t = tau * theta;
    const float al = sign < 0 ? 1.f / (float)p : 1.f - 1.f / (float)p;
    // relative to the smallest possible norm of the column (lam^(-a); sigma^(1/p) for sign > 0)
    const float pref = exp2f(al * log2f(1.f / kTau)) * (sign < 0 ? 1.f : exp2f(log2f(lam / sigma) / (float)p));
    s.wt = pref * w * tau;
  }
  s.lam = lam;
  s.shift = lam * sturm_shift(lane);
  s.above = true;
  s.first = true;
  s.d = s.u = s.ds = s.b2 = 0.f;
}
// Largest Sturm shift below every Ritz value, over lam (0: none).
__device__ __forceinline__ float node_lo(const NodeState& s) {
  const unsigned up = __ballot_sync(0xffffffffu, s.above);
  if (up >> 31) return sturm_shift(31);
  return up ? sturm_shift(__ffs(up) - 1) : 0.f;
}
// Bound after the step with alpha, beta; kNoBound once a Ritz value lies below every shift (the
// smallest one only falls, so the row is refused: lam / 2^11.2 is beyond kKappa).
constexpr float kNoBound = 1e30f;
__device__ __forceinline__ float node_step(NodeState& s, float alpha, float beta, float beta_prev) {
  if (s.first) {
    s.d = alpha + s.t;
    s.u = __fdividef(1.f, s.d);
    s.ds = alpha - s.shift;
    s.first = false;
  } else {
    s.d = alpha + s.t - __fdividef(s.b2, s.d);
    s.u = __fdividef(s.u * beta_prev, s.d);
    s.ds = alpha - s.shift - __fdividef(s.b2, s.ds);
  }
  s.above = s.above && s.ds > 0.f;
  s.b2 = beta * beta;
  const float lo = node_lo(s) * s.lam;
  return lo > 0.f ? warp_sum_f(__fdividef(s.wt * beta * fabsf(s.u), lo + s.t)) : kNoBound;
}

// Lanczos from the vector the callers left in r.v (norm 1; NE elements per thread): T in
// al / be, the vectors in r.V.  Returns the number of steps (the same on every thread); *est
// the bound relative to the result (node warp's lanes), lo the bracket of the smallest Ritz
// value over lam (node warp's lanes).
//
// Two barriers a step: r.v holds the unnormalised w = beta_k v_k, products are taken with it
// (the accumulators' start scaled by a power of two above beta_k) and their sums multiplied by
// 1/beta_k, so the norm's reduction needs no barrier of its own; alpha_k = v^T S v comes out of
// the products' row sums (with beta = |w| the stable form of Paige 1972).
template <int NW, class T> __device__ __forceinline__ T row_sum(const T* part, int i, int mp, int nb) {
  T s = part[i];
  for (int x = 1; x < nb; ++x) {
    const T q = part[x * mp + i];
    if constexpr (!kDf<T>) {
      s += q;
    } else {                                          // grid parts add exactly
      s.h += q.h;
      s.l += q.l;
    }
  }
  if constexpr (kDf<T>) s = quick(s.h, s.l);
  return s;
}

template <int NE, class T, int NW, bool GP, bool ALL, bool BWD>
__device__ int lanczos(const Row<T, NW, GP, ALL, BWD>& r, int p, int sign, float tol, float* est, float* lo) {
  constexpr int cap = cap_of(NW);
  constexpr int NM = NW * 32;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const bool mat = warp < NW, node = kLone<NW, ALL> || warp == NW;
  T w[NE], vp[NE];
#pragma unroll
  for (int e = 0; e < NE; ++e) {
    const int i = tid + e * NM;
    vp[e] = zero<T>();
    w[e] = mat && i < r.mp ? r.v_at(i) : zero<T>();
  }
  NodeState ns;
  if (node) node_init(ns, (float)r.nodes()[lane], (float)r.nodes()[kNodesAll + lane], r.lam, r.sigma, p, sign, lane);
  float bound = kNoBound, bprev = 0.f, C = r.C;
  T beta = zero<T>(), inv = one<T>();
  int k = 0;
  for (;; ++k) {
    const int nv = NE > 1 ? NW : min(NW, r.nb);       // warps that hold elements
    if (k > 0) {
      const T n2 = total_of<NW>(r.red() + 16, lane, nv);
      if (warp < nv || node) {
        const bool end = !(hi(n2) > 1e-34f);          // the space is exhausted
        inv = end ? zero<T>() : inv_sqrt(n2);
        beta = end ? zero<T>() : mul(n2, inv);
      }
      const int ex = (int)((__float_as_uint(hi(n2)) >> 23) & 0xFF) - 127;
      C = r.C * __int_as_float((((ex + 2) >> 1) + 127) << 23);       // 2^((ex+2)/2) >= beta
    }
    if (mat && k < cap) {
      T dot = zero<T>();
      for_blocks(r, warp, [&](int t, int I, int J) {
        auto go = [&](const float4* b) {
          if (I == J) block_mul<false>(b, r.v(), I, J, C, r.part(), r.mp, lane, dot);
          else block_mul<true>(b, r.v(), I, J, C, r.part(), r.mp, lane, dot);
        };
        if (ALL || t < r.ns) go(r.sblk(t)); else go(r.gblk_at(t));
      });
      dot = warp_total(dot);
      if (lane == 0) r.red()[warp] = dot;
    }
    if (node && k > 0) {
      const float b = hi(beta);
      bound = node_step(ns, hi(r.al()[k - 1]), b, bprev);
      bprev = b;
      // NaN ends the run too: the row is then refused
      if (lane == 0) {
        r.be()[k - 1] = beta;
        r.flag()[0] = !(bound > tol) || bound >= kNoBound || k >= cap;
      }
    }
    sync_all<NW, ALL>();
    const bool stop = k > 0 && r.flag()[0];
    if (warp < nv) {
      const T al = mul(mul(total_of<NW>(r.red(), lane, NW), inv), inv);
      T n2 = zero<T>();
#pragma unroll
      for (int e = 0; e < NE; ++e) {
        const int i = tid + e * NM;
        if (i < r.mp) {
          const T v = mul(w[e], inv);
          r.V[(size_t)k * r.mp + i] = v;
          if (!stop) {
            const T sv = mul(row_sum<NW>(r.part(), i, r.mp, r.nb), inv);
            w[e] = sub(sub(sv, mul(beta, vp[e])), mul(al, v));
            vp[e] = v;
            r.set_v(i, w[e]);
            n2 = NE > 1 ? add(n2, mul(w[e], w[e])) : mul(w[e], w[e]);
          }
        }
      }
      if (!stop) {
        n2 = warp_total(n2);
        if (lane == 0) r.red()[16 + warp] = n2;
        if (tid == 0) r.al()[k] = al;
      }
    }
    if (stop) break;
    sync_all<NW, ALL>();
  }
  sync_all<NW, ALL>();
  if (node) {
    *est = bound;
    *lo = node_lo(ns);
  }
  return k;
}

// tau for a smallest Ritz value of lo lam.
__device__ __forceinline__ float tau_of(float lam, float lo) {
  return lam * (lo >= kLoWide ? kTau : sqrtf(lo));
}

// Node solutions x = (T + t)^(-1) e_1 (node q of the lane, the whole warp calls it), times the
// node's weight, in r.X[k][lane]; a bottom-up elimination leaves the right-hand side e_1 alone,
// so one sweep up for the pivots and one down for x.
// The weight is tau w_q wt0 (times t for x^(1/p), whose adjoint weighs t (x + t)^(-1)).
template <class T, int NW, bool GP, bool ALL, bool BWD>
__device__ void node_solve(const Row<T, NW, GP, ALL, BWD>& r, int K, float tau_f, int q, bool weighted,
                           bool times_t, T wt0) {
  const int lane = threadIdx.x & 31;
  const T tau = as(tau_f, (T*)nullptr);
  const T t = mul(tau, as(r.nodes()[q], (T*)nullptr));
  T wt = mul(tau, as(r.nodes()[kNodesAll + q], (T*)nullptr));
  if (times_t) wt = mul(wt, t);
  wt = mul(wt, wt0);
  T x = rcp(add(r.al()[K - 1], t));
  for (int k = K - 2; k >= 0; --k) {
    const T g = mul(r.be()[k], x);
    r.set_x(k, lane, g);
    x = rcp(sub(add(r.al()[k], t), mul(r.be()[k], g)));
  }
  if (weighted) x = mul(x, wt);
  for (int k = 0; k < K; ++k) {
    T g = zero<T>();
    if (k + 1 < K) g = r.x_at(k, lane);
    r.set_x(k, lane, x);
    x = neg(mul(g, x));
  }
  __syncwarp();
}

// coef[k] (+)= sum over the nodes of X[k][.].
template <class T, int NW, bool GP, bool ALL, bool BWD>
__device__ void sum_nodes(const Row<T, NW, GP, ALL, BWD>& r, int K, bool more) {
  for (int k = threadIdx.x & 31; k < K; k += 32) {
    T s = r.x_at(k, 0);
    for (int q = 1; q < kNodes; ++q) s = add(s, r.x_at(k, q));
    r.coef()[k] = more ? add(r.coef()[k], s) : s;
  }
  __syncwarp();
}

// coef = f(T) e_1 up to the factor tau^(-a); f(x) = x x^(-a) (`times_t`) multiplies by T, which
// adds the component K.  Returns the number of coefficients.  The whole (node) warp calls it.
template <class T, int NW, bool GP, bool ALL, bool BWD>
__device__ int root_coefs(const Row<T, NW, GP, ALL, BWD>& r, int K, int p, float lo, bool times_t, int lane) {
  if (p == 1) {
    // one node, t = 0: a lane's work, all of it in shared memory (through X and the sum over the
    // nodes: mixed inverse n = 2000, orders up to 28, 175 -> 165 us; FP64, where nothing hides it,
    // 256 -> 248)
    if (lane == 0) {
      T x = rcp(r.al()[K - 1]);
      for (int k = K - 2; k >= 0; --k) {
        const T g = mul(r.be()[k], x);
        r.coef()[k + 1] = g;
        x = rcp(sub(r.al()[k], mul(r.be()[k], g)));
      }
      r.coef()[0] = x;
      for (int k = 1; k < K; ++k) {
        x = neg(mul(r.coef()[k], x));
        r.coef()[k] = x;
      }
    }
    __syncwarp();
    return K;
  }
  const float tau = tau_of(r.lam, lo);
  if (lo >= kLoWide) {
    node_solve(r, K, tau, lane, true, false, one<T>());
    sum_nodes(r, K, false);
  } else {
#pragma unroll 1
    for (int h = 0; h < kNodesWide / 32; ++h) {
      node_solve(r, K, tau, kNodes + 32 * h + lane, true, false, one<T>());
      sum_nodes(r, K, h > 0);
    }
  }
  if (!times_t) return K;
  T c[(cap_of(NW) + 32) / 32];   // cap + 1 components, one per lane
#pragma unroll
  for (int u = 0; u < (cap_of(NW) + 32) / 32; ++u) {
    const int k = lane + 32 * u;
    T s = zero<T>();
    if (k < K) s = mul(r.al()[k], r.coef()[k]);
    if (k > 0 && k <= K) s = add(s, mul(r.be()[k - 1], r.coef()[k - 1]));
    if (k + 1 < K) s = add(s, mul(r.be()[k], r.coef()[k + 1]));
    c[u] = s;
  }
  __syncwarp();
#pragma unroll
  for (int u = 0; u < (cap_of(NW) + 32) / 32; ++u) {
    const int k = lane + 32 * u;
    if (k <= K) r.coef()[k] = c[u];
  }
  __syncwarp();
  return K + 1;
}

// FP32 Cholesky of S - sigma I in place of the blocks (S is not needed any more): U^T U, block
// rows top down.  The warp that updates the next diagonal block factorises it at once, while
// the others finish the update.  Called by the NW matrix warps; true when every pivot is
// positive.  S's rounding to FP32 and the factorisation's own move eigenvalues by at most about
// m 2^-24 lam: 9.2e-5 lam at the largest order, a fifth of sigma = lam / kKappa = 5e-4 lam there
// (a fortieth at order 192), so what passes has lambda_min above 0.8 sigma at least.
template <class T, int NW, bool GP, bool ALL, bool BWD>
__device__ bool cholesky(const Row<T, NW, GP, ALL, BWD>& r) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  float* invd = reinterpret_cast<float*>(r.part());    // 32 reciprocal pivots' roots
  int* bad = r.flag() + 1;
  for_blocks(r, warp, [&](int t, int I, int J) {     // leading parts, row-major 32 x 32
    float4* b = r.blk(t);
    float x[32];
#pragma unroll
    for (int i = 0; i < 16; ++i) elem_hi(b[i * 32 + lane], x[2 * i], x[2 * i + 1], (T*)nullptr);
    __syncwarp();
    const int a4 = (lane >> 2) * 4, b8 = (lane & 3) * 8;
    if (I == J) {
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 8; ++j)
          if (a4 + i == b8 + j) x[i * 8 + j] = I * kB + a4 + i < r.m ? x[i * 8 + j] - r.sigma : 1.f;
    }
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 2; ++j)
        b[(a4 + i) * 8 + (lane & 3) * 2 + j] =
            make_float4(x[i * 8 + 4 * j], x[i * 8 + 4 * j + 1], x[i * 8 + 4 * j + 2], x[i * 8 + 4 * j + 3]);
  });
  sync_mat<NW>();
  auto factor = [&](int I) {                          // one warp; lane = column
    float* b = reinterpret_cast<float*>(r.blk(r.tri(I, I)));
    float x[32];
#pragma unroll
    for (int i = 0; i < 32; ++i) x[i] = b[i * 32 + lane];
    bool ok = true;
#pragma unroll
    for (int k = 0; k < 32; ++k) {
      const float piv = __shfl_sync(0xffffffffu, x[k], k);
      ok = ok && piv > 0.f;
      const float inv = rsqrtf(piv);
      const float u = x[k] * inv;                     // row k of U
#pragma unroll
      for (int i = k + 1; i < 32; ++i)                // x_ic -= u_ki u_kc, u_ki = a_ik / sqrt(pivot)
        x[i] = fmaf(-__shfl_sync(0xffffffffu, u, i), u, x[i]);
      b[k * 32 + lane] = u;
      if (lane == 0) invd[k] = inv;
    }
    if (!ok && lane == 0) *bad = 1;
  };
  if (warp == 0) factor(0);
  sync_mat<NW>();
  for (int I = 0; I + 1 < r.nb; ++I) {
    if (*bad) break;
    const float4* u4 = r.blk(r.tri(I, I));
    for (int J = I + 1 + warp; J < r.nb; J += NW) {   // U_IJ = U_II^-T A_IJ; lane = column
      float* b = reinterpret_cast<float*>(r.blk(r.tri(I, J)));
      float x[32];
#pragma unroll
      for (int i = 0; i < 32; ++i) x[i] = b[i * 32 + lane];
#pragma unroll
      for (int k = 0; k < 32; ++k) {
        x[k] *= invd[k];
#pragma unroll
        for (int q = (k + 1) / 4; q < 8; ++q) {
          const float4 u = u4[k * 8 + q];
          if (4 * q > k) x[4 * q] = fmaf(-u.x, x[k], x[4 * q]);
          if (4 * q + 1 > k) x[4 * q + 1] = fmaf(-u.y, x[k], x[4 * q + 1]);
          if (4 * q + 2 > k) x[4 * q + 2] = fmaf(-u.z, x[k], x[4 * q + 2]);
          if (4 * q + 3 > k) x[4 * q + 3] = fmaf(-u.w, x[k], x[4 * q + 3]);
        }
        b[k * 32 + lane] = x[k];
      }
    }
    sync_mat<NW>();
    auto update = [&](int J, int Kb) {                // A_JK -= U_IJ^T U_IK
      const float4* p = r.blk(r.tri(I, J));
      const float4* q = r.blk(r.tri(I, Kb));
      float4* d = r.blk(r.tri(J, Kb));
      const int a4 = lane >> 2, b8 = lane & 3;
      float acc[4][8] = {};
#pragma unroll 2
      for (int k = 0; k < 32; ++k) {
        const float4 x = p[k * 8 + a4], y0 = q[k * 8 + b8 * 2], y1 = q[k * 8 + b8 * 2 + 1];
        const float xs[4] = {x.x, x.y, x.z, x.w};
        const float ys[8] = {y0.x, y0.y, y0.z, y0.w, y1.x, y1.y, y1.z, y1.w};
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
          for (int j = 0; j < 8; ++j) acc[i][j] = fmaf(xs[i], ys[j], acc[i][j]);
      }
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 2; ++j) {
          float4 z = d[(a4 * 4 + i) * 8 + b8 * 2 + j];
          z.x -= acc[i][4 * j];
          z.y -= acc[i][4 * j + 1];
          z.z -= acc[i][4 * j + 2];
          z.w -= acc[i][4 * j + 3];
          d[(a4 * 4 + i) * 8 + b8 * 2 + j] = z;
        }
    };
    if (warp == 0) {
      update(I + 1, I + 1);
      __syncwarp();
      factor(I + 1);
    }
    constexpr int NO = NW > 1 ? NW - 1 : 1;           // the other warps share the other blocks
    if (NW == 1 || warp > 0) {
      const int mine = NW == 1 ? 0 : warp - 1;
      int t = 0;
      for (int J = I + 1; J < r.nb; ++J)
        for (int Kb = J; Kb < r.nb; ++Kb) {
          if (J == I + 1 && Kb == J) continue;
          if (t++ % NO == mine) update(J, Kb);
        }
    }
    sync_mat<NW>();
  }
  return *bad == 0;
}

// The condition estimate lambda_bar / lambda_min that the mixed engines compare with kappa_max: eight
// power steps on I - S / lambda_bar from a vector of +-1, in FP32 (see start_lo_slices; the norm
// is taken of the last two vectors only).  S's blocks are in place; the row's vector and sums are
// overwritten.  Called by the NW matrix warps, while the node warp solves for the coefficients
// (rows of at most 32 entries: a lane per row of S, held in registers).
template <int NW, bool GP, bool ALL>
__device__ __noinline__ float condition_estimate(const Args& a, int m, float lam) {
  constexpr int NM = NW * 32;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  Row<float, NW, GP, ALL, false> q;
  const float start = rsqrtf((float)m), scale = 1.f / lam;
  float last = 0.f, before = 0.f;
  if constexpr (NW == 1) {
    const float4* b = q.sblk();
    float s[kB], v = lane < m ? (lane % 3 == 0 ? start : -start) : 0.f;
#pragma unroll
    for (int c = 0; c < kB; c += 2) {
      const float4 x = b[pair_at(lane, c)];
      s[c] = x.x;
      s[c + 1] = x.y;
    }
#pragma unroll 1
    for (int t = 0; t < kStartLoSteps; ++t) {
      float y[4] = {};
#pragma unroll
      for (int c = 0; c < kB; ++c) y[c & 3] = fmaf(s[c], __shfl_sync(0xffffffffu, v, c), y[c & 3]);
      if (t + 1 == kStartLoSteps) before = warp_total(v * v);
      v -= scale * ((y[0] + y[1]) + (y[2] + y[3]));
    }
    last = warp_total(v * v);
  } else {
    bind_storage(q, a);
    q.m = m;
    q.nb = (m + kB - 1) / kB;
    q.mp = q.nb * kB;
    for (int i = tid; i < q.mp; i += NM) q.set_v(i, i < m ? (i % 3 == 0 ? start : -start) : 0.f);
    for (int t = 0; t < kStartLoSteps; ++t) {
      sync_mat<NW>();
      float dot = 0.f;
      for_blocks(q, warp, [&](int b, int I, int J) {
        auto go = [&](const float4* x) {
          if (I == J) block_mul<false>(x, q.v(), I, J, 0.f, q.part(), q.mp, lane, dot);
          else block_mul<true>(x, q.v(), I, J, 0.f, q.part(), q.mp, lane, dot);
        };
        if (ALL || b < q.ns) go(q.sblk(b)); else go(q.gblk_at(b));
      });
      sync_mat<NW>();
      before = last = 0.f;
      for (int i = tid; i < q.mp; i += NM) {
        const float v = q.v_at(i), d = v - scale * row_sum<NW>(q.part(), i, q.mp, q.nb);
        q.set_v(i, d);
        before = fmaf(v, v, before);
        last = fmaf(d, d, last);
      }
    }
    before = warp_total(before);
    last = warp_total(last);
    if (lane == 0) {
      q.red()[warp] = before;
      q.red()[16 + warp] = last;
    }
    sync_mat<NW>();
    before = total_of<NW>(q.red(), lane, NW);
    last = total_of<NW>(q.red() + 16, lane, NW);
  }
  const float norm = before > 0.f ? sqrtf(last / before) : 0.f;
  return norm < 1.f ? 1.f / (1.f - norm) : 3.0e38f;
}

// r = e_pos - S x in FP64 for x (FP64, r.m entries, in the units of the values): the pattern rows
// are read again, in full, and their entries' columns found as in the gather.  All warps.
template <class T, int NW, bool GP, bool ALL, bool BWD>
__device__ void residual(const Row<T, NW, GP, ALL, BWD>& r, const Args& a, const double* x, double* out) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  constexpr int NWALL = threads_of<NW, ALL>() / 32;
  const Buckets bk = make_buckets(r);
  constexpr int U = 4;
  for (int k = warp; k < r.m; k += NWALL) {
    const int e1 = r.ext()[k].y;
    double s = 0.0;
    for (int e0 = a.rowptr[r.R()[k]]; e0 < e1; e0 += 32 * U) {
      int col[U], l[U];
      double v[U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int e = e0 + u * 32 + lane;
        col[u] = e < e1 ? a.colind[e] : -1;
        v[u] = e < e1 ? a.vals[e] : 0.0;
      }
      find_cols<U>(r, bk, col, l);
#pragma unroll
      for (int u = 0; u < U; ++u)
        if (l[u] >= 0) s = fma(v[u], x[l[u]], s);
    }
    s = warp_sum(s);
    if (lane == 0) out[k] = (k == r.pos ? 1.0 : 0.0) - s;
  }
}

// Row r.j goes to the general path.
template <class T, int NW, bool GP, bool ALL, bool BWD>
__device__ __forceinline__ void leave(const Row<T, NW, GP, ALL, BWD>& r, const Args& a) {
  if (r.m <= a.small_max) a.redo_small[atomicAdd(&a.ctr->n_redo_small, 1)] = r.j;
  else a.redo_list[atomicAdd(&a.ctr->n_redo, 1)] = r.j;
}

// Steps that the coupled iteration would take on spec(M) in [lo, 1] (reported as the row's
// iteration count and the method's flops, which are counted independently of the engine).
__device__ inline int coupled_steps(float lo, int p, int m, bool fp64) {
  const float stop = fp64 ? 1e-7f : (p == 1 ? 1e-4f : 0.05f * rsqrtf((float)m));
  int it = 0;
  while (1.f - lo > stop && it < 40) {
    const float next = scaled_step(lo, p).lo_next;
    ++it;
    if (!(next > lo)) break;                          // FP32 resolution near 1
    lo = next;
  }
  return it;
}

}  // namespace kry
}  // namespace submat
#endif
