// Conjugate gradients on A x = b, plain or with the submatrix method's K ~ A^(-1/2) as the
// preconditioner in the form of Sec. 4.4: CG on K^T A K y = K^T b, then x = K y.
//
// A solve is one cooperative kernel: the whole iteration runs on the device with a grid barrier
// between its phases.  (With a launch per phase and two scalars read by the host per step, a
// step took 72 us at n = 4096, whatever the matrix: launches and the host's round trips.)
// CSR products take a group of lanes per row, the values of K^T are gathered through the plan's
// transposed map, and dot products are reduced in a fixed order that does not depend on the grid
// (kDotBlocks partial sums of kDotThreads strided elements, then their sum, which every block
// forms for itself), so a solve gives the same bits on every call.
// Measured on GB300, a step with / without K: 5-point operator n = 4096, 74 / 57 -> 31 / 18 us;
// n = 160000, 236 / 118 -> 49 / 28 us; overlap matrix n = 4096 (154 entries a row), 73 / 56 ->
// 35 / 20 us.  Bound by the latency of its six (four) barriers and of the FP64 reductions and
// scalars between them; one cluster of 16 blocks instead of the grid timed the same.
#include <algorithm>
#include <cmath>
#include <cooperative_groups.h>
#include "common.cuh"

namespace submat {
namespace {

constexpr int kDotBlocks = 256, kDotThreads = 256;

// kt[e] for e = (r, c): K's value at (c, r), the entry tpos[e] of row c.
__global__ void transpose_vals_kernel(const int32_t* __restrict__ rowptr,
                                      const int32_t* __restrict__ colind,
                                      const int32_t* __restrict__ tpos,
                                      const double* __restrict__ vals, double* __restrict__ kt,
                                      int64_t nnz) {
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < nnz;
       e += (int64_t)gridDim.x * blockDim.x)
    kt[e] = vals[rowptr[colind[e]] + tpos[e]];
}

constexpr int kThreadsCg = 1024;


// y = M x.  G = 32: a warp per row, lanes over the entries, a butterfly of the lanes' sums.
// G = 1 (rows of at most 8 entries): a thread per row, its products added in the butterfly's order
// (the lanes beyond the row would only add zeros): 2.7 times fewer FP64 instructions, which
// issue at 2 lanes a clock.
template <int G>
__device__ void spmv(const CgArgs& a, const double* vals, const double* x, double* y) {
  if constexpr (G == 1) {
    const int nt = gridDim.x * blockDim.x;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < a.n; i += nt) {
      const int b = a.rowptr[i], m = a.rowptr[i + 1] - b;
      double v[8];
#pragma unroll
      for (int k = 0; k < 8; ++k) v[k] = k < m ? vals[b + k] * x[a.colind[b + k]] : 0.0;
      y[i] = ((v[0] + v[4]) + (v[2] + v[6])) + ((v[1] + v[5]) + (v[3] + v[7]));
    }
  } else {
    const int lane = threadIdx.x & 31, warps = (gridDim.x * blockDim.x) >> 5;
    for (int i = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; i < a.n; i += warps) {
      double s = 0.0;
      for (int e = a.rowptr[i] + lane; e < a.rowptr[i + 1]; e += 32) s = fma(vals[e], x[a.colind[e]], s);
      s = warp_sum(s);
      if (lane == 0) y[i] = s;
    }
  }
}

// Partial sum of one virtual block (8 warps): its elements, strided by the virtual grid, through
// f(i); slot: the caller's group of 8 warps within the block.
template <class F>
__device__ void partials(int n, double* part, double* red, F f) {
  const int lane = threadIdx.x & 31, warp = (threadIdx.x >> 5) & 7, slot = threadIdx.x >> 8;
  const int per = kThreadsCg / kDotThreads;
  for (int b0 = blockIdx.x * per; b0 < kDotBlocks; b0 += gridDim.x * per) {
    const int b = b0 + slot;
    const bool some = b < kDotBlocks && b * kDotThreads < n;      // (an empty one's sum is 0)
    if (some) {
      double s = 0.0;
      for (int i = b * kDotThreads + (threadIdx.x & 255); i < n; i += kDotBlocks * kDotThreads) s = f(i, s);
      s = warp_sum(s);
      if (lane == 0) red[slot * 8 + warp] = s;
    }
    __syncthreads();
    if ((threadIdx.x & 255) == 0 && b < kDotBlocks) {
      double t = 0.0;
      if (some)
        for (int w = 0; w < 8; ++w) t += red[slot * 8 + w];
      part[b] = t;
    }
    __syncthreads();
  }
}
// The sum of the partial sums and the step's scalars (f, on one thread: 32 warps of it would take
// the FP64 pipe microseconds), left in val[0..2] for the block.
template <class F>
__device__ void total(const double* part, double* red, F f) {
  static_assert(kDotBlocks == 256, "one partial sum per thread of 8 warps");
  if (threadIdx.x < 256) {
    double s = 0.0;
    s += part[threadIdx.x];
    s = warp_sum(s);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int w = 0; w < 8; ++w) t += red[w];
    f(t);
  }
  __syncthreads();
}

template <int G>
__global__ void __launch_bounds__(kThreadsCg) cg_solve_kernel(CgArgs a) {
  auto sync = [] { cooperative_groups::this_grid().sync(); };
  __shared__ double red[32];
  const bool pre = a.k != nullptr;
  const int t0 = blockIdx.x * blockDim.x + threadIdx.x, nt = gridDim.x * blockDim.x;
  if (pre) {
    spmv<G>(a, a.kt, a.b, a.r);                          // r = K^T b
    sync();
  }
  for (int i = t0; i < a.n; i += nt) {
    const double ri = pre ? a.r[i] : a.b[i];
    if (!pre) a.r[i] = ri;
    a.p[i] = ri;
    a.y[i] = 0.0;
  }
  sync();
  partials(a.n, a.part, red, [&](int i, double s) { return fma(a.r[i], a.r[i], s); });
  sync();
  // on one thread of each block, the same on all: r.r, |b| and whether to go on
  __shared__ double rr, bnorm, scal;
  __shared__ int go;
  int it = 0, status = 0;
  total(a.part, red, [&](double t) {
    rr = t;
    bnorm = sqrt(t);
    go = bnorm > 0.0 && sqrt(rr) > a.tol * bnorm && a.max_iter > 0;
  });
  // part holds 2 kDotBlocks sums: p.q and r.r alternate, so that one is read while the other is
  // written
  while (go) {
    if (pre) {                                                    // q = K^T A K p
      spmv<G>(a, a.k, a.p, a.t1);
      sync();
      spmv<G>(a, a.a, a.t1, a.t2);
      sync();
      spmv<G>(a, a.kt, a.t2, a.q);
    } else {                                                      // q = A p
      spmv<G>(a, a.a, a.p, a.q);
    }
    sync();
    partials(a.n, a.part + kDotBlocks, red, [&](int i, double s) { return fma(a.p[i], a.q[i], s); });
    sync();
    total(a.part + kDotBlocks, red, [&](double pq) {
      scal = rr / pq;                                             // alpha
      go = pq > 0.0 && !isinf(pq);
    });
    if (!go) {                                                    // not positive definite
      status = 1;
      break;
    }
    const double alpha = scal;
    partials(a.n, a.part, red, [&](int i, double s) {
      a.y[i] = fma(alpha, a.p[i], a.y[i]);
      const double ri = fma(-alpha, a.q[i], a.r[i]);
      a.r[i] = ri;
      return fma(ri, ri, s);
    });
    sync();
    ++it;
    total(a.part, red, [&](double t) {
      scal = t / rr;                                              // beta
      rr = t;
      go = sqrt(rr) > a.tol * bnorm && it < a.max_iter;
    });
    const double beta = scal;
    for (int i = t0; i < a.n; i += nt) a.p[i] = fma(beta, a.p[i], a.r[i]);
    sync();
  }
  if (pre) spmv<G>(a, a.k, a.y, a.x);                             // x = K y
  if (t0 == 0) *a.out = CgResult{rr, bnorm, it, status};
}

}  // namespace

cudaError_t cg_transpose_vals(const int32_t* rowptr, const int32_t* colind, const int32_t* tpos,
                              const double* vals, double* kt, int64_t nnz, cudaStream_t s) {
  const int blocks = (int)std::min<int64_t>((nnz + 255) / 256, 65535);
  if (blocks > 0) transpose_vals_kernel<<<blocks, 256, 0, s>>>(rowptr, colind, tpos, vals, kt, nnz);
  return cudaGetLastError();
}

cudaError_t cg_solve(const CgArgs& a, int m_max, int n_sm, cudaStream_t s) {
  const void* f = m_max <= 8 ? (const void*)cg_solve_kernel<1> : (const void*)cg_solve_kernel<32>;
  const int64_t need = ((int64_t)a.n * (m_max <= 8 ? 1 : 32) + kThreadsCg - 1) / kThreadsCg;
  int per_sm = 0;
  const cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, f, kThreadsCg, 0);
  if (e != cudaSuccess) return e;
  // (16 to 152 blocks time alike at n = 4096; one to four leave the partial sums to too few)
  const int blocks = (int)std::min<int64_t>(std::max<int64_t>(need, 64), (int64_t)per_sm * n_sm);
  CgArgs args = a;
  void* params[] = {&args};
  return cudaLaunchCooperativeKernel(f, dim3(blocks), dim3(kThreadsCg), params, 0, s);
}

size_t cg_dot_scratch() { return 2 * kDotBlocks; }

}  // namespace submat
