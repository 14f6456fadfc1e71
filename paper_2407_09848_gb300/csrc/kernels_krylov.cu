// Outer-solver kernels (preconditioned CG, Sec. 4), the coarsest-level dense
// solve, and the power-iteration estimate.  All reductions are deterministic
// (fixed grid, fixed summation tree: see grid_sum), so a solve repeated on
// the same input performs the same iterations bit for bit.
#include <atomic>

#include "kernels_common.cuh"

namespace amgps {

namespace {
// kernels enqueued by this process (all contexts, all host threads)
std::atomic<int64_t> g_launches{0};
}
int64_t launches_enqueued() { return g_launches.load(std::memory_order_relaxed); }
void count_launch() { g_launches.fetch_add(1, std::memory_order_relaxed); }

int reduction_grid(int64_t work_items, int nsm, int per_sm) {
  int64_t g = (work_items + kBlock - 1) / kBlock;
  const int64_t cap = (int64_t)nsm * per_sm;
  if (g > cap) g = cap;
  if (g < 1) g = 1;
  return (int)g;
}

// Entries a thread of the streaming reductions loads before it uses any.
constexpr int kLoads = 4;

// q = A p and p.q (S_PQ).  One warp per slice, grid-stride over slices.
__global__ void __launch_bounds__(kBlock, 4) k_spmv_dot(const DevMat<double> A,
                                                     const double* p, double* q, const RedWork w,
                                                     double* scal) {
  pdl_wait();
  pdl_go();
  const int lane = threadIdx.x & 31;
  const int64_t nw = (int64_t)gridDim.x * kWarpsPerBlock;
  double acc = 0.0;
  for (int64_t s = (int64_t)blockIdx.x * kWarpsPerBlock + (threadIdx.x >> 5); s < A.nslices;
       s += nw) {
    const int64_t row = s * kSlice + lane;
    const double t = row_spmv<1, double, double>(A, s, lane, row, p, 0.0);
    if (row < A.n) {
      q[row] = t;
      acc = fma(ldv<false>(p + row), t, acc);
    }
  }
  grid_sum(
      acc, w, [&] { return __ldcg(scal + S_RZ); },
      [&](double tot, double rz) {
        scal[S_PQ] = tot;
        scal[S_ALPHA] = rz / tot;  // once per iteration, not once per thread
      });
}

void launch_spmv_dot(const DevMat<double>& A, const double* p, double* q, const RedWork& w,
                     double* scal, cudaStream_t s) {
  launch_dep(k_spmv_dot, w.grid, kBlock, 0, s, A, p, q, w, scal);
}

// A batch of products: blockIdx.y is the vector, with its own row of partials
// and its own counter.
__global__ void __launch_bounds__(kBlock, 4) k_spmv_dot_mv(const DevMat<double> A, const double* p,
                                                           double* q, RedWork w, double* out,
                                                           int stride) {
  pdl_wait();
  pdl_go();
  const int lane = threadIdx.x & 31, v = blockIdx.y;
  p += v * A.n;
  q += v * A.n;
  w.part += (size_t)v * gridDim.x;
  w.counter += v;
  const int64_t nw = (int64_t)gridDim.x * kWarpsPerBlock;
  double acc = 0.0;
  for (int64_t s = (int64_t)blockIdx.x * kWarpsPerBlock + (threadIdx.x >> 5); s < A.nslices;
       s += nw) {
    const int64_t row = s * kSlice + lane;
    const double t = row_spmv<1, double, double>(A, s, lane, row, p, 0.0);
    if (row < A.n) {
      q[row] = t;
      acc = fma(ldv<false>(p + row), t, acc);
    }
  }
  grid_sum(acc, w, [&](double tot) { out[v * stride] = tot; });
}

void launch_spmv_dot_mv(const DevMat<double>& A, const double* p, double* q, const RedWork& w,
                        double* out, int stride, int nvec, cudaStream_t s) {
  launch_dep(k_spmv_dot_mv, dim3(w.grid, nvec), kBlock, 0, s, A, p, q, w, out, stride);
}

// Three sums in one pass (the one-reduction flexible CG): partials are laid
// out [v0 of every block | v1 ... | v2 ...] in w.part (3 x grid doubles); the
// last block adds each column in index order and calls fin(t0, t1, t2).
template <class Fin>
__device__ __forceinline__ void grid_sum3(double v0, double v1, double v2, const RedWork& w,
                                          Fin fin) {
  __shared__ double sh[kBlock];
  __shared__ bool last;
  const double b0 = block_sum(v0, sh);
  const double b1 = block_sum(v1, sh);
  const double b2 = block_sum(v2, sh);
  if (threadIdx.x == 0) {
    w.part[blockIdx.x] = b0;
    w.part[gridDim.x + blockIdx.x] = b1;
    w.part[2 * gridDim.x + blockIdx.x] = b2;
    __threadfence();
    const unsigned t = atomicAdd(w.counter, 1u);
    last = (t == gridDim.x - 1);
  }
  __syncthreads();
  if (last) {
    __threadfence();
    double t[3];
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      double s = 0.0;
      for (int i = threadIdx.x; i < (int)gridDim.x; i += blockDim.x)
        s += __ldcg(w.part + j * gridDim.x + i);
      t[j] = block_sum(s, sh);
    }
    if (threadIdx.x == 0) {
      fin(t[0], t[1], t[2]);
      *w.counter = 0u;
    }
  }
}

// One-reduction flexible CG (the outer solver of Sec. 4): w = A z and the
// three inner products rho = z.r, gamma = z.q_old, delta = z.w in a single
// grid reduction.  The last block forms beta = gamma / eta_old (the
// A-orthogonalisation of z against p_old), eta = p.A p = delta - beta gamma
// (by symmetry of A, with q = A p), and alpha = rho / eta.
__global__ void __launch_bounds__(kBlock, 4) k_spmv_dot3(const DevMat<double> A,
                                                      const double* z, double* w, const double* r,
                                                      const double* q, int first, const RedWork rw,
                                                      double* scal) {
  pdl_wait();
  pdl_go();
  const int lane = threadIdx.x & 31;
  const int64_t nw = (int64_t)gridDim.x * kWarpsPerBlock;
  double zr = 0.0, zq = 0.0, zw = 0.0;
  for (int64_t s = (int64_t)blockIdx.x * kWarpsPerBlock + (threadIdx.x >> 5); s < A.nslices;
       s += nw) {
    const int64_t row = s * kSlice + lane;
    const double t = row_spmv<1, double, double>(A, s, lane, row, z, 0.0);
    if (row < A.n) {
      w[row] = t;
      const double zi = ldv<false>(z + row);
      zw = fma(zi, t, zw);
      zr = fma(zi, ldv<false>(r + row), zr);
      if (!first) zq = fma(zi, ldv<false>(q + row), zq);
    }
  }
  grid_sum3(zr, zq, zw, rw, [&](double rho, double gam, double del) {
    const double beta = first ? 0.0 : gam / scal[S_PQ];
    const double eta = first ? del : del - beta * gam;
    scal[S_RZ] = rho;
    scal[S_GAMMA] = gam;
    scal[S_DELTA] = del;
    scal[S_BETA] = beta;
    scal[S_PQ] = eta;
    scal[S_ALPHA] = rho / eta;
  });
}

void launch_spmv_dot3(const DevMat<double>& A, const double* z, double* w, const double* r,
                      const double* q, int first, const RedWork& rw, double* scal,
                      cudaStream_t s) {
  launch_dep(k_spmv_dot3, rw.grid, kBlock, 0, s, A, z, w, r, q, first, rw, scal);
}

// Ends an iteration of a solve in a loop (thread 0 of the last block; rr is
// its r.r, p the scalars): the tests of the host loop in api.cu, with the same
// operations, so both take the same number of iterations.  Far from the
// tolerance the square roots and the division (some 1.5 us of dependent FP64
// instructions) are left out: rr > rtol^2 b.b with a margin no rounding spans
// while rtol^2 is a normal number (below, it loses bits or is 0).
// The one-reduction form (FCG) also needs a finite alpha.
struct LoopScalars {
  double it, pq, err, bb, rtol, maxit, alpha;
};
__device__ __forceinline__ LoopScalars loop_scalars(const double* scal) {
  return LoopScalars{__ldcg(scal + S_IT), __ldcg(scal + S_PQ),    __ldcg(scal + S_ERR),
                     __ldcg(scal + S_BB), __ldcg(scal + S_RTOL),  __ldcg(scal + S_MAXIT),
                     __ldcg(scal + S_ALPHA)};
}
template <bool FCG>
__device__ __forceinline__ void pcg_continue(cudaGraphConditionalHandle h, double* scal, double rr,
                                             const LoopScalars& p) {
  if (!h) return;
  const double it = p.it + 1.0;
  scal[S_IT] = it;
  const bool ok = p.err == 0.0 && isfinite(p.pq) && isfinite(rr) && p.pq > 0.0 &&
                  (!FCG || isfinite(p.alpha));
  bool above = p.rtol >= 1e-150 && rr > 1.0001 * (p.rtol * p.rtol) * p.bb;
  if (!above) above = !(sqrt(rr) / sqrt(p.bb) <= p.rtol);
  cudaGraphSetConditional(h, ok && above && it < p.maxit ? 1u : 0u);
}

__global__ void k_pcg_begin(double* scal, cudaGraphConditionalHandle h) {
  scal[S_ALPHA] = scal[S_BETA] = scal[S_IT] = 0.0;
  scal[S_PQ] = 1.0;
  scal[S_RZ] = INFINITY;
  const double bb = scal[S_BB];
  cudaGraphSetConditional(h, bb > 0.0 && isfinite(bb) ? 1u : 0u);
}

void launch_pcg_begin(double* scal, cudaGraphConditionalHandle h, cudaStream_t s) {
  k_pcg_begin<<<1, 1, 0, s>>>(scal, h);
  count_launch();
}

// p = z - beta p, q = w - beta q (first: p = z, q = w), x += alpha p,
// r -= alpha q, r.r (S_RR)
__global__ void __launch_bounds__(kBlock) k_fcg_update(int64_t n, const double* z,
                                                       const double* w, double* __restrict__ p,
                                                       double* __restrict__ q,
                                                       double* __restrict__ x,
                                                       double* __restrict__ r, int first,
                                                       const RedWork rw, double* scal,
                                                       const PcgLoop loop) {
  pdl_wait();
  pdl_go();
  if (loop.x) x = *loop.x;
  const double alpha = ldv<false>(scal + S_ALPHA), beta = ldv<false>(scal + S_BETA);
  double acc = 0.0;
  for (int64_t i = (int64_t)blockIdx.x * kBlock + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * kBlock) {
    const double pi = first ? z[i] : fma(-beta, p[i], z[i]);
    const double qi = first ? w[i] : fma(-beta, q[i], w[i]);
    p[i] = pi;
    q[i] = qi;
    x[i] = fma(alpha, pi, x[i]);
    const double ri = fma(-alpha, qi, r[i]);
    r[i] = ri;
    acc = fma(ri, ri, acc);
  }
  grid_sum(
      acc, rw, [&] { return loop_scalars(scal); },
      [&](double tot, const LoopScalars& ls) {
        scal[S_RR] = tot;
        pcg_continue<true>(loop.handle, scal, tot, ls);
      });
}

void launch_fcg_update(int64_t n, const double* z, const double* w, double* p, double* q,
                       double* x, double* r, int first, const RedWork& rw, double* scal,
                       cudaStream_t s, const PcgLoop& loop) {
  launch_dep(k_fcg_update, rw.grid, kBlock, 0, s, n, z, w, p, q, x, r, first, rw, scal, loop);
}

// r -= alpha q ; r.r (S_RR).  The x update of the same iteration is deferred
// to k_xpay_x, which reads p anyway.  FAM >= 0: also the first step from zero
// of the next V-cycle's smoother (the same operations as its own launch; in the
// stored-operator form that is c = M^{-1} r), which saves that launch and its
// read of r.
template <class FT, int FAM>
__global__ void __launch_bounds__(kBlock, kRedBlocksPerSm) k_r_update(int64_t n, const double* q,
                                                                      double* r, const RedWork w,
                                                                      double* scal,
                                                                      const RFirst<FT> f,
                                                                      cudaGraphConditionalHandle h) {
  pdl_wait();
  pdl_go();
  const double alpha = ldv<false>(scal + S_ALPHA);
  double acc = 0.0;
  const uint32_t m = (uint32_t)n, step = gridDim.x * kBlock;  // n < 2^31: i + 2 step fits
  auto one = [&](uint32_t i, double qi, double ri) {
    ri = fma(-alpha, qi, ri);
    r[i] = ri;
    const FT bi = (FT)ri;
    if constexpr (sizeof(FT) == 4) f.fout[i] = bi;
    if constexpr (FAM >= 0) {
      first_value<FT, FAM>(i, bi, __ldg(f.dinv + i), f.rout, f.zout, f.xout, f.c2, f.beta, f.rhoinv);
    }
    acc = fma(ri, ri, acc);
  };
  uint32_t i = blockIdx.x * kBlock + threadIdx.x;
  for (; i + step < m; i += 2 * step) {
    const double q0 = ldv<false>(q + i), r0 = ldv<false>(r + i);
    const double q1 = ldv<false>(q + i + step), r1 = ldv<false>(r + i + step);
    one(i, q0, r0);
    one(i + step, q1, r1);
  }
  if (i < m) one(i, ldv<false>(q + i), ldv<false>(r + i));
  grid_sum(
      acc, w, [&] { return loop_scalars(scal); },
      [&](double tot, const LoopScalars& ls) {
        scal[S_RR] = tot;
        pcg_continue<false>(h, scal, tot, ls);
      });
}

template <class FT>
void launch_r_update(int64_t n, const double* q, double* r, const RedWork& w, double* scal,
                     cudaStream_t s, const RFirst<FT>& f, const PcgLoop& loop) {
  auto* k = f.fam < 0              ? k_r_update<FT, -1>
            : f.fam == FAM_CHEB4   ? k_r_update<FT, FAM_CHEB4>
            : f.fam == FAM_CHEB1   ? k_r_update<FT, FAM_CHEB1>
                                   : k_r_update<FT, FAM_JAC>;
  launch_dep(k, w.grid, kBlock, 0, s, n, q, r, w, scal, f, loop.handle);
}
template void launch_r_update<double>(int64_t, const double*, double*, const RedWork&, double*,
                                      cudaStream_t, const RFirst<double>&, const PcgLoop&);
template void launch_r_update<float>(int64_t, const double*, double*, const RedWork&, double*,
                                     cudaStream_t, const RFirst<float>&, const PcgLoop&);

// x += alpha p with the previous alpha, then p = z + beta p (x_beta = 1), or
// only x += alpha p (x_beta = 0: the last iteration)
template <class ZT>
__global__ void __launch_bounds__(kBlock) k_xpay_x(int64_t n, const ZT* z, double* p,
                                                   double* x, const double* scal, int with_p,
                                                   double* const* xslot) {
  pdl_wait();
  pdl_go();
  if (xslot) x = *xslot;
  const double alpha = ldv<false>(scal + S_ALPHA), beta = ldv<false>(scal + S_BETA);
  const int64_t i = (int64_t)blockIdx.x * kBlock + threadIdx.x;
  if (i >= n) return;
  const double pi = ldv<false>(p + i), xi = ldv<false>(x + i);
  const double zi = with_p ? (double)ldv<false>(z + i) : 0.0;
  x[i] = fma(alpha, pi, xi);
  if (with_p) p[i] = fma(beta, pi, zi);
}

template <class ZT>
void launch_xpay_x(int64_t n, const ZT* z, double* p, double* x, const double* scal, int with_p,
                   cudaStream_t s, const PcgLoop& loop) {
  if (n == 0) return;
  launch_dep(k_xpay_x<ZT>, (unsigned)((n + kBlock - 1) / kBlock), kBlock, 0, s, n, z, p, x, scal,
             with_p, loop.x);
}
template void launch_xpay_x<double>(int64_t, const double*, double*, double*, const double*, int,
                                    cudaStream_t, const PcgLoop&);
template void launch_xpay_x<float>(int64_t, const float*, double*, double*, const double*, int,
                                   cudaStream_t, const PcgLoop&);

template <class BT>
__global__ void __launch_bounds__(kBlock, kRedBlocksPerSm) k_dot(int64_t n, const double* a,
                                                                 const BT* b,
                                                const RedWork w, double* scal, int slot,
                                                int rz_shift) {
  pdl_wait();
  pdl_go();
  double acc = 0.0;
  const int64_t step = (int64_t)gridDim.x * kBlock;
  for (int64_t i0 = (int64_t)blockIdx.x * kBlock + threadIdx.x; i0 < n; i0 += kLoads * step) {
    double av[kLoads];
    BT bv[kLoads];
#pragma unroll
    for (int k = 0; k < kLoads; ++k) {
      const int64_t i = i0 + k * step;
      if (i < n) {
        av[k] = ldv<false>(a + i);
        bv[k] = ldv<false>(b + i);
      }
    }
#pragma unroll
    for (int k = 0; k < kLoads; ++k)
      if (i0 + k * step < n) acc = fma(av[k], (double)bv[k], acc);
  }
  struct Old {
    double rz, rzp;
  };
  grid_sum(
      acc, w, [&] { return Old{__ldcg(scal + S_RZ), __ldcg(scal + S_RZP)}; },
      [&](double tot, const Old& old) {
        if (rz_shift) {
          scal[S_RZOLD] = old.rz;
          scal[S_RZ] = tot;
          scal[S_BETA] = (rz_shift == 2 ? tot - old.rzp : tot) / old.rz;
        } else {
          scal[slot] = tot;
        }
      });
}

template <class BT>
void launch_dot(int64_t n, const double* a, const BT* b, const RedWork& w, double* scal,
                int out_slot, int rz_mode, cudaStream_t s) {
  launch_dep(k_dot<BT>, w.grid, kBlock, 0, s, n, a, b, w, scal, out_slot, rz_mode);
}
template void launch_dot<double>(int64_t, const double*, const double*, const RedWork&, double*, int,
                                 int, cudaStream_t);
template void launch_dot<float>(int64_t, const double*, const float*, const RedWork&, double*, int,
                                int, cudaStream_t);

__global__ void __launch_bounds__(kBlock) k_sub(int64_t n, const double* x, const double* y,
                                                double* out) {
  const int64_t i = (int64_t)blockIdx.x * kBlock + threadIdx.x;
  pdl_wait();
  pdl_go();
  if (i < n) out[i] = ldv<false>(x + i) - ldv<false>(y + i);
}

void launch_sub(int64_t n, const double* x, const double* y, double* out, cudaStream_t s) {
  if (n == 0) return;
  launch_dep(k_sub, (unsigned)((n + kBlock - 1) / kBlock), kBlock, 0, s, n, x, y, out);
}

__global__ void __launch_bounds__(kBlock) k_scale_dev(int64_t n, const double* x, double* out,
                                                      const double* sd, int stride,
                                                      double factor) {
  pdl_wait();
  pdl_go();
  const double f = factor / ldv<false>(sd + blockIdx.y * stride);
  const int64_t i = (int64_t)blockIdx.x * kBlock + threadIdx.x, o = blockIdx.y * n;
  if (i < n) out[o + i] = f * ldv<false>(x + o + i);
}

void launch_scale_dev(int64_t n, const double* x, double* out, const double* s_dev, int stride,
                      double factor, int nvec, cudaStream_t s) {
  if (n == 0) return;
  launch_dep(k_scale_dev, dim3((unsigned)((n + kBlock - 1) / kBlock), nvec), kBlock, 0, s, n, x,
             out, s_dev, stride, factor);
}

// Coarsest level: x = A_c^{-1} b with the inverse formed at load time from the
// Cholesky factor (FP64).  One warp per row, lanes stride the columns.
constexpr int kGemvVecs = 4;  // vectors of a batch per warp (one read of the row)
template <class XT>
__global__ void __launch_bounds__(kBlock) k_coarse_gemv(int nc, const double* __restrict__ ainv,
                                                        const XT* b, XT* x, int nvec) {
  const int lane = threadIdx.x & 31;
  const int i = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  if (i >= nc) return;
  const int v0 = blockIdx.y * kGemvVecs;
  const size_t o = (size_t)v0 * nc;
  coarse_gemv_row<XT, false, true>(i, nc, ainv, b + o, x + o, lane, min(kGemvVecs, nvec - v0));
}

template <class XT>
void launch_coarse_gemv(int nc, const double* ainv, const XT* b, XT* x, int nvec,
                        cudaStream_t s) {
  if (nc == 0) return;
  const int gy = (nvec + kGemvVecs - 1) / kGemvVecs, blk = small_block((int64_t)nc * 32 * gy);
  const dim3 g(blocks_of((int64_t)nc * 32, blk), gy);
  launch_dep(k_coarse_gemv<XT>, g, blk, 0, s, nc, ainv, b, x, nvec);
}

// Dense Cholesky A = L L^T (right-looking, one block, in place in `work`,
// row-major), then A^{-1} column by column (forward and back substitution),
// written row-major into ainv (A^{-1} is symmetric).  status = 1 if a pivot is
// not positive.  Set-up only: runs once per hierarchy load.
__global__ void __launch_bounds__(1024) k_chol_inverse(int n, double* L, double* ainv,
                                                      int* status) {
  __shared__ double piv;
  for (int j = 0; j < n; ++j) {
    if (threadIdx.x == 0) {
      const double d = L[(size_t)j * n + j];
      if (!(d > 0.0)) {
        *status = 1;
        piv = -1.0;
      } else {
        piv = sqrt(d);
        L[(size_t)j * n + j] = piv;
      }
    }
    __syncthreads();
    if (piv < 0.0) return;
    for (int i = j + 1 + threadIdx.x; i < n; i += blockDim.x) L[(size_t)i * n + j] /= piv;
    __syncthreads();
    const int64_t m = n - j - 1;
    const int64_t npairs = m * (m + 1) / 2;
    for (int64_t q = threadIdx.x; q < npairs; q += blockDim.x) {
      int64_t ii = (int64_t)((sqrt(8.0 * (double)q + 1.0) - 1.0) * 0.5);
      while (ii * (ii + 1) / 2 > q) --ii;
      while ((ii + 1) * (ii + 2) / 2 <= q) ++ii;
      const int64_t kk = q - ii * (ii + 1) / 2;
      const int64_t i = j + 1 + ii, k = j + 1 + kk;
      L[i * n + k] -= L[i * n + j] * L[k * n + j];
    }
    __syncthreads();
  }
  for (int c = threadIdx.x; c < n; c += blockDim.x) {
    double* y = ainv + (size_t)c * n;
    for (int i = 0; i < n; ++i) {
      if (i < c) {
        y[i] = 0.0;
        continue;
      }
      double s = (i == c) ? 1.0 : 0.0;
      for (int k = c; k < i; ++k) s -= L[(size_t)i * n + k] * y[k];
      y[i] = s / L[(size_t)i * n + i];
    }
    for (int i = n - 1; i >= 0; --i) {
      double s = y[i];
      for (int k = i + 1; k < n; ++k) s -= L[(size_t)k * n + i] * y[k];
      y[i] = s / L[(size_t)i * n + i];
    }
  }
}

void launch_chol_inverse(int n, double* work, double* ainv, int* status, cudaStream_t s) {
  k_chol_inverse<<<1, 1024, 0, s>>>(n, work, ainv, status);
  count_launch();
}

// w = M^{-1} A v and ||w||^2 into scal[S_NRM] (one power-iteration product).
template <class VT, class XT>
__global__ void __launch_bounds__(kBlock, 4) k_power_step(const DevMat<VT> A,
                                                       const XT* __restrict__ v,
                                                       const XT* __restrict__ dinv,
                                                       XT* __restrict__ w, const RedWork rw,
                                                       double* scal) {
  const int lane = threadIdx.x & 31;
  const int64_t nw = (int64_t)gridDim.x * kWarpsPerBlock;
  double acc = 0.0;
  for (int64_t s = (int64_t)blockIdx.x * kWarpsPerBlock + (threadIdx.x >> 5); s < A.nslices;
       s += nw) {
    const int64_t row = s * kSlice + lane;
    const XT t = row_spmv<1, VT, XT>(A, s, lane, row, v, XT(0));
    if (row < A.n) {
      const XT wi = t * dinv[row];
      w[row] = wi;
      acc += (double)wi * (double)wi;
    }
  }
  grid_sum(acc, rw, [&](double tot) { scal[S_NRM] = tot; });
}

template <class VT, class XT>
void launch_power_step(const DevMat<VT>& A, const XT* v, const XT* dinv, XT* w, const RedWork& rw,
                       double* scal, cudaStream_t s) {
  k_power_step<VT, XT><<<rw.grid, kBlock, 0, s>>>(A, v, dinv, w, rw, scal);
  count_launch();
}

template <class XT>
__global__ void __launch_bounds__(kBlock) k_scale_by_norm(int64_t n, const XT* __restrict__ w,
                                                          XT* __restrict__ v,
                                                          const double* __restrict__ scal,
                                                          int slot) {
  const double inv = 1.0 / sqrt(scal[slot]);
  const int64_t i = (int64_t)blockIdx.x * kBlock + threadIdx.x;
  if (i < n) v[i] = XT((double)w[i] * inv);
}

template <class XT>
void launch_scale_by_norm(int64_t n, const XT* w, XT* v, const double* scal, int slot,
                          cudaStream_t s) {
  if (n == 0) return;
  k_scale_by_norm<XT><<<(unsigned)((n + kBlock - 1) / kBlock), kBlock, 0, s>>>(n, w, v, scal,
                                                                                slot);
  count_launch();
}

template <class XT>
__global__ void __launch_bounds__(kBlock) k_norm2(int64_t n, const XT* __restrict__ v,
                                                  const RedWork rw, double* scal, int slot) {
  double acc = 0.0;
  for (int64_t i = (int64_t)blockIdx.x * kBlock + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * kBlock)
    acc += (double)v[i] * (double)v[i];
  grid_sum(acc, rw, [&](double tot) { scal[slot] = tot; });
}

template <class XT>
void launch_norm2(int64_t n, const XT* v, const RedWork& rw, double* scal, int slot,
                  cudaStream_t s) {
  k_norm2<XT><<<rw.grid, kBlock, 0, s>>>(n, v, rw, scal, slot);
  count_launch();
}

template void launch_coarse_gemv<double>(int, const double*, const double*, double*, int,
                                         cudaStream_t);
template void launch_coarse_gemv<float>(int, const double*, const float*, float*, int,
                                        cudaStream_t);
template void launch_power_step<double, double>(const DevMat<double>&, const double*, const double*,
                                                double*, const RedWork&, double*, cudaStream_t);
template void launch_power_step<float, float>(const DevMat<float>&, const float*, const float*,
                                                float*, const RedWork&, double*, cudaStream_t);
template void launch_power_step<__nv_bfloat16, float>(const DevMat<__nv_bfloat16>&, const float*,
                                                      const float*, float*, const RedWork&,
                                                      double*, cudaStream_t);
template void launch_scale_by_norm<double>(int64_t, const double*, double*, const double*, int,
                                           cudaStream_t);
template void launch_scale_by_norm<float>(int64_t, const float*, float*, const double*, int,
                                          cudaStream_t);
template void launch_norm2<double>(int64_t, const double*, const RedWork&, double*, int,
                                   cudaStream_t);
template void launch_norm2<float>(int64_t, const float*, const RedWork&, double*, int,
                                  cudaStream_t);

}  // namespace amgps
