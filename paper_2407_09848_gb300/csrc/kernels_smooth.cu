// Smoother, transfer and conversion kernels of the V-cycle (Sec. 2 and 3).
//
// One launch of k_step is one degree step of a polynomial smoother: the SpMV
// with the current recurrence vector, the residual update, the l1-Jacobi
// scaling and the recurrence / solution updates share a single pass over A and
// the vectors (the fusion Sec. 3 obtains with its psb_upd_xyz kernel):
//
//   4th kind (Eq. polsmoother / polsmootheropt), step producing z_{j+1}:
//     t = A z_j ; r_j = r_{j-1} - t
//     z_{j+1} = c1 z_j + c2 M^{-1} r_j         c1 = (2j-1)/(2j+3), c2 = (8j+4)/(2j+3)/rho
//     x += beta_{j+1} z_{j+1}
//   1st kind (Algorithm 1), step producing d^(j):
//     t = A d^(j-1) ; r^(j) = r^(j-1) - (1/rho) M^{-1} t
//     d^(j) = rho_j rho_{j-1} d^(j-1) + (2 rho_j/delta) r^(j) ; x += d^(j)
//   l1-Jacobi sweep: x_new = x + M^{-1}(b - A x)
//
// D^{-1} = 1/M (Eq. l1smooth) is formed once per level (re-deriving M_i from
// the row plus an IEEE division every step would cost about four times the
// FP64 instructions of the whole step).  On FP64 and FP32 levels the
// polynomial steps go further and run on the row-scaled values a_ij / M_i with
// the residual kept as M^{-1} r (rho M^{-1} r for the 1st kind): the families
// FAM_CHEB4S/SR and FAM_CHEB1S/SR, which need no 1/M product or stream except
// where rin is still b.  The row's own vectors are loaded before the SpMV so
// their latency overlaps it.  z ping-pongs between two buffers because
// neighbouring rows gather z_j in the same launch that writes z_{j+1}.  Levels
// with wide rows use the split form (several warps per slice).
#include <type_traits>

#include "kernels_common.cuh"

namespace amgps {

template <class VT, class XT, int FAM, bool INIT, bool WR, bool ZOWN>
__global__ void __launch_bounds__(kBlock, 4) k_step(const StepArgs<VT, XT> a) {
  const int lane = threadIdx.x & 31;
  int64_t s = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  if (a.slices) {
    if (s >= a.nlist) return;
    s = __ldg(a.slices + s);
  } else if (s >= a.A.nslices) {
    return;
  }
  step_slice<VT, XT, FAM, INIT, WR, ZOWN, false, true>(a, s, lane);
}

// Vectors of a batch that one warp takes through its slice: the 7-point values
// (56 B a row, more than half of a step's bytes) are then read once for four
// vectors, and the step is bound by FP64 issue alone.
constexpr int kVecs = 4;
template <class VT, class XT, int FAM, bool INIT, bool WR, bool ZOWN>
__global__ void __launch_bounds__(kBlock, 4) k_step_mv(const StepArgs<VT, XT> a) {
  const int64_t s = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  if (s >= a.A.nslices) return;
  const int v0 = blockIdx.y * kVecs;
  step_slice_mv<VT, XT, FAM, INIT, WR, ZOWN>(a, s, threadIdx.x & 31, v0, min(v0 + kVecs, a.nvec));
}

// Split form for levels with wide rows: one block per slice, a.split warps;
// warp g sums entries [g w / G, (g+1) w / G) of each row, warp 0 adds the
// partials in warp order (deterministic) and finishes the rows.
template <class VT, class XT, int FAM, bool INIT, bool WR, bool ZOWN>
__global__ void __launch_bounds__(32 * kMaxSplit) k_step_split(const StepArgs<VT, XT> a) {
  __shared__ XT part[kMaxSplit][32];
  const int lane = threadIdx.x & 31, g = threadIdx.x >> 5, G = blockDim.x >> 5;
  int64_t s = blockIdx.x;
  if (a.slices) {
    if (s >= a.nlist) return;
    s = __ldg(a.slices + s);
  } else if (s >= a.A.nslices) {
    return;
  }
  const int64_t row = s * kSlice + lane;
  const bool live = row < a.A.n;
  const int64_t o = (int64_t)blockIdx.y * a.A.n, ro = o + row;  // vector of a batch
  using F = StepForm<FAM, INIT>;
  const bool own = live && g == 0;
  XT rin = XT(0), xin = XT(0), zo = XT(0);
  const XT di = (own && step_needs_dinv<FAM>()) ? __ldg(a.dinv + row) : XT(0);
  const SliceDesc d = ld_desc(a.A.sd + s);
  const int k0 = (int)((int64_t)d.w * g / G), k1 = (int)((int64_t)d.w * (g + 1) / G);
  // FP32 values go eight at a time, not ahead (300,000 rows of 125, 4 warps a slice,
  // four steps and the call: 281 us four ahead, 250 so; BF16 410 and 442)
  constexpr int kBatch = std::is_same<VT, float>::value ? 8 : 4;
  part[g][lane] = row_accumulate<F::kSign, VT, XT, false, true, kBatch, kBatch == 4, sizeof(VT) == 8>(
      a.A, d, lane, row, a.u + o,
      [&] {
        if (!own) return XT(0);
        rin = ldv<false>(a.rin + ro);
        if (FAM != FAM_RES) xin = ldv<false>(a.xin + ro);
        if (ZOWN) zo = ldv<false>(a.zown + ro);
        return step_init<FAM, F::kResidual>(rin, di);
      },
      k0, k1);
  __syncthreads();
  if (!own) return;
  XT acc = part[0][lane];
  for (int q = 1; q < G; ++q) acc += part[q][lane];
  step_finish<VT, XT, FAM, INIT, WR, ZOWN>(a, ro, acc, rin, xin, di, zo);
}

// Split form of the FP64 levels with too few slices for the SMs: a slice's 32
// rows are also shared out over E blocks (R = 32 / E rows each), E lanes of a
// warp working on one row, so the split of the level is E x G.  With one block
// per slice the 54 slices of a 1728-row level of 573 entries a row kept 54 SMs
// busy, their FP64 pipes alone for 5 us; four steps there take 39.0 us instead of
// 47.5 (call included).  Where one block per slice fills the SMs the shorter
// runs of a row's values cost more than they give (432 slices: 56.3 us instead
// of 51.3), so E is the smallest with two blocks an SM.  G warps of a block
// share the rows' entries (G = 1: a block holds kWideUnits independent units).
constexpr int kWideLanes = 8;  // the largest E
constexpr int kWideUnits = 4;
struct WideShape {
  int E, G, units;  // lanes per row, warps per unit, units per block
};
inline WideShape wide_shape(int split, int64_t nslices) {
  WideShape w;
  w.E = 1;
  while (w.E < kWideLanes && w.E < split && nslices * w.E < 2 * kSms) w.E *= 2;
  w.G = split / w.E;
  w.units = w.G == 1 ? kWideUnits : 1;
  return w;
}

// The part of a row sum that unit `unit` (a slice's rows first .. first + R-1)
// leaves to its warp 0: calls body(row, sum) for every row there.
template <int SIGN, int E, class Init, class Body>
__device__ __forceinline__ void wide_unit(const DevMat<double>& A, const double* u, int G, Init init,
                                          Body body) {
  constexpr int R = 32 / E;
  __shared__ double part[kMaxSplit / 2][R];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int g = G > 1 ? warp : 0;
  const int64_t nunits = A.nslices * E;
  const int64_t unit = G > 1 ? (int64_t)blockIdx.x : (int64_t)blockIdx.x * kWideUnits + warp;
  if (unit >= nunits) return;  // whole warps; G = 1 needs no block-wide meeting
  const int64_t s = unit / E;
  const int first = (int)(unit % E) * R;
  const SliceDesc d = ld_desc(A.sd + s);
  const int64_t row0 = s * kSlice + first, row = row0 + lane % R;
  const int k0 = (int)((int64_t)d.w * g / G), k1 = (int)((int64_t)d.w * (g + 1) / G);
  const bool own = g == 0 && lane < R && row < A.n;
  double t = row_accumulate_wide<SIGN, E>(
      A, d, first, row0, u, [&] { return own ? init(row) : 0.0; }, k0, k1);
  if (G > 1) {
    if (lane < R) part[g][lane] = t;
    __syncthreads();
    if (g == 0)
      for (int q = 1; q < G; ++q) t += part[q][lane % R];
  }
  if (own) body(row, t);
}

template <int E, int FAM, bool INIT, bool WR, bool ZOWN>
__global__ void __launch_bounds__(32 * (kMaxSplit / E)) k_step_wide(const StepArgs<double, double> a,
                                                              int G) {
  const int64_t o = (int64_t)blockIdx.y * a.A.n;  // vector of a batch
  using F = StepForm<FAM, INIT>;
  double rin = 0.0, xin = 0.0, zo = 0.0, di = 0.0;
  wide_unit<F::kSign, E>(
      a.A, a.u + o, G,
      [&](int64_t row) {
        if (step_needs_dinv<FAM>()) di = __ldg(a.dinv + row);
        rin = ldv<false>(a.rin + o + row);
        if (FAM != FAM_RES) xin = ldv<false>(a.xin + o + row);
        if (ZOWN) zo = ldv<false>(a.zown + o + row);
        return step_init<FAM, F::kResidual>(rin, di);
      },
      [&](int64_t row, double t) {
        step_finish<double, double, FAM, INIT, WR, ZOWN>(a, o + row, t, rin, xin, di, zo);
      });
}

template <int FAM, bool INIT, bool WR, bool ZOWN>
static void go_wide(const StepArgs<double, double>& a, const WideShape& w, cudaStream_t s) {
  const dim3 g((unsigned)((a.A.nslices * w.E + w.units - 1) / w.units), a.nvec);
  auto* k = w.E == 2   ? k_step_wide<2, FAM, INIT, WR, ZOWN>
            : w.E == 4 ? k_step_wide<4, FAM, INIT, WR, ZOWN>
                       : k_step_wide<8, FAM, INIT, WR, ZOWN>;
  launch_dep(k, g, 32 * w.G * w.units, 0, s, a, w.G);
}

template <class VT, class XT, int FAM, bool INIT, bool WR, bool ZOWN>
static void go(const StepArgs<VT, XT>& a, int64_t work, cudaStream_t s) {
  constexpr bool f64 = std::is_same<VT, double>::value && std::is_same<XT, double>::value;
  if constexpr (f64) {
    if (a.nvec > 1 && a.split == 1) {  // batches run on all slices
      const int gy = (a.nvec + kVecs - 1) / kVecs, blk = small_block(work * kSlice * gy);
      launch_dep(k_step_mv<VT, XT, FAM, INIT, WR, ZOWN>, dim3(blocks_of(work * kSlice, blk), gy), blk,
                 0, s, a);
      return;
    }
  }
  if constexpr (f64 && !is_op(FAM)) {  // FP32 rows keep their order of summation
    const WideShape w = wide_shape(a.split, work);
    if (w.E > 1) {
      go_wide<FAM, INIT, WR, ZOWN>(a, w, s);
      return;
    }
  }
  if (a.split > 1) {
    launch_dep(k_step_split<VT, XT, FAM, INIT, WR, ZOWN>, dim3((unsigned)work, a.nvec),
               32 * a.split, 0, s, a);
  } else {
    const int blk = small_block(work * kSlice);
    launch_dep(k_step<VT, XT, FAM, INIT, WR, ZOWN>, blocks_of(work * kSlice, blk), blk, 0, s, a);
  }
}

template <class VT, class XT, int FAM, bool INIT>
static void dispatch_wr(const StepArgs<VT, XT>& a, int64_t work, cudaStream_t s) {
  const bool z = a.zown != nullptr;
  if (a.write_r) {
    if (z) go<VT, XT, FAM, INIT, true, true>(a, work, s);
    else go<VT, XT, FAM, INIT, true, false>(a, work, s);
  } else {
    if (z) go<VT, XT, FAM, INIT, false, true>(a, work, s);
    else go<VT, XT, FAM, INIT, false, false>(a, work, s);
  }
}

// Stored-operator steps (FP64 levels, one warp per slice): the flags of
// FAM_OP / FAM_OPT from the arguments.
template <class VT, class XT>
static void dispatch_op(const StepArgs<VT, XT>& a, int64_t work, cudaStream_t s) {
  if constexpr (std::is_same<VT, double>::value && std::is_same<XT, double>::value) {
    const bool s0 = a.rin != nullptr, s1 = a.xin != nullptr, wr = a.write_r;
    if (a.fam == FAM_OPT) {
      if (wr) go<VT, XT, FAM_OPT, true, true, false>(a, work, s);
      else go<VT, XT, FAM_OPT, true, false, false>(a, work, s);
    } else if (!s0) {
      go<VT, XT, FAM_OP, false, false, false>(a, work, s);
    } else if (!s1) {
      if (wr) go<VT, XT, FAM_OP, true, true, false>(a, work, s);
      else go<VT, XT, FAM_OP, true, false, false>(a, work, s);
    } else {
      if (wr) go<VT, XT, FAM_OP, true, true, true>(a, work, s);
      else go<VT, XT, FAM_OP, true, false, true>(a, work, s);
    }
  }
}

template <class VT, class XT>
void launch_step(const StepArgs<VT, XT>& a, cudaStream_t s) {
  const int64_t work = a.slices ? a.nlist : a.A.nslices;
  if (work == 0) return;
  if (is_op(a.fam)) {
    dispatch_op<VT, XT>(a, work, s);
    return;
  }
  switch (a.fam) {
    case FAM_CHEB4:
      if (a.init) dispatch_wr<VT, XT, FAM_CHEB4, true>(a, work, s);
      else dispatch_wr<VT, XT, FAM_CHEB4, false>(a, work, s);
      break;
    case FAM_CHEB4S:
      dispatch_wr<VT, XT, FAM_CHEB4S, false>(a, work, s);
      break;
    case FAM_CHEB4SR:
      if (a.init) dispatch_wr<VT, XT, FAM_CHEB4SR, true>(a, work, s);
      else dispatch_wr<VT, XT, FAM_CHEB4SR, false>(a, work, s);
      break;
    case FAM_CHEB1S:
      dispatch_wr<VT, XT, FAM_CHEB1S, false>(a, work, s);
      break;
    case FAM_CHEB1SR:
      dispatch_wr<VT, XT, FAM_CHEB1SR, true>(a, work, s);
      break;
    case FAM_CHEB1:
      if (a.init) dispatch_wr<VT, XT, FAM_CHEB1, true>(a, work, s);
      else dispatch_wr<VT, XT, FAM_CHEB1, false>(a, work, s);
      break;
    case FAM_RES:
      go<VT, XT, FAM_RES, true, false, false>(a, work, s);
      break;
    default:
      go<VT, XT, FAM_JAC, true, false, false>(a, work, s);
  }
}

// First step from x = 0 (no product with A): first_row (kernels_common.cuh).
template <class XT, int FAM>
__global__ void __launch_bounds__(kBlock) k_first(int64_t n, const XT* b,
                                                  const XT* __restrict__ dinv, XT* rout, XT* zout,
                                                  XT* xout, XT c2, XT beta, XT rhoinv) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const XT di = dinv[i];
  pdl_wait();
  pdl_go_one_wave();
  const int64_t o = (int64_t)blockIdx.y * n;  // vector of a batch
  first_row<XT, FAM>(i, b + o, di, rout + o, zout + o, xout + o, c2, beta, rhoinv);
}

template <class XT>
void launch_first(int fam, int64_t n, const XT* b, const XT* dinv, XT* rout, XT* zout, XT* xout,
                  XT c2, XT beta, XT rhoinv, int nvec, cudaStream_t s) {
  if (n == 0) return;
  const int blk = small_block(n * nvec);
  const dim3 g(blocks_of(n, blk), nvec);
  auto* k = fam == FAM_CHEB4   ? k_first<XT, FAM_CHEB4>
            : fam == FAM_CHEB1 ? k_first<XT, FAM_CHEB1>
                               : k_first<XT, FAM_JAC>;
  launch_dep(k, g, blk, 0, s, n, b, dinv, rout, zout, xout, c2, beta, rhoinv);
}

// b_c = P^T res for an unsmoothed aggregation P (Sec. 2): one thread per coarse
// row adds the residuals of its children (cidx[cptr[I] .. cptr[I+1])) in list
// order, so the sum does not depend on scheduling.  The residual itself comes
// from the FAM_RES step (pipelined and coalesced like the smoother steps).
template <class XT>
__global__ void __launch_bounds__(kBlock, 6) k_aggregate(const int32_t* __restrict__ cptr,
                                                      const int32_t* __restrict__ cidx, int64_t n,
                                                      int64_t nc, const XT* res, XT* bc) {
  const int64_t I = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (I >= nc) return;
  aggregate_row<XT, false, true>(I, cptr, cidx, res + blockIdx.y * n, bc + blockIdx.y * nc);
}

template <class XT>
void launch_aggregate(const int32_t* cptr, const int32_t* cidx, int64_t n, int64_t nc,
                      const XT* res, XT* bc, int nvec, cudaStream_t s) {
  if (nc == 0) return;
  const int blk = small_block(nc * nvec);
  const dim3 g(blocks_of(nc, blk), nvec);
  launch_dep(k_aggregate<XT>, g, blk, 0, s, cptr, cidx, n, nc, res, bc);
}

// Residual, restriction and the coarse level's first step in one kernel (small
// levels): eight lanes per coarse row, one child each (more children: further
// rounds), the residuals added in list order through shuffles.  What it saves
// is two launches and the wait for each: 9 kernels a level instead of 11.  With
// small_block: 32^3 solve 785 -> 751 us, FP32 128^3 9680 -> 9393, V-cycle on
// 61x53x47 95.1 -> 89.8, gradients on 97x81x72 1315 -> 1268.
template <class VT, class XT>
__global__ void __launch_bounds__(kBlock, 2) k_restrict(const RestrictArgs<VT, XT> a) {
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int lane = threadIdx.x & 31, q = lane & 7;
  const int64_t I = min(t >> 3, a.nc - 1);  // lanes past the end repeat the last row
  const bool live = (t >> 3) < a.nc;
  const int64_t o = (int64_t)blockIdx.y * a.A.n, oc = (int64_t)blockIdx.y * a.nc;
  const int q0 = __ldg(a.cptr + I), q1 = __ldg(a.cptr + I + 1);
  const XT di = a.fam >= 0 ? __ldg(a.dinv + I) : XT(0);
  // the residual of child `at` (clamped to the list: every lane takes part)
  auto residual = [&](int at, auto wait) {
    const int64_t row = __ldg(a.cidx + min(at, q1 - 1));
    const SliceDesc d = ld_desc(a.A.sd + (row >> 5));
    return std::pair<int64_t, XT>(
        row, row_accumulate<-1, VT, XT, false, decltype(wait)::value, sizeof(XT) == 8 ? 4 : 8,
                            false>(a.A, d, (int)(row & 31), row, a.u + o,
                                   [&] { return ldv<false>(a.b + o + row); }, 0, d.w));
  };
  XT acc = XT(0);
  // one round per eight children of the warp's longest list (the same number
  // for all its lanes: they meet in the shuffles)
  const int rounds = (__reduce_max_sync(0xffffffffu, q1 - q0) + 7) / 8;
  for (int k = 0; k < rounds; ++k) {
    const int at = q0 + 8 * k + q;
    const auto res = k == 0 ? residual(at, std::true_type{}) : residual(at, std::false_type{});
    if (live && at < q1) a.r[o + res.first] = res.second;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const XT v = __shfl_sync(0xffffffffu, res.second, (lane & ~7) + j);
      if (q0 + 8 * k + j < q1) acc += v;
    }
  }
  if (!live || q != 0) return;
  a.bc[oc + I] = acc;
  if (a.fam < 0) return;
  XT *ro = a.rout + oc, *zo = a.zout + oc, *xo = a.xout + oc;
  if (a.fam == FAM_CHEB4) first_value<XT, FAM_CHEB4>(I, acc, di, ro, zo, xo, a.c2, a.beta, a.rhoinv);
  else if (a.fam == FAM_CHEB1)
    first_value<XT, FAM_CHEB1>(I, acc, di, ro, zo, xo, a.c2, a.beta, a.rhoinv);
  else first_value<XT, FAM_JAC>(I, acc, di, ro, zo, xo, a.c2, a.beta, a.rhoinv);
}

template <class VT, class XT>
void launch_restrict(const RestrictArgs<VT, XT>& a, int nvec, cudaStream_t s) {
  const int64_t threads = a.nc * 8;
  const int blk = small_block(threads * nvec);
  launch_dep(k_restrict<VT, XT>, dim3(blocks_of(threads, blk), nvec), blk, 0, s, a);
}
template void launch_restrict<double, double>(const RestrictArgs<double, double>&, int, cudaStream_t);
template void launch_restrict<float, float>(const RestrictArgs<float, float>&, int, cudaStream_t);
template void launch_restrict<__nv_bfloat16, float>(const RestrictArgs<__nv_bfloat16, float>&, int,
                                                    cudaStream_t);

// x += P e_c (gather through the aggregate map).
template <class XT>
__global__ void __launch_bounds__(kBlock) k_prolong(int64_t n, int64_t nc,
                                                    const int32_t* __restrict__ agg, const XT* ec,
                                                    XT* x) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) prolong_row<XT, false, true>(i, agg, ec + blockIdx.y * nc, x + blockIdx.y * n);
}

template <class XT>
void launch_prolong(int64_t n, int64_t nc, const int32_t* agg, const XT* ec, XT* x, int nvec,
                    cudaStream_t s) {
  if (n == 0) return;
  const int blk = small_block(n * nvec);
  const dim3 g(blocks_of(n, blk), nvec);
  launch_dep(k_prolong<XT>, g, blk, 0, s, n, nc, agg, ec, x);
}

template <class XT>
__global__ void __launch_bounds__(kBlock) k_add(int64_t n, const XT* x, const XT* y,
                                                XT* out) {
  const int64_t i = (int64_t)blockIdx.x * kBlock + threadIdx.x;
  pdl_wait();
  pdl_go();
  if (i < n) out[i] = x[i] + y[i];
}

template <class XT>
void launch_add(int64_t n, const XT* x, const XT* y, XT* out, cudaStream_t s) {
  if (n == 0) return;
  launch_dep(k_add<XT>, (unsigned)((n + kBlock - 1) / kBlock), kBlock, 0, s, n, x, y, out);
}

// 1/M_i with M_i of Eq. l1smooth (a_ii + sum_{j != i} |a_ij|), formed once per level.
template <class VT, class XT>
__global__ void __launch_bounds__(kBlock) k_l1diag(const DevMat<VT> A, XT* __restrict__ dinv) {
  const int lane = threadIdx.x & 31;
  const int64_t s = (int64_t)blockIdx.x * kWarpsPerBlock + (threadIdx.x >> 5);
  if (s >= A.nslices) return;
  const int64_t row = s * kSlice + lane;
  const SliceDesc d = A.sd[s];
  const int64_t nm1 = A.n - 1;
  XT m = XT(0);
  for (int k = 0; k < d.w; ++k) {
    const int64_t e = d.vbase + (int64_t)k * kSlice + lane;
    const XT a = XT(ldval(A.val + e));
    int64_t c;
    if (d.cref >= 0) {
      c = row + (int64_t)A.off[d.cref + k];
      c = c < 0 ? 0 : (c > nm1 ? nm1 : c);
    } else {
      c = A.col[e];
    }
    m += (c == row) ? a : absv(a);
  }
  if (row < A.n) dinv[row] = XT(1) / m;
}

template <class VT, class XT>
void launch_l1diag(const DevMat<VT>& A, XT* dinv, cudaStream_t s) {
  if (A.nslices == 0) return;
  dim3 g((unsigned)((A.nslices + kWarpsPerBlock - 1) / kWarpsPerBlock));
  k_l1diag<VT, XT><<<g, kBlock, 0, s>>>(A, dinv);
  count_launch();
}

// The coarse correction and first post-smoothing step, one row per thread.
// Streams 80 B a row (4 values, their code, aggregate, 1/M, r, x in; two
// vectors out) where the prolongation and the step with the full row moved
// 117; the gathered e is an eighth of the level and stays in L2.  256^3 solve
// 93.8 -> 90.0 ms, one V-cycle on 61x53x47 101.6 -> 95.8 us.
template <bool Z>
__global__ void __launch_bounds__(kBlock) k_correct(const CorrArgs a) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < a.n) correct_row<Z, false, true>(a, i, blockIdx.y);
}

void launch_correct(const CorrArgs& a, int nvec, cudaStream_t s) {
  if (a.n == 0) return;
  const int blk = small_block(a.n * nvec);
  launch_dep(a.zout ? k_correct<true> : k_correct<false>, dim3(blocks_of(a.n, blk), nvec), blk, 0, s, a);
}

// Set-up of M^{-1} A P, one row per lane of a slice: the row's entries are
// added to the slot of their aggregate in storage order; a slot's column is
// coded as the index of its offset from the row's own aggregate in `delta`
// (filled with atomicCAS; which index an offset gets changes no result).
__global__ void __launch_bounds__(kBlock) k_build_correct(const DevMat<double> B,
                                                          const int32_t* __restrict__ agg,
                                                          double* __restrict__ val,
                                                          uint32_t* __restrict__ code,
                                                          int32_t* delta, int* bad) {
  const int lane = threadIdx.x & 31;
  const int64_t s = (int64_t)blockIdx.x * kWarpsPerBlock + (threadIdx.x >> 5);
  if (s >= B.nslices) return;
  const int64_t row = s * kSlice + lane;
  const SliceDesc d = ld_desc(B.sd + s);
  double w[kCorrEntries] = {};
  int32_t c[kCorrEntries] = {};
  int used = 1;
  bool ok = true;
  uint32_t bits = 0;
  if (row < B.n) {
    c[0] = agg[row];
    for (int k = 0; k < d.w; ++k) {
      const int64_t e = d.vbase + (int64_t)k * kSlice + lane;
      const double a = B.val[e];
      if (a == 0.0) continue;  // padding (or an entry that adds nothing)
      const int64_t cc = d.cref >= 0 ? row + (int64_t)B.off[d.cref + k] : (int64_t)B.col[e];
      const int32_t g = agg[cc];
      bool found = false;
#pragma unroll
      for (int q = 0; q < kCorrEntries; ++q)
        if (!found && q < used && c[q] == g) {
          w[q] += a;
          found = true;
        }
      if (found) continue;
      if (used == kCorrEntries) {
        ok = false;
        break;
      }
#pragma unroll
      for (int q = 1; q < kCorrEntries; ++q)
        if (q == used) {
          c[q] = g;
          w[q] = a;
        }
      ++used;
    }
#pragma unroll
    for (int q = 1; q < kCorrEntries; ++q) {
      if (q >= used || !ok) continue;
      const int32_t dl = c[q] - c[0];
      uint32_t h = ((uint32_t)dl * 2654435761u) >> 22;
      int probes = 0;
      for (;; h = (h + 1) & (kCorrTable - 1)) {
        if (h != 0) {  // entry 0 stands for "own aggregate"
          const int32_t prev = atomicCAS(delta + h, kCorrEmpty, dl);
          if (prev == kCorrEmpty || prev == dl) break;
        }
        if (++probes > kCorrTable / 2) {
          ok = false;
          break;
        }
      }
      bits |= h << (10 * (q - 1));
    }
    code[row] = bits;
  }
#pragma unroll
  for (int q = 0; q < kCorrEntries; ++q)
    val[s * (kCorrEntries * kSlice) + q * kSlice + lane] = w[q];
  if (!ok) atomicExch(bad, 1);
}

void launch_build_correct(const DevMat<double>& B, const int32_t* agg, double* val, uint32_t* code,
                          int32_t* delta, int* bad, cudaStream_t s) {
  if (B.nslices == 0) return;
  k_build_correct<<<(unsigned)((B.nslices + kWarpsPerBlock - 1) / kWarpsPerBlock), kBlock, 0, s>>>(
      B, agg, val, code, delta, bad);
  count_launch();
}

// Operator values of one stored-operator step, m = tau I - sigma B, entry by
// entry of B's layout.  The row's diagonal slot: offset 0 of a uniform slice,
// else the first stored column equal to the row (explicit rows are sorted by
// column and padded after their entries).  Rows past n keep zeros.
__global__ void __launch_bounds__(kBlock) k_build_op(const DevMat<double> B, double tau,
                                                     double sigma, double* __restrict__ out) {
  const int lane = threadIdx.x & 31;
  const int64_t s = (int64_t)blockIdx.x * kWarpsPerBlock + (threadIdx.x >> 5);
  if (s >= B.nslices) return;
  const int64_t row = s * kSlice + lane;
  const SliceDesc d = B.sd[s];
  bool seen = false;
  for (int k = 0; k < d.w; ++k) {
    const int64_t e = d.vbase + (int64_t)k * kSlice + lane;
    bool dg;
    if (d.cref >= 0) {
      dg = B.off[d.cref + k] == 0;
    } else {
      dg = !seen && B.col[e] == row;
      seen = seen || dg;
    }
    const double v = B.val[e];
    out[e] = row < B.n ? (dg ? fma(-sigma, v, tau) : -sigma * v) : 0.0;
  }
}

void launch_build_op(const DevMat<double>& B, double tau, double sigma, double* out,
                     cudaStream_t s) {
  if (B.nslices == 0) return;
  dim3 g((unsigned)((B.nslices + kWarpsPerBlock - 1) / kWarpsPerBlock));
  k_build_op<<<g, kBlock, 0, s>>>(B, tau, sigma, out);
  count_launch();
}

template <class A, class B>
__global__ void __launch_bounds__(kBlock) k_convert(int64_t n, const A* in, B* out) {
  const int64_t i = (int64_t)blockIdx.x * kBlock + threadIdx.x;
  pdl_wait();
  pdl_go_one_wave();
  if (i < n) out[i] = B(in[i]);
}

template <class A, class B>
void launch_convert(int64_t n, const A* in, B* out, cudaStream_t s) {
  if (n == 0) return;
  launch_dep(k_convert<A, B>, (unsigned)((n + kBlock - 1) / kBlock), kBlock, 0, s, n, in, out);
}

#define AMGPS_INST(VT, XT)                                                                   \
  template void launch_step<VT, XT>(const StepArgs<VT, XT>&, cudaStream_t);                  \
  template void launch_l1diag<VT, XT>(const DevMat<VT>&, XT*, cudaStream_t);
AMGPS_INST(double, double)
AMGPS_INST(float, float)
AMGPS_INST(__nv_bfloat16, float)
#undef AMGPS_INST

template void launch_first<double>(int, int64_t, const double*, const double*, double*, double*,
                                   double*, double, double, double, int, cudaStream_t);
template void launch_first<float>(int, int64_t, const float*, const float*, float*, float*,
                                  float*, float, float, float, int, cudaStream_t);
template void launch_aggregate<double>(const int32_t*, const int32_t*, int64_t, int64_t, const double*,
                                       double*, int, cudaStream_t);
template void launch_aggregate<float>(const int32_t*, const int32_t*, int64_t, int64_t, const float*,
                                       float*, int, cudaStream_t);
template void launch_prolong<double>(int64_t, int64_t, const int32_t*, const double*, double*, int,
                                     cudaStream_t);
template void launch_add<double>(int64_t, const double*, const double*, double*, cudaStream_t);
template void launch_prolong<float>(int64_t, int64_t, const int32_t*, const float*, float*, int,
                                     cudaStream_t);
template void launch_convert<double, float>(int64_t, const double*, float*, cudaStream_t);
template void launch_convert<float, double>(int64_t, const float*, double*, cudaStream_t);
template void launch_convert<double, double>(int64_t, const double*, double*, cudaStream_t);

// Transfers through a general prolongator (explicit SELL-32, FP64 values):
// y = M u (add = 0) or y += M u (add = 1).  M = R = P^T restricts
// (b_c = P^T r), M = P prolongs (x += P x_c).  One warp per slice, or with
// split > 1 one block per slice whose warps share the row's entries (partials
// added in warp order).
template <class XT>
__global__ void __launch_bounds__(kBlock, 4) k_xfer(const DevMat<double> M, const XT* u, XT* y,
                                                 int add) {
  const int lane = threadIdx.x & 31;
  const int64_t s = (int64_t)blockIdx.x * kWarpsPerBlock + (threadIdx.x >> 5);
  if (s >= M.nslices) return;
  const int64_t row = s * kSlice + lane;
  const SliceDesc d = ld_desc(M.sd + s);
  const XT t = row_accumulate<1, double, XT, false, true, 8, false>(
      M, d, lane, row, u, [&] { return (add && row < M.n) ? ldv<false>(y + row) : XT(0); }, 0, d.w);
  if (row < M.n) y[row] = t;
}

template <class XT>
__global__ void __launch_bounds__(32 * kMaxSplit) k_xfer_split(const DevMat<double> M, const XT* u,
                                                               XT* y, int add) {
  __shared__ XT part[kMaxSplit][32];
  const int lane = threadIdx.x & 31, g = threadIdx.x >> 5, G = blockDim.x >> 5;
  const int64_t s = blockIdx.x;
  if (s >= M.nslices) return;
  const int64_t row = s * kSlice + lane;
  const bool live = row < M.n;
  const SliceDesc d = ld_desc(M.sd + s);
  const int k0 = (int)((int64_t)d.w * g / G), k1 = (int)((int64_t)d.w * (g + 1) / G);
  part[g][lane] = row_accumulate<1, double, XT, false, true, 4, true>(
      M, d, lane, row, u,
      [&] { return (add && live && g == 0) ? ldv<false>(y + row) : XT(0); }, k0, k1);
  __syncthreads();
  if (g != 0 || !live) return;
  XT t = part[0][lane];
  for (int q = 1; q < G; ++q) t += part[q][lane];
  y[row] = t;
}

template <int E>
__global__ void __launch_bounds__(32 * (kMaxSplit / E)) k_xfer_wide(const DevMat<double> M,
                                                              const double* u, double* y, int add,
                                                              int G) {
  wide_unit<1, E>(
      M, u, G, [&](int64_t row) { return add ? ldv<false>(y + row) : 0.0; },
      [&](int64_t row, double t) { y[row] = t; });
}

template <class XT>
void launch_xfer(const DevMat<double>& M, const XT* u, XT* y, int add, int split, cudaStream_t s) {
  if (M.nslices == 0) return;
  if constexpr (std::is_same<XT, double>::value) {
    const WideShape w = wide_shape(split, M.nslices);
    if (w.E > 1) {
      auto* k = w.E == 2 ? k_xfer_wide<2> : w.E == 4 ? k_xfer_wide<4> : k_xfer_wide<8>;
      launch_dep(k, (unsigned)((M.nslices * w.E + w.units - 1) / w.units), 32 * w.G * w.units, 0, s,
                 M, u, y, add, w.G);
      return;
    }
  }
  if (split > 1)
    launch_dep(k_xfer_split<XT>, (unsigned)M.nslices, 32 * split, 0, s, M, u, y, add);
  else
    launch_dep(k_xfer<XT>, (unsigned)((M.nslices + kWarpsPerBlock - 1) / kWarpsPerBlock), kBlock, 0,
               s, M, u, y, add);
}
template void launch_xfer<double>(const DevMat<double>&, const double*, double*, int, int,
                                  cudaStream_t);
template void launch_xfer<float>(const DevMat<double>&, const float*, float*, int, int,
                                 cudaStream_t);

}  // namespace amgps
