// Device helpers shared by the kernel translation units.
#pragma once

#include <utility>

#include "amgps_internal.h"

namespace amgps {

// Matrix values are streamed once per step: cache-streaming loads (evict-first
// in L1 and L2) keep them from displacing the vectors that neighbouring rows
// gather.  BF16 values are widened to FP32.
__device__ __forceinline__ double ldval(const double* p) { return __ldcs(p); }
__device__ __forceinline__ float ldval(const float* p) { return __ldcs(p); }
__device__ __forceinline__ float ldval(const __nv_bfloat16* p) {
  unsigned short s = __ldcs(reinterpret_cast<const unsigned short*>(p));
  return __bfloat162float(__ushort_as_bfloat16(s));
}

template <class T>
__device__ __forceinline__ T absv(T v) { return v < T(0) ? -v : v; }

// ---- programmatic dependent launch ----
// The kernels of a V-cycle and of the outer solver are launched so that their
// blocks may start while the previous kernel of the stream still runs
// (launch_dep below).  pdl_wait() returns when that kernel has finished and
// its writes are visible; before it a kernel may only read what no kernel of
// the chain writes -- the matrix arrays, the aggregate maps, 1/M -- and may
// write nothing.  pdl_go() lets the next kernel's blocks start; it comes
// after the wait, so at most two kernels of a chain overlap.
__device__ __forceinline__ void pdl_wait() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
}
__device__ __forceinline__ void pdl_go() {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}
// For kernels that only stream vectors, one row a thread: of one resident wave
// (eight blocks on each SM) or less.  The instruction costs 0.37 ns a block, one
// block after another, and beyond a wave that is more than a start under such a
// kernel's tail gives: 2.1 million rows (8192 blocks) 9.1 us with it, 5.3
// without, 8.2 as an ordinary launch; one FP32 step on 128^3 30.3 / 19.5 / 24.9 us.
__device__ __forceinline__ void pdl_go_one_wave() {
  if (gridDim.x * gridDim.y <= 8 * 152) pdl_go();
}

// Load of a vector entry.  CG = false: a plain cached load, issued where it
// stands (volatile: neither the compiler nor the read-only path may move it
// before pdl_wait).  CG = true: an L2 (coherent) load, for the persistent
// kernel that reads in one phase what other blocks wrote in an earlier phase
// of the same launch.
__device__ __forceinline__ double ldg_ca(const double* p) {
  double v;
  asm volatile("ld.global.f64 %0, [%1];" : "=d"(v) : "l"(__cvta_generic_to_global(p)));
  return v;
}
__device__ __forceinline__ float ldg_ca(const float* p) {
  float v;
  asm volatile("ld.global.f32 %0, [%1];" : "=f"(v) : "l"(__cvta_generic_to_global(p)));
  return v;
}
template <bool CG, class T>
__device__ __forceinline__ T ldv(const T* p) {
  if constexpr (CG) return __ldcg(p);
  else return ldg_ca(p);
}

// Slice descriptor (constant while any kernel runs): one 16-byte load.
__device__ __forceinline__ SliceDesc ld_desc(const SliceDesc* p) {
  const int4 v = __ldg(reinterpret_cast<const int4*>(p));
  SliceDesc d;
  d.vbase = (int64_t)(uint32_t)v.x | ((int64_t)v.y << 32);
  d.w = v.z;
  d.cref = v.w;
  return d;
}

// init() + SIGN * (A u)_row over the entries k in [k0, k1) of row `row`
// (position `lane` in slice `s`), in storage order (SIGN = +1 or -1, so a
// residual b - A u comes out of the same multiply-adds).  Rows past n (tail
// of the last slice) see only zero padding and clamped, in-range columns.
// FP64 arithmetic is the scarce resource on this GPU (its FP64 pipe issues
// about 2 FMAs per clock per SM), so the row costs exactly one multiply-add
// per stored entry and nothing else.
// WAIT: the kernel's pdl_wait() / pdl_go() happen here, after the first
// entries of the row (values and columns) are on their way and before
// init(), which loads the row's own vector entries: what a dependent launch
// still has to wait for is then one round of vector loads.  On the levels of a
// few thousand rows, where a kernel is three dependent loads long, that is
// most of its time.  Rows of other lengths go NB entries at a time; PIPE (the
// kernels of wide rows): the next NB values and columns are fetched while the
// current products are formed.  U8 (the split step): rows of a uniform slice,
// which load no columns, go eight at a time instead (FP64, 100,000 rows of 251
// in a band, 4 warps a slice, four steps and the call: 258 -> 226 us).
template <int SIGN, class VT, class XT, bool CG, bool WAIT, int NB, bool PIPE, bool U8 = false,
          class Init>
__device__ __forceinline__ XT row_accumulate(const DevMat<VT>& A, const SliceDesc d, int lane,
                                             int64_t row, const XT* u, Init init, int k0, int k1) {
  const int64_t nm1 = A.n - 1;
  auto fetch = [&](int k, XT& av, int32_t& cv) {
    const int64_t e = d.vbase + (int64_t)k * kSlice + lane;
    av = XT(ldval(A.val + e));
    if (d.cref >= 0) {
      const int64_t cc = row + (int64_t)__ldg(A.off + d.cref + k);
      cv = (int32_t)(cc < 0 ? 0 : (cc > nm1 ? nm1 : cc));
    } else {
      cv = __ldg(A.col + e);
    }
  };
  if (k1 - k0 == 7) {
    // the seven entries of a 7-point row without guards: on GB300's narrow
    // FP64 pipe a predicated-off multiply-add still takes an issue slot
    // (same operations in the same order as the general loop below)
    XT a[7], uv[7];
    int32_t c[7];
#pragma unroll
    for (int kk = 0; kk < 7; ++kk) fetch(k0 + kk, a[kk], c[kk]);
    if constexpr (WAIT) {
      pdl_wait();
      pdl_go();
    }
    XT t = init();
#pragma unroll
    for (int kk = 0; kk < 7; ++kk) uv[kk] = ldv<CG>(u + c[kk]);
#pragma unroll
    for (int kk = 0; kk < 7; ++kk) t = fma(SIGN > 0 ? a[kk] : -a[kk], uv[kk], t);
    return t;
  }
  auto batches = [&](auto nb, auto pipe) {
    constexpr int N = decltype(nb)::value;
    constexpr bool kAhead = decltype(pipe)::value;
    XT a[N];
    int32_t c[N];
    auto fetch_batch = [&](int kb) {
#pragma unroll
      for (int kk = 0; kk < N; ++kk)
        if (kb + kk < k1) fetch(kb + kk, a[kk], c[kk]);
    };
    fetch_batch(k0);
    if constexpr (WAIT) {
      pdl_wait();
      pdl_go();
    }
    XT t = init();
    for (int kb = k0; kb < k1; kb += N) {
      XT av[N], uv[N];
#pragma unroll
      for (int kk = 0; kk < N; ++kk) {
        if (kb + kk < k1) uv[kk] = ldv<CG>(u + c[kk]);
        av[kk] = a[kk];
      }
      if (kAhead && kb + N < k1) fetch_batch(kb + N);
#pragma unroll
      for (int kk = 0; kk < N; ++kk)
        if (kb + kk < k1) t = fma(SIGN > 0 ? av[kk] : -av[kk], uv[kk], t);
      if (!kAhead && kb + N < k1) fetch_batch(kb + N);
    }
    return t;
  };
  if constexpr (U8) {
    if (d.cref >= 0) return batches(std::integral_constant<int, 8>{}, std::false_type{});
  }
  return batches(std::integral_constant<int, NB>{}, std::integral_constant<bool, PIPE>{});
}

// The same sum with the entries of a row shared by E lanes of a warp: lane
// q R + r (R = 32 / E) takes entries k0 + q, k0 + q + E, ... of row r0 + r of the
// slice (r0 = `first`), the E partial sums are then added over the lanes, and
// every lane of a row ends with its sum.  init() counts in lanes q = 0 only.
template <int SIGN, int E, class Init>
__device__ __forceinline__ double row_accumulate_wide(const DevMat<double>& A, const SliceDesc d,
                                                      int first, int64_t row0, const double* u,
                                                      Init init, int k0, int k1) {
  constexpr int R = 32 / E, NB = 4;
  const int lane = threadIdx.x & 31, r = lane % R, q = lane / R;
  const int64_t nm1 = A.n - 1, row = row0 + r;
  const double* val = A.val + d.vbase + first + r;
  double a[NB];
  int32_t c[NB];
  auto fetch = [&](int kb) {
#pragma unroll
    for (int j = 0; j < NB; ++j) {
      const int k = kb + j * E;
      if (k < k1) {
        a[j] = ldval(val + (int64_t)k * kSlice);
        if (d.cref >= 0) {
          const int64_t cc = row + (int64_t)__ldg(A.off + d.cref + k);
          c[j] = (int32_t)(cc < 0 ? 0 : (cc > nm1 ? nm1 : cc));
        } else {
          c[j] = __ldg(A.col + d.vbase + first + r + (int64_t)k * kSlice);
        }
      }
    }
  };
  fetch(k0 + q);
  pdl_wait();
  pdl_go();
  double t = init();
  for (int kb = k0 + q; kb < k1; kb += NB * E) {
    double av[NB], uv[NB];
#pragma unroll
    for (int j = 0; j < NB; ++j) {
      if (kb + j * E < k1) uv[j] = ldv<false>(u + c[j]);
      av[j] = a[j];
    }
    fetch(kb + NB * E);
#pragma unroll
    for (int j = 0; j < NB; ++j)
      if (kb + j * E < k1) t = fma(SIGN > 0 ? av[j] : -av[j], uv[j], t);
  }
  __syncwarp();
#pragma unroll
  for (int o = R; o < 32; o *= 2) t += __shfl_xor_sync(0xffffffffu, t, o);
  return t;
}

// The whole row: entries 0 .. w-1 of the slice.
template <int SIGN, class VT, class XT>
__device__ __forceinline__ XT row_spmv(const DevMat<VT>& A, int64_t s, int lane, int64_t row,
                                       const XT* u, XT init) {
  const SliceDesc d = ld_desc(A.sd + s);
  return row_accumulate<SIGN, VT, XT, false, false, 4, false>(
      A, d, lane, row, u, [&] { return init; }, 0, d.w);
}

// The SpMV of one smoother step is accumulated as init + SIGN * (A u):
// r_j = r_{j-1} - A z_j directly for the 4th kind, the 1st-kind initial step
// and Jacobi (init = r_in, SIGN = -1); the plain product t = A d for the
// other 1st-kind steps (init = 0, SIGN = +1).
// The stored-operator steps add their operator's products to the vector terms
// (FAM_OP) or subtract the row-scaled products from q (FAM_OPT).
template <int FAM, bool INIT>
struct StepForm {
  static constexpr bool kResidual = !(FAM == FAM_CHEB1 && !INIT);
  static constexpr int kSign = FAM == FAM_OP ? 1 : (kResidual ? -1 : 1);
};

// Whether a step reads 1/M: every step but the residual, the scaled
// 4th-kind step with scaled rin and the stored-operator steps.
template <int FAM>
__device__ __forceinline__ constexpr bool step_needs_dinv() {
  return FAM != FAM_RES && FAM != FAM_CHEB4S && FAM != FAM_CHEB1S && !is_op(FAM);
}

// Stored-operator steps: the vector terms the accumulation starts from
// (s0 = slot-0 entry of the row, s1 = slot-1 entry), then the stores.  A
// FAM_OPT step whose slot 0 is still the unscaled right-hand side (rin_raw)
// scales it itself: c = M^{-1} b needs no pass of its own.
template <class VT, class XT, int FAM, bool INIT, bool WR, bool ZOWN>
__device__ __forceinline__ XT op_init(const StepArgs<VT, XT>& a, int64_t row, XT s0, XT s1) {
  XT acc = XT(0);
  if constexpr (FAM == FAM_OPT) {
    acc = a.rin_raw ? s0 * __ldg(a.dinv + row) : s0;
  } else {
    if constexpr (INIT) acc = WR ? s0 : a.c2 * s0;
    if constexpr (ZOWN) acc = INIT ? fma(a.c1, s1, acc) : a.c1 * s1;
  }
  return acc;
}
template <class VT, class XT, int FAM, bool WR>
__device__ __forceinline__ void op_finish(const StepArgs<VT, XT>& a, int64_t row, XT acc, XT ucen) {
  a.zout[row] = acc;
  if constexpr (FAM == FAM_OPT && WR) a.rout[row] = fma(a.beta, acc, ucen);
}

// Starting value of the accumulation: rin for the residual forms ((1/M) rin
// when a scaled step's rin is still unscaled), 0 otherwise.
template <int FAM, bool RESID, class XT>
__device__ __forceinline__ XT step_init(XT rin, XT di) {
  if constexpr (!RESID) return XT(0);
  else if constexpr (FAM == FAM_CHEB4SR || FAM == FAM_CHEB1SR) return rin * di;
  else return rin;
}

// Epilogue of one smoother step for one row, given the accumulated SpMV and
// the row's own vector entries (see kernels_smooth.cu for the recurrences).
template <class VT, class XT, int FAM, bool INIT, bool WR, bool ZOWN>
__device__ __forceinline__ void step_finish(const StepArgs<VT, XT>& a, int64_t row, XT acc, XT rin,
                                            XT xin, XT di, XT zo) {
  if constexpr (is_cheb4(FAM)) {
    const XT r = acc;  // r_j, or M^{-1} r_j in the scaled forms
    if (WR) a.rout[row] = r;
    XT z;
    if constexpr (FAM == FAM_CHEB4) z = a.c2 * (r * di);
    else z = a.c2 * r;
    if (ZOWN) z = fma(a.c1, zo, z);
    a.zout[row] = z;
    a.xout[row] = fma(a.beta, z, xin);
  } else if constexpr (FAM == FAM_CHEB1) {
    XT r;
    if (INIT) r = a.rhoinv * (acc * di);
    else r = fma(-(a.rhoinv * di), acc, rin);
    if (WR) a.rout[row] = r;
    XT z = a.c2 * r;
    if (ZOWN) z = fma(a.c1, zo, z);
    a.zout[row] = z;
    a.xout[row] = xin + z;
  } else if constexpr (FAM == FAM_CHEB1S || FAM == FAM_CHEB1SR) {
    const XT r = acc;  // rho M^{-1} r
    if (WR) a.rout[row] = r;
    XT z = a.c2 * r;  // c2 carries the 1/rho
    if (ZOWN) z = fma(a.c1, zo, z);
    a.zout[row] = z;
    a.xout[row] = xin + z;
  } else if constexpr (FAM == FAM_JAC) {
    a.xout[row] = fma(acc, di, xin);
  } else {
    a.zout[row] = acc;  // FAM_RES: the true residual b - A x
  }
}

// One smoother step on the 32 rows of slice s, one row per lane, operands
// read from global memory (the direct form of the step).  WAIT: see
// row_accumulate (1/M is fetched before the wait as well).
template <class VT, class XT, int FAM, bool INIT, bool WR, bool ZOWN, bool CG = false,
          bool WAIT = false>
__device__ __forceinline__ void step_slice(const StepArgs<VT, XT>& a, int64_t s, int lane) {
  const int64_t row = s * kSlice + lane;
  const bool live = row < a.A.n;
  const SliceDesc d = ld_desc(a.A.sd + s);
  constexpr int kSign = StepForm<FAM, INIT>::kSign;
  if constexpr (is_op(FAM)) {
    XT uc = XT(0);
    const XT acc = row_accumulate<kSign, VT, XT, CG, WAIT, sizeof(XT) == 8 ? 4 : 8, WAIT && sizeof(XT) == 8>(
        a.A, d, lane, row, a.u,
        [&] {
          XT s0 = XT(0), s1 = XT(0);
          if (live) {
            if (reads_slot0<FAM, INIT>()) s0 = ldv<CG>(a.rin + row);
            if (reads_slot1<FAM, ZOWN>()) s1 = ldv<CG>(a.xin + row);
            if (FAM == FAM_OPT && WR) uc = ldv<CG>(a.u + row);
          }
          return op_init<VT, XT, FAM, INIT, WR, ZOWN>(a, live ? row : 0, s0, s1);
        },
        0, d.w);
    if (live) op_finish<VT, XT, FAM, WR>(a, row, acc, uc);
    return;
  }
  XT rin = XT(0), xin = XT(0), zo = XT(0), di = XT(0);
  if (live && step_needs_dinv<FAM>()) di = __ldg(a.dinv + row);  // formed at set-up
  const XT acc = row_accumulate<kSign, VT, XT, CG, WAIT, sizeof(XT) == 8 ? 4 : 8, WAIT && sizeof(XT) == 8>(
      a.A, d, lane, row, a.u,
      [&] {
        if (live) {
          rin = ldv<CG>(a.rin + row);
          if (FAM != FAM_RES) xin = ldv<CG>(a.xin + row);
          if (ZOWN) zo = ldv<CG>(a.zown + row);
        }
        return step_init<FAM, StepForm<FAM, INIT>::kResidual>(rin, di);
      },
      0, d.w);
  if (!live) return;
  step_finish<VT, XT, FAM, INIT, WR, ZOWN>(a, row, acc, rin, xin, di, zo);
}

// The same step for vectors v0 .. v1-1 of a batch (vector v at +v n of every
// vector argument): a 7-point slice loads its values, columns and 1/M once for
// all of them.  Each vector's operations and their order are those of
// step_slice.
template <class VT, class XT, int FAM, bool INIT, bool WR, bool ZOWN>
__device__ __forceinline__ void step_slice_mv(const StepArgs<VT, XT>& a, int64_t s, int lane,
                                              int v0, int v1) {
  const int64_t n = a.A.n, row = s * kSlice + lane;
  const SliceDesc d = ld_desc(a.A.sd + s);
  constexpr int kSign = StepForm<FAM, INIT>::kSign;
  if (d.w == 7) {
    // a lane past n works on row n - 1 and stores nothing
    const bool live = row < n;
    const int64_t lr = live ? row : n - 1;
    XT av[7];
    int32_t cv[7];
#pragma unroll
    for (int k = 0; k < 7; ++k) {
      const int64_t e = d.vbase + (int64_t)k * kSlice + lane;
      av[k] = XT(__ldg(a.A.val + e));
      if (d.cref >= 0) {
        const int64_t cc = row + (int64_t)__ldg(a.A.off + d.cref + k);
        cv[k] = (int32_t)(cc < 0 ? 0 : (cc > n - 1 ? n - 1 : cc));
      } else {
        cv[k] = __ldg(a.A.col + e);
      }
    }
    XT di = XT(0);
    if (step_needs_dinv<FAM>()) di = __ldg(a.dinv + lr);
    pdl_wait();
    pdl_go();
    for (int v = v0; v < v1; ++v) {
      const int64_t o = v * n, ro = o + lr;
      XT rin = XT(0), xin = XT(0), zo = XT(0), uc = XT(0), uv[7], t;
      if constexpr (is_op(FAM)) {
        if (reads_slot0<FAM, INIT>()) rin = ldv<false>(a.rin + ro);
        if (reads_slot1<FAM, ZOWN>()) xin = ldv<false>(a.xin + ro);
        if (FAM == FAM_OPT && WR) uc = ldv<false>(a.u + ro);
      } else {
        rin = ldv<false>(a.rin + ro);
        if (FAM != FAM_RES) xin = ldv<false>(a.xin + ro);
        if (ZOWN) zo = ldv<false>(a.zown + ro);
      }
      const XT* u = a.u + o;
#pragma unroll
      for (int k = 0; k < 7; ++k) uv[k] = ldv<false>(u + cv[k]);
      if constexpr (is_op(FAM)) t = op_init<VT, XT, FAM, INIT, WR, ZOWN>(a, lr, rin, xin);
      else t = step_init<FAM, StepForm<FAM, INIT>::kResidual>(rin, di);
#pragma unroll
      for (int k = 0; k < 7; ++k) t = fma(kSign > 0 ? av[k] : -av[k], uv[k], t);
      if (live) {
        if constexpr (is_op(FAM)) op_finish<VT, XT, FAM, WR>(a, ro, t, uc);
        else step_finish<VT, XT, FAM, INIT, WR, ZOWN>(a, ro, t, rin, xin, di, zo);
      }
    }
    return;
  }
  pdl_wait();
  pdl_go();
  for (int v = v0; v < v1; ++v) {
    StepArgs<VT, XT> b = a;
    const int64_t o = v * n;
    b.u += o;
    if (b.rin) b.rin += o;
    if (b.rout) b.rout += o;
    if (b.zown) b.zown += o;
    if (b.zout) b.zout += o;
    if (b.xin) b.xin += o;
    if (b.xout) b.xout += o;
    step_slice<VT, XT, FAM, INIT, WR, ZOWN>(b, s, lane);
  }
}

// Per-element bodies of the elementwise V-cycle kernels, shared by their own
// launches (kernels_smooth.cu, kernels_krylov.cu) and by the persistent
// coarse-level kernel (kernels_cycle.cu), so both give the same bits.

// First step from x = 0 (no product with A), row i, with di = 1/M_i:
//   4th kind: z_1 = c2 M^{-1} b, x = beta_1 z_1 (r_0 = b is not copied)
//   1st kind: r^(0) = (1/rho) M^{-1} b, d^(0) = r^(0)/theta, x = d^(0)
//   Jacobi:   x = M^{-1} b
template <class XT, int FAM>
__device__ __forceinline__ void first_value(int64_t i, XT bi, XT di, XT* rout, XT* zout, XT* xout,
                                            XT c2, XT beta, XT rhoinv) {
  const XT bm = bi * di;
  if constexpr (FAM == FAM_CHEB4) {
    const XT z = c2 * bm;
    zout[i] = z;
    xout[i] = beta * z;
  } else if constexpr (FAM == FAM_CHEB1) {
    const XT r = rhoinv * bm;
    rout[i] = r;
    const XT z = c2 * r;
    zout[i] = z;
    xout[i] = z;
  } else {
    xout[i] = bm;
  }
}
template <class XT, int FAM, bool CG = false>
__device__ __forceinline__ void first_row(int64_t i, const XT* b, XT di, XT* rout, XT* zout,
                                          XT* xout, XT c2, XT beta, XT rhoinv) {
  first_value<XT, FAM>(i, ldv<CG>(b + i), di, rout, zout, xout, c2, beta, rhoinv);
}

// b_c[I] = sum of res over the children of coarse row I, in list order.  The
// first eight children (all of a 2x2x2 block) are looked up before the wait
// and loaded together.
template <class XT, bool CG = false, bool WAIT = false>
__device__ __forceinline__ void aggregate_row(int64_t I, const int32_t* cptr, const int32_t* cidx,
                                              const XT* res, XT* bc) {
  const int q0 = __ldg(cptr + I), q1 = __ldg(cptr + I + 1);
  int32_t c[8];
#pragma unroll
  for (int k = 0; k < 8; ++k)
    if (q0 + k < q1) c[k] = __ldg(cidx + q0 + k);
  if constexpr (WAIT) {
    pdl_wait();
    pdl_go();
  }
  XT v[8];
#pragma unroll
  for (int k = 0; k < 8; ++k)
    if (q0 + k < q1) v[k] = ldv<CG>(res + c[k]);
  XT acc = XT(0);
#pragma unroll
  for (int k = 0; k < 8; ++k)
    if (q0 + k < q1) acc += v[k];
  for (int q = q0 + 8; q < q1; ++q) acc += ldv<CG>(res + __ldg(cidx + q));
  bc[I] = acc;
}

// x_i += e_c[agg_i]
template <class XT, bool CG = false, bool WAIT = false>
__device__ __forceinline__ void prolong_row(int64_t i, const int32_t* agg, const XT* ec, XT* x) {
  const int32_t c = __ldg(agg + i);
  if constexpr (WAIT) {
    pdl_wait();
    pdl_go();
  }
  const XT xi = ldv<CG>(x + i);
  x[i] = xi + ldv<CG>(ec + c);
}

// Row i of the coarse correction (see CorrArgs).  Z: z is wanted (a guarded
// multiplication would take an FP64 issue slot all the same: 256^3 solve 85.0 ->
// 83.7 ms without it).
template <bool Z, bool CG = false, bool WAIT = false>
__device__ __forceinline__ void correct_row(const CorrArgs& a, int64_t i, int64_t v) {
  const int64_t at = (i >> 5) * (kCorrEntries * kSlice) + (i & 31);
  double w[kCorrEntries], e[kCorrEntries];
  int32_t c[kCorrEntries];
  const uint32_t code = __ldcs(a.m.code + i);
  c[0] = __ldg(a.m.agg + i);
#pragma unroll
  for (int k = 0; k < kCorrEntries; ++k) w[k] = __ldcs(a.m.val + at + kSlice * k);
  const double di = __ldg(a.dinv + i);
#pragma unroll
  for (int k = 1; k < kCorrEntries; ++k)
    c[k] = c[0] + __ldg(a.m.delta + ((code >> (10 * (k - 1))) & (kCorrTable - 1)));
  if constexpr (WAIT) {
    pdl_wait();
    pdl_go();
  }
  const int64_t j = v * a.n + i;
  const double* ev = a.e + v * a.nc;
  const double r = ldv<CG>(a.r + j), x = ldv<CG>(a.x + j);
#pragma unroll
  for (int k = 0; k < kCorrEntries; ++k) e[k] = ldv<CG>(ev + c[k]);
  double s = r * di;
#pragma unroll
  for (int k = 0; k < kCorrEntries; ++k) s = fma(-w[k], e[k], s);
  const double x0 = x + e[0];
  if (a.x0out) a.x0out[j] = x0;
  if (a.sout) a.sout[j] = s;
  if constexpr (Z) {
    s *= a.c2;
    a.zout[j] = s;
  }
  a.xout[j] = fma(a.beta, s, x0);
}

// x_i = (A_c^{-1} b)_i for the coarsest level, one warp per row: lane l sums
// columns l, l + 32, ... in order, then a fixed butterfly adds the lanes.  The
// first 16 entries of a lane (512 columns) are loaded together, before the
// wait, and serve all nv vectors (vector v at b + v nc, x + v nc).  Columns past
// 512 go kMore at a time: one by one, a lane waited for each (1024 columns, one
// product and the call 8.9 us, so 7.0).
template <class XT, bool CG = false, bool WAIT = false>
__device__ __forceinline__ void coarse_gemv_row(int i, int nc, const double* ainv, const XT* b,
                                                XT* x, int lane, int nv = 1) {
  constexpr int kMore = 8;
  const double* row = ainv + (size_t)i * nc;
  double av[16];
#pragma unroll
  for (int k = 0; k < 16; ++k)
    if (lane + 32 * k < nc) av[k] = __ldg(row + lane + 32 * k);
  if constexpr (WAIT) {
    pdl_wait();
    pdl_go();
  }
  for (int v = 0; v < nv; ++v, b += nc, x += nc) {
    XT bv[16];
#pragma unroll
    for (int k = 0; k < 16; ++k)
      if (lane + 32 * k < nc) bv[k] = ldv<CG>(b + lane + 32 * k);
    double acc = 0.0;
#pragma unroll
    for (int k = 0; k < 16; ++k)
      if (lane + 32 * k < nc) acc = fma(av[k], (double)bv[k], acc);
    for (int j0 = lane + 512; j0 < nc; j0 += 32 * kMore) {
      double a2[kMore];
      XT b2[kMore];
#pragma unroll
      for (int k = 0; k < kMore; ++k)
        if (j0 + 32 * k < nc) {
          a2[k] = __ldg(row + j0 + 32 * k);
          b2[k] = ldv<CG>(b + j0 + 32 * k);
        }
#pragma unroll
      for (int k = 0; k < kMore; ++k)
        if (j0 + 32 * k < nc) acc = fma(a2[k], (double)b2[k], acc);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if (lane == 0) x[i] = XT(acc);
  }
}

// Sum over a block of kBlock threads; result valid in warp 0.  One warp adds
// the values (eight a lane in thread order, then a butterfly): 12 FP64 warp
// instructions of 16 clocks on the SM's one narrow pipe, where a butterfly in
// each of the eight warps takes 45.
__device__ __forceinline__ double block_sum(double v, double* sh) {
  __syncthreads();
  sh[threadIdx.x] = v;
  __syncthreads();
  if (threadIdx.x >= 32) return 0.0;
  v = sh[threadIdx.x];
#pragma unroll
  for (int k = 1; k < kWarpsPerBlock; ++k) v += sh[threadIdx.x + 32 * k];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Deterministic grid-wide sum: each block writes its partial, the last block to
// arrive adds the partials in index order with a fixed tree and thread 0 calls
// fin(total, pre()), with pre() -- the scalars fin needs -- loaded beside the
// partials; then the counter is re-armed.  The grid size is a pure function of
// the problem size, so the result is bitwise reproducible.  (The whole block
// adds the partials: one warp alone, without block barriers, was slower, 32^3
// solve 736 against 721 us.)
template <class Pre, class Fin>
__device__ __forceinline__ void grid_sum(double v, const RedWork& w, Pre pre, Fin fin) {
  __shared__ double sh[kBlock];
  __shared__ bool last;
  const double b = block_sum(v, sh);
  if (threadIdx.x == 0) {
    w.part[blockIdx.x] = b;
    __threadfence();
    last = atomicAdd(w.counter, 1u) == gridDim.x - 1;
  }
  __syncthreads();
  if (!last) return;
  __threadfence();
  const auto pr = pre();
  double s = 0.0;
  for (int i = threadIdx.x; i < (int)gridDim.x; i += kBlock) s += __ldcg(w.part + i);
  s = block_sum(s, sh);
  if (threadIdx.x == 0) {
    fin(s, pr);
    *w.counter = 0u;
  }
}
template <class Fin>
__device__ __forceinline__ void grid_sum(double v, const RedWork& w, Fin fin) {
  grid_sum(v, w, [] { return 0; }, [&](double s, int) { fin(s); });
}

// Threads per block of a kernel of `threads` one-row threads (or lanes): 256,
// fewer on levels that would leave SMs without a block -- an SM issues one FP64
// warp instruction in 16 clocks, so the eight warps of a block take eight
// times one warp's time (4096-row level: 0.5 us of FP64 issue on 16 SMs, 0.06
// on 128).
// (GB300's SMs as a fixed number: it also decides how many lanes share a wide
// row, and with that an order of summation, which is not the device's affair.)
constexpr int kSms = 152;
inline int small_block(int64_t threads) {
  const int64_t warps = (threads + 31) / 32, per = (warps + kSms - 1) / kSms;
  return 32 * (int)(per < 1 ? 1 : per > kWarpsPerBlock ? kWarpsPerBlock : per);
}
inline unsigned blocks_of(int64_t threads, int block) {
  return (unsigned)((threads + block - 1) / block);
}

// Launch of a kernel that calls pdl_wait() as the programmatic dependent of
// the kernel before it on stream s (in a captured graph: a programmatic
// edge).  Behind anything but a kernel (a copy, a memset, an event) it is an
// ordinary launch.
template <class... P, class... A>
void launch_dep(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t s,
                A&&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  cudaLaunchKernelEx(&cfg, kernel, std::forward<A>(args)...);
  count_launch();
}

}  // namespace amgps
