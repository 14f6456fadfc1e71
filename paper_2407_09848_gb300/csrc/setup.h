// Device CSR and the launchers of the hierarchy set-up kernels
// (kernels_setup.cu): smoothed-aggregation prolongator and Galerkin product.
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

namespace amgps {

// Most distinct columns a row of a sparse product (or of a transpose: narrow
// and wide) may have in each form of the kernels.
enum GemmForm { kTiny = 0, kSmall = 1, kNarrow = 2, kWide = 3 };
constexpr int kRowMaxTiny = 96;
constexpr int kRowMaxSmall = 384;
constexpr int kRowMaxNarrow = 768;
constexpr int kRowMaxWide = 6144;

struct DevCsr {
  int64_t n_rows = 0, n_cols = 0, nnz = 0;
  int32_t* rowptr = nullptr;
  int32_t* col = nullptr;
  double* val = nullptr;
};

// C = A B.  fill = false: counts[i] = distinct columns of row i of C.
// fill = true: C.rowptr set from those counts; writes C.col (ascending per
// row) and C.val.  *err = 1 if a row exceeds the form's column limit.
void launch_spgemm(const DevCsr& A, const DevCsr& B, int32_t* counts, const DevCsr& C, int* err,
                   bool fill, GemmForm form, int nsm, cudaStream_t s);
// Dense form of C = A B for B.n_cols <= kDenseMaxCols: same results as the
// hashed forms (bitwise), no row limit.
// Up to kDenseFirst columns it is the first choice (a row's scan over all the
// columns is then no longer than over a table); up to kDenseMaxCols it takes
// the place of the wide form.
constexpr int64_t kDenseFirst = 1024;
constexpr int64_t kDenseMaxCols = 16384;
void launch_spgemm_dense(const DevCsr& A, const DevCsr& B, int32_t* counts, const DevCsr& C,
                         int* err, bool fill, int nsm, cudaStream_t s);
// rowptr[0..n] from the n counts; sums: scan_blocks(n) + 1 entries, the last one
// then holds the total
int64_t scan_blocks(int64_t n);
void launch_scan(int64_t n, const int32_t* cnt, int32_t* rowptr, int64_t* sums, cudaStream_t s);
// row pointers and values of n rows with one unit entry each
void launch_unit_rows(int64_t n, int32_t* rowptr, double* val, cudaStream_t s);
// diag[i] = a_ii and per-block maxima of sum_j |a_ij| / a_ii into part[];
// returns the number of blocks (partials)
int launch_rowstat(const DevCsr& A, double* diag, double* part, int nsm, cudaStream_t s);
// in place on A P_hat: entries become [j == agg_i] - omega (1/a_ii) (A P_hat)_ij
void launch_sa_combine(const DevCsr& AP, const int32_t* agg, const double* diag, double omega,
                       cudaStream_t s);
// transpose T = M^T: count entries per column, scatter with per-row cursors
// (from the prefix sums of the counts), then sort each row of T by column
void launch_col_count(int64_t nnz, const int32_t* col, int32_t* cnt, cudaStream_t s);
void launch_transpose_fill(const DevCsr& M, int32_t* cursor, const DevCsr& T, cudaStream_t s);
void launch_sort_rows(const DevCsr& T, int* err, bool wide, int nsm, cudaStream_t s);

}  // namespace amgps
