// gqt_slices.h -- FP64 matrix products by integer slices on the tensor cores
// (gqt_slices.cu).
#pragma once

#include <cuda_runtime.h>

#include <cstddef>

namespace gqt {

constexpr int SLICES = 7;     // base-256 digits of a value
constexpr int SLICE_K = 16;   // contraction elements per chunk
constexpr int SLICE_WAIT = 1 << 24;  // polls of a device wait where no handle sets them

// A matrix of `rows` rows (K-major) in `planes` real planes, sliced:
// [plane * SLICES + slice][chunk][row][16] FP16.
struct SliceOperand {
  const void* data;
  int rows, planes;
};

// n results of the same shape; result p is the sum over its terms of A-plane a[p][t]
// times the transpose of B-plane b[p][t], negated where neg[p][t].
struct SliceParts {
  int n, terms;
  int a[2][2], b[2][2], neg[2][2];
};

size_t slice_bytes(int rows, int planes, int nchunk);
// Largest biased exponents of the rows of x [rows][k] times weights w [k].
void launch_row_exps(const double* x, int rows, size_t k, const double* w, int* exps, cudaStream_t st);
// The same exponents of the complex rows of x0 and x1 [rows][k], and how unevenly their
// values spread: spread[r] = (2^exponent / rms) / n^(1/4) over the row's nonzero values, n
// of them (complex) in a sum of `chunk` elements; infinite for a row with an infinity or a
// NaN or nothing but denormals.  An entry whose two spreads multiply to more than
// SLICE_SPREAD is summed more exactly by FP64 multiply-adds over such chunks than by
// slices.  exps, spread: [x0's rows, x1's rows]; scratch: row_spread_bytes.
constexpr float SLICE_SPREAD = 5.f;
size_t row_spread_bytes(int rows, size_t k);
void launch_row_spreads(const double* x0, const double* x1, int rows, size_t k, double chunk, void* scratch, int* exps,
                        float* spread, cudaStream_t st);
// Slices of elements [k0, k0 + 16 nchunk) of each row (zeros past k).
void launch_slice_rows(const double* x, int comp, int rows, size_t stride, size_t k, size_t k0, const double* w,
                       int nchunk, const int* exps, void* out, cudaStream_t st);
// Slices of cos(n acos(E_e / dE)), n < m, rows e < ne, at scale 2^0 (zeros where |E| >= dE).
void launch_cos_slices(const double* E, int ne, double dE, int m, int nchunk, void* out, cudaStream_t st);
int slice_splits(int rows_a, int rows_b, int parts, int nchunk);
// out[split][part][rows_a][rows_b] (+)= the products of the scaled rows: times
// 2^(exp_a - 1022 + exp_b - 1022) for the true values.  *err: bit 16 where a device
// wait of `limit` polls gave up, 32 where the drain after it did.
void launch_slice_gemm(const SliceOperand& a, const SliceOperand& b, const SliceParts& parts, int nchunk, int splits,
                       double* out, bool add, int* err, int limit, cudaStream_t st);

}  // namespace gqt
