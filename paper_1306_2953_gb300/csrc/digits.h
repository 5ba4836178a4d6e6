// FP64- and FP32-accurate contractions on the tensor cores by integer digits
// (see digits.cu).  err (here and in linalg.h): a device word that becomes 1 once
// a bounded wait of the call has given up (its results are then NaN), or nullptr.
#pragma once

#include <cuda_runtime.h>

#include <cstdint>

namespace rs {

// Ints of scratch the overlap of nx and ny columns needs.
inline int64_t digit_gram_scratch_ints(int nx, int ny) { return (int64_t)nx + ny; }

// S (nx x ny, FP64, row stride lds) = dV X^T Y over npts points.  Accuracy: a
// product is off by at most 9 * 2^-62 (FP64) or 8 * 2^-54 (FP32) of 2^(Ex + Ey), the powers of two
// above its columns' largest entries.
// scratch: digit_gram_scratch_ints ints of device memory, or nullptr (taken
// from the library's stream-ordered pool); it is left holding the keys of the
// columns (see column_keys), X's and then, where Y is another block, Y's.  Asynchronous.
template <typename T>
int digit_gram(const T *X, int64_t ldx, int nx, const T *Y, int64_t ldy, int ny, int64_t npts, double dV, double *S,
               int64_t lds, int *scratch, cudaStream_t st, int *err = nullptr);

// keys[k] (device): the size of column k of X, as digit_rot takes it (a bit pattern of its
// largest absolute value; 0: a column of zeros).
template <typename T> int column_keys(const T *X, int64_t ldx, int n, int64_t npts, int *keys, cudaStream_t st);

// Y (m columns) = alpha X C + beta Y, X [npts][ldx] (n columns), C FP64
// [n][ldc]; Y may be X itself (same pointer and leading dimension) when
// beta == 0.  digit_rot_takes says whether the sizes are taken.  xkeys: the keys of X's
// columns, or nullptr where they are of one size (orthonormal states, normalised
// directions): a product is off by at most 9 * 2^-62 (FP64) or 6 * 2^-38 (FP32) of
// 2^(Ex + Ec), the powers of two above the largest entry of its row of X, the columns brought to
// one size, and of its column of C, the rows taken the other way.
bool digit_rot_takes(int n, int m, bool in_place);
template <typename T>
int digit_rot(const T *X, int64_t ldx, int n, const double *C, int64_t ldc, int m, T *Y, int64_t ldy, int64_t npts,
              double alpha, double beta, const int *xkeys, cudaStream_t st, int *err = nullptr);

// S = dV X^T Y of FP32 data to FP32 accuracy by BF16 pieces, FP32 sums over at
// most 2048 points.  Asynchronous.
int piece_gram(const float *X, int64_t ldx, int nx, const float *Y, int64_t ldy, int ny, int64_t npts, double dV, double *S,
               int64_t lds, cudaStream_t st, int *err = nullptr);

// FP32 rotation to FP32 accuracy by BF16 pieces (Y may be X itself, same leading
// dimension, for m <= 1024 and beta == 0).  work: piece_rot_bytes(n, m) bytes,
// 16-byte aligned.  Asynchronous.
int64_t piece_rot_bytes(int n, int m);
int piece_rot(const float *X, int64_t ldx, int n, const double *C, int64_t ldc, int m, float *Y, int64_t ldy, int64_t npts,
              double alpha, double beta, void *work, cudaStream_t st, int *err = nullptr);

}  // namespace rs
