// gint_la.cuh -- float64 dense linear algebra of the propagation steps (gint_la.cu): the blocked
// L D L^T factorisation (no pivoting) with its solve, for real symmetric and complex symmetric
// (A^T = A, no conjugation) matrices.  Its products are those of gint_sg.cuh.
#pragma once
#include <cuda_runtime.h>

#include "gint_sg.cuh"

namespace gla {

// Block width of the factorisation: a 64-wide real contraction either way.
template <typename T>
struct LdlBlock {
  static constexpr int NB = sizeof(T) == 16 ? 32 : 64;
};
// Elements of T that ldl_solve_factor needs as workspace for n x n with nrhs right-hand sides.
template <typename T>
inline size_t ldl_work(long long n, long long nrhs) {
  return (size_t)(n + nrhs) * LdlBlock<T>::NB + (size_t)n;
}
// Operand rows of its largest launch of products (for sg_bytes, contraction 64).
template <typename T>
inline long long ldl_rows(long long n, long long nrhs) {
  return (sizeof(T) == 16 ? 5 : 3) * n + nrhs + 1024;
}

// Solves A X = B in place (B: nrhs columns of n, leading dimension ldb) by A = L D L^T of the n x n matrix
// A (column-major, leading dimension lda; only the lower triangle is read and it is overwritten).
// *info (device) = first j + 1 whose pivot d_j is zero or not finite (spd: not positive), else unchanged
// (the caller zeroes it).
template <typename T>
int ldl_factor_solve(int n, T *A, long long lda, int nrhs, T *B, long long ldb, T *work, int *info, bool spd,
                     const SgWork &ws, cudaStream_t st);

}  // namespace gla
