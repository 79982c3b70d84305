// gint_sg.cuh -- float64 matrix products on the tensor cores: every operand is cut into exact 8-bit
// integer digits, the digit products run as float16 MMAs whose float32 sums are exact integers, and the
// digit levels are recombined in 96-bit integer arithmetic (gint_sg.cu).
#pragma once
#include <cuda_runtime.h>
#include <stddef.h>

#include <utility>

#include "gint.h"

namespace gla {

// Launch in stream order with programmatic serialization: the kernel may begin while its predecessor on the
// stream is still running and must execute griddepcontrol.wait before it touches what that one wrote.
template <typename... P, typename... Q>
int sg_launch(void (*kern)(P...), dim3 grid, unsigned threads, size_t smem, cudaStream_t st, Q &&...args) {
  cudaLaunchConfig_t c{};
  c.gridDim = grid;
  c.blockDim = dim3(threads);
  c.dynamicSmemBytes = smem;
  c.stream = st;
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  c.attrs = &at;
  c.numAttrs = 1;
  return cudaLaunchKernelEx(&c, kern, static_cast<P>(std::forward<Q>(args))...) == cudaSuccess ? GINT_OK : GINT_ECUDA;
}

// Real operand view of a product: element (r, k), r the output row (or column) index and k the
// contraction index, is
//   p[(r >> 1) rh + (r & 1) rl + (k >> 1) kh + (k & 1) kl], times ks[k >> 1] when ks is not null; half: ks in
//   two factors, ks 2^-h (1) for the left operand and 2^h (2) for the right one, 2^h next to |ks|^(1/2); and times
//   2^(kp[k] + rp[r]) when kp is not null (rp null: 0),
// or, for `rot` (the left operand of a complex product seen as a real one: output rows 2 i = real and
// 2 i + 1 = imaginary part, contraction 2 k = real and 2 k + 1 = imaginary part of the right operand),
//   +- p[(r >> 1) rh + (k >> 1) kh + ((r ^ k) & 1)], minus when r is even and k odd.
struct SgView {
  const double *p;
  long long rh, rl, kh, kl;
  int rot;
  const double *ks;
  int half;
  const int *kp, *rp;
};
inline SgView sg_real(const double *p, long long sr, long long sk) {
  return SgView{p, 2 * sr, sr, 2 * sk, sk, 0, nullptr};
}
// complex operands (interleaved double2; strides in complex elements): left (2 rows per complex row)
// and right (rows complex, contraction 2 k + part)
inline SgView sg_cplx_left(const double2 *p, long long sr, long long sk) {
  return SgView{reinterpret_cast<const double *>(p), 2 * sr, 0, 2 * sk, 0, 1, nullptr};
}
inline SgView sg_cplx_right(const double2 *p, long long sr, long long sk) {
  return SgView{reinterpret_cast<const double *>(p), 4 * sr, 2 * sr, 2 * sk, 1, 0, nullptr};
}

// One product C (+)= +-A B: element (i, j) at C[(i >> 1) crh + (i & 1) crl + (j >> 1) cch + (j & 1) ccl].
// mode 0: every element; 1: only (i >> cs) >= j (cs = 1: rows are real / imaginary pairs); 2: i >= j, each
// value also written to (j, i).  beta: add to C (else overwrite); neg: subtract the product.
struct SgProduct {
  int M, N, K, mode, cs, neg, beta;
  SgView A, B;
  double *C;
  long long crh, crl, cch, ccl;
};

// Scratch of the products (device), given back by its owner: buf holds the packed digits and the row
// exponents; status takes error bit 1 when a bounded wait gave up.
struct SgWork {
  unsigned char *buf;
  size_t bytes;
  unsigned *status;
  int num_sms;
};
// Bytes for products with at most `rows` operand rows in total (left rows plus right rows, each padded to
// 128) and contraction at most K (longer contractions are cut into ranges of kSgK).
size_t sg_bytes(long long rows, long long K);

// Where a launch's operand digits go: left and right operand of each product in turn.
struct SgOperand {
  SgView v;
  int R, K, nq, tr;    // rows, contraction, chunks of 16 k, rows of a tile (128 left, 64 right)
  int rfast;           // consecutive rows are closer in memory than consecutive k
  unsigned char *dst;  // digit blocks, see gint_sg.cu
  int *e;              // exponent field of each row's largest magnitude
};
constexpr int kPackRows = 32;  // rows of a packing block
struct SgPack {
  SgOperand op[4];
  int first[5];  // first row block of each operand; first[n..4] = total
};

// np (1 or 2) products of the same K in one launch (K <= 64: packed in one pass), asynchronous on st.
// packed (K <= 64): the operands' digits and exponents are already where sg_operands says.
int sg_gemm(const SgProduct *pr, int np, const SgWork &ws, cudaStream_t st, bool packed = false);
int sg_operands(const SgProduct *pr, int np, const SgWork &ws, SgPack *pk);

}  // namespace gla
