// gint_sgpack.cuh -- packing of the digit products' operands (gint_sg.cu), also done by the kernels that form or wait for
// an operand themselves (gint_la.cu).
#pragma once
#include "gint_sg.cuh"
#include "gint_sgdev.cuh"

namespace gla {
using namespace sgdev;

__device__ __forceinline__ double sg_at(const SgView &v, int r, int k) {
  if (v.rot) {
    const double x = v.p[(long long)(r >> 1) * v.rh + (long long)(k >> 1) * v.kh + ((r ^ k) & 1)];
    return (!(r & 1) && (k & 1)) ? -x : x;
  }
  double x = v.p[(long long)(r >> 1) * v.rh + (long long)(r & 1) * v.rl + (long long)(k >> 1) * v.kh +
                 (long long)(k & 1) * v.kl];
  if (v.ks) {
    double s = v.ks[k >> 1];
    if (v.half) {
      const int e = (__double2hiint(s) >> 20) & 0x7ff, h = e == 0 || e == 0x7ff ? 0 : (e - 1023) >> 1;
      s = v.half == 1 ? s * __hiloint2double((1023 - h) << 20, 0) : __hiloint2double((1023 + h) << 20, 0);
    }
    x *= s;
  }
  if (v.kp) x = times_pow2(x, v.kp[k] + (v.rp ? v.rp[r] : 0));
  return x;
}

constexpr int kPR = kPackRows, kPK = 64, kPT = 256;  // rows and k of a packing block, its threads
__device__ __forceinline__ void sg_load_tile(const SgOperand &o, int tid, int r0, int k0, double (*t)[kPK + 1]) {
#pragma unroll
  for (int q = 0; q < kPR * kPK / kPT; ++q) {
    const int e = tid + kPT * q;
    const int r = o.rfast ? e % kPR : e / kPK, k = o.rfast ? e / kPR : e % kPK;
    t[r][k] = (r0 + r < o.R && k0 + k < o.K) ? sg_at(o.v, r0 + r, k0 + k) : 0.0;
  }
}
// The eight threads of a row: largest exponent field of its kPK elements (in all of them).
__device__ __forceinline__ int sg_row_exp(const double (*t)[kPK + 1], int tid) {
  const int r = tid >> 3, g = tid & 7;
  int m = 1;
#pragma unroll
  for (int j = 0; j < 8; ++j) m = max(m, exp_field(t[r][g + 8 * j]));
#pragma unroll
  for (int o = 1; o < 8; o <<= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
  return m;
}
// Digits of k = 8 g .. 8 g + 7 of row r.
template <typename X>
__device__ __forceinline__ void sg_store_group(const SgOperand &o, int r, int g, int em, X x) {
  const int chunk = g >> 1;
  if (chunk >= o.nq) return;
  const size_t blk = (size_t)kDig * o.tr * kCK * 2;
  store_digits(x, em, o.dst + ((size_t)(r / o.tr) * o.nq + chunk) * blk + (size_t)((r % o.tr) >> 3) * 256 + (g & 1) * 128 + (r & 7) * 16,
               (size_t)o.tr * kCK * 2);
}

}  // namespace gla
