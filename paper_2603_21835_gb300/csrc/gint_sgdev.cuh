// gint_sgdev.cuh -- device pieces of the exact digit products shared by the dense products (gint_sg.cu) and the
// float64 grid passes (gint_fx.cu): digits of float64 values, the accumulator levels and their recombination.
#pragma once
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "gint_ptx.cuh"

namespace sgdev {

constexpr int kDig = 8;                  // digits of an operand, and levels kept
constexpr int kTM = 128, kTN = 64;       // output tile
constexpr int kCK = 16;                  // k of a chunk (one MMA K step)
constexpr int kRangeChunks = 8;          // chunks per exact accumulation range (128 k)
constexpr uint32_t kABytes = kDig * kTM * kCK * 2, kBBytes = kDig * kTN * kCK * 2;
constexpr uint32_t kStage = kABytes + kBBytes;
constexpr int kStages = 4;
constexpr int kNonFinite = 2047;         // row exponent field of a row with an infinity or a NaN
static_assert(kDig * kTN == 512, "the levels fill the tensor memory");

// See sg_launch: wait for the predecessor's results, then let the successor be launched.
__device__ __forceinline__ void grid_wait() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

// Exponent field of |x|, at least 1 (denormals share the exponent of the smallest normal numbers).
__device__ __forceinline__ int exp_field(double x) {
  return max(1, (int)((__double_as_longlong(x) >> 52) & 0x7ff));
}

static __device__ __noinline__ double times_pow2_slow(double x, int e) {
  const int a = e >> 1, b = e - a;  // (|e| <= 2044)
  return x * __hiloint2double((1023 + a) << 20, 0) * __hiloint2double((1023 + b) << 20, 0);
}
// x 2^e: on the integer pipe while x and the result are normal (a float64 multiplication takes the SM's pipe 16 clocks
// a warp), |e| <= 2044.
__device__ __forceinline__ double times_pow2(double x, int e) {
  const int hi = __double2hiint(x), t = (hi >> 20) & 0x7ff;
  if (e == 0 || ((hi & 0x7fffffff) | __double2loint(x)) == 0) return x;
  if (t != 0 && t != 0x7ff && (unsigned)(t + e - 1) < 2046u) return __hiloint2double(hi + (e << 20), __double2loint(x));
  return times_pow2_slow(x, e);
}
// Digits of the eight values x(0 .. 7) of one row, whose largest magnitude has exponent field em: q = x 2^(62 - e)
// rounded to an integer, its balanced base-256 digits as float16, digit s as 16 bytes at d + s step.  em ==
// kNonFinite: zeros (such rows are summed without digits).
template <typename X>
__device__ __forceinline__ void store_digits(X x, int em, unsigned char *d, size_t step) {
  uint32_t lo[8], hi[8];  // the bytes of q + 0x80..80
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    const long long b = __double_as_longlong(x(j));
    const int ex = (int)((b >> 52) & 0x7ff);
    unsigned long long m = (unsigned long long)b & 0xfffffffffffffull;
    if (ex) m |= 0x10000000000000ull;
    const int s = max(ex, 1) - em + 9;  // q = m 2^s, rounded
    unsigned long long q;
    if (s >= 0)
      q = m << s;
    else
      q = s < -54 ? 0ull : (m + (1ull << (-s - 1))) >> -s;
    if (em == kNonFinite) q = 0ull;
    if (b < 0) q = 0ull - q;
    q += 0x8080808080808080ull;
    lo[j] = (uint32_t)q;
    hi[j] = (uint32_t)(q >> 32);
  }
  const __half2 off = __floats2half2_rn(1152.f, 1152.f);  // float16 bits 0x6400 | b are 1024 + b
#pragma unroll
  for (int s = 0; s < kDig; ++s) {  // digit s: byte 7 - s
    uint32_t w[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const uint32_t a = s < 4 ? hi[2 * j] : lo[2 * j], c = s < 4 ? hi[2 * j + 1] : lo[2 * j + 1];
      const uint32_t sel = 3 - (s & 3);
      const uint32_t v = (__byte_perm(a, c, sel | ((sel + 4) << 8)) & 0x00ff00ffu) | 0x64006400u;
      const __half2 h = __hsub2(*reinterpret_cast<const __half2 *>(&v), off);
      w[j] = *reinterpret_cast<const uint32_t *>(&h);
    }
    *reinterpret_cast<uint4 *>(d + (size_t)s * step) = make_uint4(w[0], w[1], w[2], w[3]);
  }
}

// A 96-bit two's complement integer, least significant word first.
struct Fx {
  uint32_t w0, w1, w2;
};
// x += v 2^32 and x += v
__device__ __forceinline__ void fx_add_hi(Fx &x, long long v) {
  asm("add.cc.u32 %0, %0, %2;\n addc.u32 %1, %1, %3;"
      : "+r"(x.w1), "+r"(x.w2)
      : "r"((uint32_t)v), "r"((uint32_t)((unsigned long long)v >> 32)));
}
__device__ __forceinline__ void fx_add_lo(Fx &x, long long v) {
  const uint32_t h = (uint32_t)((unsigned long long)v >> 32);
  asm("add.cc.u32 %0, %0, %3;\n addc.cc.u32 %1, %1, %4;\n addc.u32 %2, %2, %5;"
      : "+r"(x.w0), "+r"(x.w1), "+r"(x.w2)
      : "r"((uint32_t)v), "r"(h), "r"((uint32_t)((int)h >> 31)));
}
// Four adjacent levels of one element: v0 2^24 + v1 2^16 + v2 2^8 + v3.  SMALL: all below 2^22 in magnitude,
// so that adding 1.5 2^23 leaves the integer in the low bits (the float-to-integer conversion runs on a pipe
// a quarter as wide) and two levels still fit 32 bits.
template <bool SMALL>
__device__ __forceinline__ long long fx_levels(float v0, float v1, float v2, float v3) {
  if (SMALL) {
    constexpr uint32_t M = 0x4B400000u, B = M * 257u;
    const uint32_t m0 = __float_as_uint(v0 + 12582912.f), m1 = __float_as_uint(v1 + 12582912.f);
    const uint32_t m2 = __float_as_uint(v2 + 12582912.f), m3 = __float_as_uint(v3 + 12582912.f);
    const int p = (int)((m0 << 8) + m1 - B), q = (int)((m2 << 8) + m3 - B);
    return (long long)p * 65536 + q;
  }
  return (((long long)__float2int_rn(v0) * 256 + __float2int_rn(v1)) * 256 + __float2int_rn(v2)) * 256 + __float2int_rn(v3);
}

// x 2^E rounded to float64: the magnitude normalised by word moves and one funnel shift, some thirty 32-bit
// instructions (converting 64-bit integers would take three float64 ones, 48 clocks of the SM's pipe per warp).
__device__ __forceinline__ double fx_to_double(Fx x, int E) {
  const uint32_t sg = (uint32_t)((int)x.w2 >> 31);
  asm("add.cc.u32 %0, %0, %3;\n addc.cc.u32 %1, %1, %3;\n addc.u32 %2, %2, %3;"
      : "+r"(x.w0), "+r"(x.w1), "+r"(x.w2)
      : "r"(sg));  // -x = ~(x - 1)
  uint32_t w0 = x.w0 ^ sg, w1 = x.w1 ^ sg, w2 = x.w2 ^ sg;
  int k = E + 43;
  if (w2 == 0u) {
    w2 = w1;
    w1 = w0;
    w0 = 0u;
    k -= 32;
  }
  if (w2 == 0u) {
    if (w1 == 0u) return 0.0;
    w2 = w1;
    w1 = 0u;
    k -= 32;
  }
  const int n = __clz(w2);
  const uint32_t hi32 = __funnelshift_l(w1, w2, n), lo32 = __funnelshift_l(w0, w1, n);
  k -= n;  // value = (hi32 : lo32) / 2^11 * 2^k, the leading bit set
  const uint32_t f1 = hi32 >> 11, f0 = __funnelshift_r(lo32, hi32, 11), rnd = (lo32 >> 10) & 1u;
  if ((unsigned)(k + 1073) < 2043u) {
    const unsigned long long m = (((unsigned long long)(f1 + ((uint32_t)(k + 1074) << 20) + (sg & 0x80000000u)) << 32) | f0) + rnd;
    return __longlong_as_double((long long)m);
  }
  // denormal, zero or overflow: scaled in two exact steps and one rounding
  const int kc = min(max(k, -1140), 1030), ka = kc >> 1, kb = kc - ka;
  const double v = (double)(long long)((((unsigned long long)f1 << 32) | f0) + rnd) * __hiloint2double((ka + 1023) << 20, 0) *
                   __hiloint2double((kb + 1023) << 20, 0);
  return sg ? -v : v;
}

// Four loads of 4 columns, `step` columns apart, under one wait.
__device__ __forceinline__ void tmem_ld4x4(uint32_t taddr, uint32_t step, float (*v)[4]) {
  uint32_t r[4][4];
#pragma unroll
  for (int l = 0; l < 4; ++l)
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[l][0]), "=r"(r[l][1]), "=r"(r[l][2]), "=r"(r[l][3])
                 : "r"(taddr + l * step)
                 : "memory");
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int l = 0; l < 4; ++l)
#pragma unroll
    for (int j = 0; j < 4; ++j) v[l][j] = __uint_as_float(r[l][j]);
}

// The 12 MMAs of one chunk (16 k): left digits at a0 (digit d at + d 4 KB), right digits at b0 (digit t at + t 2 KB) as
// runs of digits of up to four 64-row operands, into the accumulator columns 64 l .. of level l.  acc: 0 for the
// first chunk of a range.  The levels 0-3, then 4-7, so that their halves can be drained apart.
__device__ __forceinline__ void mma_levels_hi(uint32_t tmem, uint64_t a0, uint64_t b0, uint32_t acc) {
  constexpr uint64_t kAStep = kTM * kCK * 2 / 16;  // one digit's operand
#pragma unroll
  for (int d = 0; d < 4; ++d)  // levels d .. 3 (digits 0 .. 3 - d of the right operand)
    gptx::mma_f16(tmem + kTN * d, a0 + d * kAStep, b0, gptx::idesc_f16(kTM, kTN * (4 - d)), d ? 1u : acc);
}
__device__ __forceinline__ void mma_levels_lo(uint32_t tmem, uint64_t a0, uint64_t b0, uint32_t acc) {
  constexpr uint64_t kAStep = kTM * kCK * 2 / 16, kBStep = kTN * kCK * 2 / 16;
  // levels max(4, d) .. 7 (digits from max(4 - d, 0)); the short ones in the middle, so that the queue holds the
  // longest MMAs while the issuing warp turns to the next chunk
  constexpr int order[kDig] = {0, 7, 6, 5, 4, 3, 2, 1};
#pragma unroll
  for (int q = 0; q < kDig; ++q) {
    const int d = order[q], l0 = d < 4 ? 4 : d;
    gptx::mma_f16(tmem + kTN * l0, a0 + d * kAStep, b0 + (l0 - d) * kBStep, gptx::idesc_f16(kTM, kTN * (8 - l0)), d ? 1u : acc);
  }
}

// One warp's half drain: levels 4 h .. 4 h + 3 of its 32 rows x 16 columns (lbase: its lane and column base) added
// into x.
__device__ __forceinline__ void drain_half(uint32_t lbase, int h, Fx *x) {
#pragma unroll
  for (int c4 = 0; c4 < 16; c4 += 4) {
    float y[4][4];
    tmem_ld4x4(lbase + kTN * 4 * h + c4, kTN, y);
    float mx = 0.f;
#pragma unroll
    for (int j = 0; j < 4; ++j)
      mx = fmaxf(fmaxf(mx, fmaxf(fabsf(y[0][j]), fabsf(y[1][j]))), fmaxf(fabsf(y[2][j]), fabsf(y[3][j])));
    if (__all_sync(0xffffffffu, mx < 4194304.f)) {
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const long long v = fx_levels<true>(y[0][j], y[1][j], y[2][j], y[3][j]);
        if (h)
          fx_add_lo(x[c4 + j], v);
        else
          fx_add_hi(x[c4 + j], v);
      }
    } else {  // digits that line up: sums up to 2^24
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const long long v = fx_levels<false>(y[0][j], y[1][j], y[2][j], y[3][j]);
        if (h)
          fx_add_lo(x[c4 + j], v);
        else
          fx_add_hi(x[c4 + j], v);
      }
    }
  }
}

}  // namespace sgdev
