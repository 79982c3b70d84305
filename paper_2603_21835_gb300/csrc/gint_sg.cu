// gint_sg.cu -- float64 matrix products on the tcgen05 tensor cores (gint_sg.cuh).
//
// The GB300 multiplies float64 on its CUDA cores at 2 fused multiply-adds per clock per SM (1.25 TFLOP/s)
// and float16 on its tensor cores some 1500 times faster, so a float64 product is cheaper as many exact
// float16 ones: the error-free splitting of Ozaki, Ogita, Oishi and Rump ("Error-free transformations of
// matrix multiplication by using fast routines of matrix multiplication", 2012), here with integer digits.
//
//   x_rk = q_rk 2^(e_r - 62), q an integer of at most 62 bits (e_r: the exponent of row r's largest
//   magnitude, so the rounding of q is 2^-63 of that maximum and values within 2^9 of it are exact);
//   q = sum_s d_s 256^(7 - s), s = 0..7, d_s in [-128, 127] (balanced digits: the bytes of q + 0x80..80
//   less 128), exact in float16;
//   sum_k x_ik y_jk = 2^(..) sum_{l = s + t} 256^(14 - l) sum_k d_s d_t, levels l = 0..7 kept (the
//   dropped ones are below 2^-60 of the largest products: float64 rounding of one product is 2^-53).
//   An element's error is below 2^-58 per term of the product of its two rows' largest magnitudes, and one float64
//   rounding: in norms that is better than a float64 chain, but terms far below the maxima of both rows lose bits that
//   a chain keeps.  Callers balance a contraction index whose magnitudes run against each other in the two operands
//   (basis functions of unequal norms, pivots) with powers of two.
//
// The MMAs of level l add at most 8 x 128 products of magnitude 2^14 per accumulator in a range of 128 k:
// at most 2^24, so every float32 partial sum is an exact integer whatever the tensor core's rounding.
// After each range the eight levels are drained into two 64-bit integers per element (levels 0-3 and
// 4-7), and the element is converted to float64 once at the end of the contraction (one rounding; the
// CUDA cores' float64 chain has one per multiply-add).
//
// k_sg_max / k_sg_pack: row exponents and digit blocks.  Block (row tile of TR = 128 left / 64 right rows,
//   chunk of 16 k): [digit 8][row group TR / 8][k group 2][8 rows][8 k] float16, K-major core matrices
//   (LBO 128, SBO 256), so a right block is one operand of 512 rows (digit, column).
// k_sg_mma: persistent, one CTA of 18 warps per SM.  Warp 17 streams the two blocks of a chunk (48 KB) by
//   bulk copies into a 4-stage ring; warp 16 issues 12 MMAs per chunk, digit s of the left times a run of
//   digits of the right as ONE operand of up to 4 x 64 rows, which land in the accumulator columns
//   64 (s + t) .. of level s + t: 512 columns of tensor memory hold all eight levels of a 128 x 64 tile.
//   Warps 0-15 drain and store a tile while the next one's MMAs run.
// Bound: 36 digit products, 1152 tensor cycles a chunk (1210 measured).
#include <cuda_fp16.h>
#include <stdint.h>

#include <algorithm>

#include "gint.h"
#include "gint_ptx.cuh"
#include "gint_sg.cuh"
#include "gint_sgpack.cuh"

namespace gla {
namespace {
using namespace gptx;
using namespace sgdev;

constexpr int kSgK = 1024;               // longest contraction packed at once
constexpr uint32_t kSgSmem = kStages * kStage;
constexpr int kDrainWarps = 16, kMmaWarp = 16, kLoadWarp = 17, kSgThreads = 32 * (kDrainWarps + 2);
constexpr long long kWaitNs = 2000000000LL;  // bounded waits: 2 s
constexpr unsigned kErrTimeout = 1u, kErrInflight = 2u;

// ---------------------------------------------------------------------------------------- packing
__device__ __forceinline__ const SgOperand &sg_operand(const SgPack &P, int &rb) {
  int i = 0;
  while (i < 3 && (int)blockIdx.x >= P.first[i + 1]) ++i;
  rb = (int)blockIdx.x - P.first[i];
  return P.op[i];
}

// Row exponents of long contractions (e zeroed before): blockIdx.y = range of 64 k.
__global__ void __launch_bounds__(kPT) k_sg_max(const __grid_constant__ SgPack P) {
  __shared__ double t[kPR][kPK + 1];
  int rb;
  const SgOperand &o = sg_operand(P, rb);
  const int r0 = rb * kPR;
  grid_wait();
  sg_load_tile(o, threadIdx.x, r0, blockIdx.y * kPK, t);
  __syncthreads();
  const int m = sg_row_exp(t, threadIdx.x), r = r0 + (threadIdx.x >> 3);
  if ((threadIdx.x & 7) == 0 && r < o.R) atomicMax(o.e + r, m);
}

// Digits: one thread per row and 8 k.  ONE: the whole contraction is one range (K <= 64), so the exponent
// is found here; otherwise k_sg_max has left it in e.
template <bool ONE>
__global__ void __launch_bounds__(kPT) k_sg_pack(const __grid_constant__ SgPack P) {
  __shared__ double t[kPR][kPK + 1];
  int rb;
  const SgOperand &o = sg_operand(P, rb);
  const int r0 = rb * kPR, kb = ONE ? 0 : (int)blockIdx.y * kPK;
  grid_wait();
  sg_load_tile(o, threadIdx.x, r0, kb, t);
  __syncthreads();
  const int rl = threadIdx.x >> 3, r = r0 + rl;
  const int em = ONE ? sg_row_exp(t, threadIdx.x) : (r < o.R ? o.e[r] : 1);
  if (r >= o.R) return;
  if (ONE && (threadIdx.x & 7) == 0) o.e[r] = em;
  sg_store_group(o, r, kb / 8 + (threadIdx.x & 7), em, [&](int j) { return t[rl][8 * (threadIdx.x & 7) + j]; });
}

// --------------------------------------------------------------------------------------- products
struct SgProb {
  const unsigned char *PA, *PB;
  const int *eA, *eB;
  int nq, ntn, ntiles;
  SgProduct p;
};
struct SgArgs {
  SgProb pr[2];
  int tiles;  // of all products
  unsigned *status;
};
// Tile u of a product: mode 0 row-major; otherwise the lower triangle, row tile tm having
// mul (tm + 1) column tiles (mul = 1 for paired rows, 2 otherwise), cut off at the last one.
__device__ __forceinline__ void sg_tile(const SgProb &P, int u, int &tm, int &tn) {
  if (P.p.mode == 0) {
    tm = u / P.ntn;
    tn = u - tm * P.ntn;
    return;
  }
  const int mul = P.p.cs ? 1 : 2;
  tm = (int)((sqrtf(1.f + 8.f * (float)u / (float)mul) - 1.f) * 0.5f);
  while (mul * (long long)tm * (tm + 1) / 2 > u) --tm;
  while (mul * (long long)(tm + 1) * (tm + 2) / 2 <= u) ++tm;
  tn = u - (int)(mul * (long long)tm * (tm + 1) / 2);
}

// Element (i, j) of a row or column that holds an infinity or a NaN: the plain float64 sum.
__device__ __noinline__ void sg_plain(const SgProduct &p, int i, int j) {
  double a = 0.0;
  for (int k = 0; k < p.K; ++k) a = fma(sg_at(p.A, i, k), sg_at(p.B, j, k), a);
  if (p.neg) a = -a;
  double *const c = p.C + (long long)(i >> 1) * p.crh + (long long)(i & 1) * p.crl + (long long)(j >> 1) * p.cch +
                    (long long)(j & 1) * p.ccl;
  if (p.beta) a += *c;
  *c = a;
  if (p.mode == 2 && i != j)
    p.C[(long long)(j >> 1) * p.crh + (long long)(j & 1) * p.crl + (long long)(i >> 1) * p.cch + (long long)(i & 1) * p.ccl] = a;
}

// Range r of a tile is complete for levels 0-3 (accfull[0]) and 4-7 (accfull[1]); the drain warps give the
// two halves back (accfree) as they finish with each, so that half of a drain overlaps the MMAs around it.
struct SgShared {
  uint64_t full[kStages], empty[kStages], accfull[2], accfree[2];
  uint32_t tmem;
};

__global__ void __launch_bounds__(kSgThreads, 1) k_sg_mma(const __grid_constant__ SgArgs P) {
  extern __shared__ __align__(1024) unsigned char smem[];
  __shared__ SgShared sh;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  if (tid == 0) {
    for (int s = 0; s < kStages; ++s) {
      mbar_init(&sh.full[s], 1);
      mbar_init(&sh.empty[s], 1);
    }
    for (int h = 0; h < 2; ++h) {
      mbar_init(&sh.accfull[h], 1);
      mbar_init(&sh.accfree[h], kDrainWarps);
    }
    fence_mbar_init();
  }
  if (warp == kMmaWarp) {
    tmem_alloc(&sh.tmem, 512);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = sh.tmem;
  unsigned *status = P.status;
  const int n0 = P.pr[0].ntiles;
  grid_wait();

  if (warp == kLoadWarp) {
    // the copies run kStages chunks ahead of the MMAs, across tile boundaries
    int gl = 0;
    bool ok = true;
    for (int t = blockIdx.x; t < P.tiles && ok; t += gridDim.x) {
      const SgProb &pr = P.pr[t < n0 ? 0 : 1];
      int tm, tn;
      sg_tile(pr, t < n0 ? t : t - n0, tm, tn);
      const unsigned char *a = pr.PA + (size_t)tm * pr.nq * kABytes, *b = pr.PB + (size_t)tn * pr.nq * kBBytes;
      const int nq = pr.nq;
      for (int c = 0; c < nq && ok; ++c, ++gl, a += kABytes, b += kBBytes) {
        const int s = gl % kStages;
        if (gl >= kStages)
          ok = __all_sync(0xffffffffu,
                          mbar_wait(&sh.empty[s], (uint32_t)(gl / kStages - 1) & 1u, status, kErrTimeout, kWaitNs));
        if (!ok) break;
        if (lane == 0) {
          mbar_arrive_tx(&sh.full[s], kStage);
          bulk_g2s(smem + s * kStage, a, kABytes, &sh.full[s]);
          bulk_g2s(smem + s * kStage + kABytes, b, kBBytes, &sh.full[s]);
        }
        __syncwarp();
      }
    }
    // no copy may still be landing when the CTA exits
    for (int c = max(0, gl - kStages); c < gl; ++c)
      mbar_wait(&sh.full[c % kStages], (uint32_t)(c / kStages) & 1u, status, kErrTimeout, kWaitNs);
  } else if (warp == kMmaWarp) {
    // a tcgen05.mma blocks its issuer while the few places of the tensor pipe's queue are taken, so this
    // warp does nothing else (with the copies issued from it too, a chunk took 2320 clocks instead of 1210)
    const uint32_t sbase = smem_u32(smem);
    int gc = 0, gb = 0;  // chunks issued, ranges begun
    bool ok = true;
    for (int t = blockIdx.x; t < P.tiles && ok; t += gridDim.x) {
      const int nq = P.pr[t < n0 ? 0 : 1].nq;
      for (int c = 0; c < nq; ++c, ++gc) {
        const int s = gc % kStages, cr = c % kRangeChunks;
        const bool first = cr == 0, last = cr == kRangeChunks - 1 || c == nq - 1;
        if (first) ++gb;
        const uint32_t fpar = (uint32_t)(gb - 2) & 1u;  // the range before this one has been drained
        ok = mbar_wait(&sh.full[s], (uint32_t)(gc / kStages) & 1u, status, kErrTimeout, kWaitNs);
        if (first && gb > 1) ok = ok && mbar_wait(&sh.accfree[0], fpar, status, kErrTimeout, kWaitNs);
        ok = __all_sync(0xffffffffu, ok);
        if (!ok) break;
        tc_fence_after();
        const uint64_t a0 = sdesc(sbase + s * kStage, 128, 256), b0 = sdesc(sbase + s * kStage + kABytes, 128, 256);
        const uint32_t acc = first ? 0u : 1u;
        if (elect_one()) {
          mma_levels_hi(tmem, a0, b0, acc);
          if (last) mma_commit(&sh.accfull[0]);
        }
        __syncwarp();
        if (first && gb > 1) {
          ok = __all_sync(0xffffffffu, mbar_wait(&sh.accfree[1], fpar, status, kErrTimeout, kWaitNs));
          if (!ok) break;
          tc_fence_after();
        }
        if (elect_one()) {
          mma_levels_lo(tmem, a0, b0, acc);
          mma_commit(&sh.empty[s]);
          if (last) mma_commit(&sh.accfull[1]);
        }
        __syncwarp();
      }
    }
    // the MMAs issued so far are complete before the tensor memory is given back
    if (!ok && elect_one()) mma_commit(&sh.empty[gc % kStages]);
    __syncwarp();
    if (!ok || gc > 0) {
      const int g = ok ? gc - 1 : gc;
      if (!mbar_wait(&sh.empty[g % kStages], (uint32_t)(g / kStages) & 1u, status, kErrTimeout, kWaitNs) && lane == 0)
        atomicOr(status, kErrInflight);
    }
  } else {
    // warp w drains TMEM lanes 32 (w mod 4) .. + 31 (rows) and 16 columns from 16 (w / 4)
    const int c0 = (warp >> 2) * 16;
    const uint32_t lbase = tmem + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)c0;
    int gb = 0;
    bool ok = true;
    for (int t = blockIdx.x; t < P.tiles && ok; t += gridDim.x) {
      const int pi = t < n0 ? 0 : 1;
      const SgProb &pr = P.pr[pi];
      const SgProduct &p = pr.p;
      int tm, tn;
      sg_tile(pr, pi ? t - n0 : t, tm, tn);
      const int i = tm * kTM + (warp & 3) * 32 + lane, jb = tn * kTN + c0;
      const bool rowok = i < p.M;
      double *const Ci = p.C + (long long)(i >> 1) * p.crh + (long long)(i & 1) * p.crl + (long long)(jb >> 1) * p.cch;
      if (p.beta && rowok && (lane & 15) == 0)  // the old values travel to L2 while the MMAs run
        for (int j = 0; j < 16 && jb + j < p.N; ++j)
          asm volatile("prefetch.global.L2 [%0];" ::"l"(Ci + (j >> 1) * p.cch + (j & 1) * p.ccl));
      Fx x[16];
#pragma unroll
      for (int j = 0; j < 16; ++j) x[j] = Fx{0u, 0u, 0u};
      const int nr = (pr.nq + kRangeChunks - 1) / kRangeChunks;
      for (int b = 0; b < nr && ok; ++b, ++gb) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          ok = ok && __all_sync(0xffffffffu, mbar_wait(&sh.accfull[h], (uint32_t)gb & 1u, status, kErrTimeout, kWaitNs));
          if (!ok) break;
          tc_fence_after();
          drain_half(lbase, h, x);
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(&sh.accfree[h]);
        }
      }
      if (!ok) break;
      const int ea = rowok ? __ldg(pr.eA + i) : 1;
      const int4 *const eb4 = reinterpret_cast<const int4 *>(pr.eB + jb);
      const uint32_t flip = p.neg ? 0x80000000u : 0u;
      const int jend = p.mode == 0 ? p.N : min(p.N, (i >> p.cs) + 1);  // columns of this row that are wanted
      const int jn = rowok ? jend - jb : 0;
      double old[2][4];  // the next four old values travel while the current four are converted
      auto fetch = [&](int j4) {
        double *const o = old[(j4 >> 2) & 1];
        const double *const c = Ci + (long long)(j4 >> 1) * p.cch;
#pragma unroll
        for (int q = 0; q < 4; ++q)
          o[q] = p.beta && j4 + q < jn ? c[(q >> 1) * p.cch + ((q & 1) ? p.ccl : 0)] : 0.0;
      };
      fetch(0);
#pragma unroll
      for (int j4 = 0; j4 < 16; j4 += 4) {
        if (__all_sync(0xffffffffu, j4 >= jn)) break;
        if (j4 < 12) fetch(j4 + 4);
        const int4 e4 = __ldg(eb4 + j4 / 4);
        const int eb[4] = {e4.x, e4.y, e4.z, e4.w};
        double *const Cj[2] = {Ci + (long long)(j4 >> 1) * p.cch, Ci + (long long)((j4 >> 1) + 1) * p.cch};
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          double v = fx_to_double(x[j4 + q], ea + eb[q] - 2 * 1022 - 68);
          v = __hiloint2double(__double2hiint(v) ^ flip, __double2loint(v));
          if (p.beta) v += old[(j4 >> 2) & 1][q];
          if (j4 + q < jn && max(ea, eb[q]) != kNonFinite) {
            Cj[q >> 1][(q & 1) ? p.ccl : 0] = v;
            const int j = jb + j4 + q;
            if (p.mode == 2 && i != j)
              p.C[(long long)(j >> 1) * p.crh + (long long)(j & 1) * p.crl + (long long)(i >> 1) * p.cch +
                  (long long)(i & 1) * p.ccl] = v;
          }
        }
      }
      // rows and columns with an infinity or a NaN
      for (int j = jb; j < jb + 16; ++j)
        if (j < jb + jn && max(ea, __ldg(pr.eB + j)) == kNonFinite) sg_plain(p, i, j);
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == kMmaWarp) tmem_dealloc(tmem, 512);
}

constexpr size_t kAlign = 1024;
size_t pad(size_t x, size_t a) { return (x + a - 1) / a * a; }

}  // namespace

size_t sg_bytes(long long rows, long long K) {
  const size_t R = pad((size_t)rows, kTM) + 4 * kTM, k = pad((size_t)std::max<long long>(64, std::min<long long>(K, kSgK)), kCK);
  return R * k * kDig * 2 + R * sizeof(int) + 16 * kAlign;
}

// Layout and arguments of the launch for the contraction range [k0, k0 + kk).
static int sg_plan(const SgProduct *pr, int np, const SgWork &ws, int k0, int kk, SgPack &pk, SgArgs &ar, int **pe0, long long &erows) {
  const int K = pr[0].K, nq = std::max(1, (kk + kCK - 1) / kCK);
  ar.status = ws.status;
  size_t off = 0;
  unsigned char *base = ws.buf;
  int nop = 0, blocks = 0;
  for (int q = 0; q < np; ++q) erows += pad(pr[q].M, kTM) + pad(pr[q].N, kTM);
  if (pad((size_t)erows * sizeof(int), kAlign) > ws.bytes) return GINT_EINVAL;
  int *const e0 = *pe0 = reinterpret_cast<int *>(base);
  off = pad((size_t)erows * sizeof(int), kAlign);
  int *e = e0;
  for (int q = 0; q < np; ++q) {
    if (pr[q].K != K || pr[q].M < 0 || pr[q].N < 0) return GINT_EINVAL;
    SgProb &pb = ar.pr[q];
    pb.p = pr[q];
    // the range [k0, k0 + kk) of the contraction (kSgK is even: part offsets stay aligned)
    for (SgView *v : {&pb.p.A, &pb.p.B}) {
      v->p += (long long)(k0 >> 1) * v->kh;
      if (v->ks) v->ks += k0 >> 1;
      if (v->kp) v->kp += k0;
    }
    pb.p.K = kk;
    if (k0 > 0) pb.p.beta = 1;
    pb.nq = nq;
    pb.ntn = (pb.p.N + kTN - 1) / kTN;
    const long long ntm = (pb.p.M + kTM - 1) / kTM;
    long long tiles = 0;
    if (pb.p.mode == 0) {
      tiles = ntm * pb.ntn;
    } else {
      const int mul = pb.p.cs ? 1 : 2;
      for (long long tm = 0; tm < ntm; ++tm) tiles += std::min<long long>(pb.ntn, mul * (tm + 1));
    }
    if (ar.tiles + tiles > 0x3fffffffLL) return GINT_EINVAL;
    pb.ntiles = (int)tiles;
    ar.tiles += (int)tiles;
    for (int side = 0; side < 2; ++side) {
      SgOperand &o = pk.op[nop];
      o.v = side ? pb.p.B : pb.p.A;
      o.R = side ? pb.p.N : pb.p.M;
      o.K = kk;
      o.nq = nq;
      o.tr = side ? kTN : kTM;
      const long long sr = o.v.rot ? o.v.rh / 2 : std::min(o.v.rl, o.v.rh), sk = o.v.rot ? o.v.kh / 2 : std::min(o.v.kl, o.v.kh);
      o.rfast = sr <= sk;
      o.dst = base + off;
      o.e = e;
      e += pad(o.R, kTM);
      off += pad(o.R, o.tr) / o.tr * (size_t)nq * kDig * o.tr * kCK * 2;
      (side ? pb.PB : pb.PA) = o.dst;
      (side ? pb.eB : pb.eA) = o.e;
      pk.first[nop++] = blocks;
      blocks += (o.R + kPR - 1) / kPR;
    }
  }
  if (off > ws.bytes) return GINT_EINVAL;
  for (int q = nop; q < 5; ++q) pk.first[q] = blocks;
  return GINT_OK;
}

int sg_operands(const SgProduct *pr, int np, const SgWork &ws, SgPack *pk) {
  if (np < 1 || np > 2 || pr[0].K > kPK) return GINT_EINVAL;
  SgArgs ar{};
  int *e0;
  long long erows = 0;
  return sg_plan(pr, np, ws, 0, pr[0].K, *pk, ar, &e0, erows);
}

int sg_gemm(const SgProduct *pr, int np, const SgWork &ws, cudaStream_t st, bool packed) {
  if (np < 1 || np > 2 || (packed && pr[0].K > kPK)) return GINT_EINVAL;
  const int K = pr[0].K;
  if (cudaFuncSetAttribute(k_sg_mma, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSgSmem) != cudaSuccess)
    return GINT_ECUDA;
  for (int k0 = 0; k0 < std::max(K, 1); k0 += kSgK) {
    const int kk = std::min(kSgK, K - k0);
    SgPack pk{};
    SgArgs ar{};
    int *e0 = nullptr;
    long long erows = 0;
    int rc = sg_plan(pr, np, ws, k0, kk, pk, ar, &e0, erows);
    if (rc) return rc;
    if (ar.tiles == 0) return GINT_OK;
    if (packed) {  // K <= 64: one range
    } else if (kk <= kPK) {
      if ((rc = sg_launch(k_sg_pack<true>, dim3((unsigned)pk.first[4]), kPT, 0, st, pk))) return rc;
    } else {
      if (cudaMemsetAsync(e0, 0, (size_t)erows * sizeof(int), st) != cudaSuccess) return GINT_ECUDA;
      const dim3 g((unsigned)pk.first[4], (unsigned)((kk + kPK - 1) / kPK));
      k_sg_max<<<g, kPT, 0, st>>>(pk);  // after a copy engine's work: plain stream order
      if (cudaGetLastError() != cudaSuccess) return GINT_ECUDA;
      if ((rc = sg_launch(k_sg_pack<false>, g, kPT, 0, st, pk))) return rc;
    }
    if ((rc = sg_launch(k_sg_mma, dim3((unsigned)std::min(ws.num_sms, ar.tiles)), kSgThreads, kSgSmem, st, ar))) return rc;
  }
  return GINT_OK;
}

}  // namespace gla
