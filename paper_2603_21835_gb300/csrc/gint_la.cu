// gint_la.cu -- float64 dense linear algebra of the propagation steps around the grid passes (the
// Crank-Nicolson step and the energy-density matrix of paper Sec. 2): a blocked L D L^T factorisation
// without pivoting with its triangular solves, real and complex.
//
// The products (trailing updates, and the updates of the solve) run on the tensor cores (gint_sg.cu).
// What is left on the CUDA cores' float64 pipe (2 fused multiply-adds per clock per SM: a warp-wide
// float64 instruction occupies it for 16 clocks, a dependent chain sees its latency at every step) are
// the NB x NB diagonal blocks and the NB-wide substitutions: both grow with NB, the number of launches
// falls with it; NB = 32 complex or 64 real keeps the two of similar size for n of a few hundred and more.
//
// L D L^T without pivoting: the Crank-Nicolson matrix S + i dt/2 H is complex symmetric with a
// positive definite Hermitian part S, so its leading blocks are nonsingular and elimination without
// pivoting is stable for small dt (the growth stays of order 1 + dt^2 |H S^-1 H| / 4); the overlap
// S of the energy-density matrix is symmetric positive definite.  Symmetry halves the flops of a
// general LU.
//
// The right-hand sides ride along with the factorisation as further rows of the matrix ([A; B^T]): a
// panel step turns their block into W = (L^-1 B)^T and leaves D^-1 L^-1 B in B, so the forward
// substitution costs no launches of its own and only the backward one follows.
#include <algorithm>

#include "gint.h"
#include "gint_la.cuh"
#include "gint_sgpack.cuh"

namespace gla {
namespace {

__device__ __forceinline__ double shfl(double x, int lane) { return __shfl_sync(0xffffffffu, x, lane); }
__device__ __forceinline__ double2 shfl(double2 x, int lane) {
  return make_double2(__shfl_sync(0xffffffffu, x.x, lane), __shfl_sync(0xffffffffu, x.y, lane));
}

// scalar arithmetic for T = double and T = double2 (complex, no conjugation anywhere)
template <typename T>
struct Ar;
template <>
struct Ar<double> {
  static __device__ __forceinline__ double zero() { return 0.0; }
  static __device__ __forceinline__ double fms(double a, double b, double c) { return ::fma(-a, b, c); }  // c - a b
  static __device__ __forceinline__ double mul(double a, double b) { return a * b; }
  static __device__ __forceinline__ double scale(double a, double s) { return a * s; }
  static __device__ __forceinline__ double pow2(double a, int e) { return times_pow2(a, e); }
  // reciprocal's denominator and numerator: 1 / d = num / den
  static __device__ __forceinline__ double den(double d) { return d; }
  static __device__ __forceinline__ double num(double) { return 1.0; }
  static __device__ __forceinline__ bool bad_pivot(double d, bool spd) { return spd ? !(d > 0.0) : !(d != 0.0 && isfinite(d)); }
};
template <>
struct Ar<double2> {
  static __device__ __forceinline__ double2 zero() { return make_double2(0.0, 0.0); }
  static __device__ __forceinline__ double2 fms(double2 a, double2 b, double2 c) {
    return make_double2(::fma(a.y, b.y, ::fma(-a.x, b.x, c.x)), ::fma(-a.y, b.x, ::fma(-a.x, b.y, c.y)));
  }
  static __device__ __forceinline__ double2 scale(double2 a, double s) { return make_double2(a.x * s, a.y * s); }
  static __device__ __forceinline__ double2 pow2(double2 a, int e) { return make_double2(times_pow2(a.x, e), times_pow2(a.y, e)); }
  static __device__ __forceinline__ double2 mul(double2 a, double2 b) {
    return make_double2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
  }
  // 1 / d = conj(d) / |d|^2
  static __device__ __forceinline__ double den(double2 d) { return ::fma(d.y, d.y, d.x * d.x); }
  static __device__ __forceinline__ double2 num(double2 d) { return make_double2(d.x, -d.y); }
  static __device__ __forceinline__ bool bad_pivot(double2 d, bool) {
    const double m = d.x * d.x + d.y * d.y;
    return !(m > 0.0 && isfinite(m));
  }
};

// ------------------------------------------------------------------------ L D L^T, diagonal block
constexpr int kDT = 256;

// 1 / q to float64 rounding: the float32 reciprocal and one third-order Newton step, r (1 + e + e^2) with
// e = 1 - q r below 2^-22: four dependent float64 instructions where the division is about ten.  Outside the
// float32 range (and for zeros, infinities and NaNs) the division itself.
__device__ __forceinline__ double recip(double q) {
  const float f = (float)q;
  if (!(fabsf(f) > 1e-30f && fabsf(f) < 1e30f)) return 1.0 / q;
  const double r = (double)__frcp_rn(f), e = fma(-q, r, 1.0);
  return fma(r, fma(e, e, e), r);
}

// One CTA factors the nb x nb diagonal block, right-looking: at step j, l_kj = a_kj / d_j, then
// a_ik -= a_ij l_kj for i >= k > j.  The float64 chain from one pivot to the next sets the time, so warp 0 does
// nothing else: it holds column j + 1 (lane = row), applies step j to it, and forms its reciprocal and scaled
// column while the other warps apply step j to the columns behind.  Their elements stay in registers, packed
// from the triangle's last column backwards so that active ones fill whole warps; the column that warp 0 needs
// next is published in shared memory.  One barrier a step.  (Complex, NB = 32: 34 us with two barriers and a
// division in the chain, 30 us so; eight warps that all divided took 170 us for a block of 64.)
template <typename T>
__global__ void __launch_bounds__(kDT) k_ldl_diag(int nb, T *__restrict__ A, long long lda, int j0, int spd,
                                                  int *__restrict__ info, T *__restrict__ dinv) {
  constexpr int NB = LdlBlock<T>::NB, RL = NB / 32, NW = kDT - 32;
  constexpr int NE = NB * (NB - 1) / 2, PER = (NE + NW - 1) / NW;  // elements of columns 1 .. NB - 1
  __shared__ T pub[2][NB], cbuf[2][NB], lbuf[2][NB];
  const int tid = threadIdx.x;
  grid_wait();
  if (tid < 32) {
    const int lane = tid;
    bool bad = false;
    // column j of the factor: x (rows lane, lane + 32) final, published with l = x / d
    auto finish = [&](int j, const T *x) {
      T d = Ar<T>::zero();
#pragma unroll
      for (int r = 0; r < RL; ++r) {
        T v = shfl(x[r], j & 31);
        if (r == (j >> 5)) d = v;
      }
      const double q = recip(Ar<T>::den(d));
      const T nu = Ar<T>::num(d);
#pragma unroll
      for (int r = 0; r < RL; ++r) {
        const int i = lane + 32 * r;
        const T l = Ar<T>::scale(Ar<T>::mul(x[r], nu), q);
        cbuf[j & 1][i] = x[r];
        lbuf[j & 1][i] = l;
        if (i > j && i < nb) A[i + j * lda] = l;
      }
      if (lane == 0) {
        if (!bad && Ar<T>::bad_pivot(d, spd)) {
          bad = true;
          atomicCAS(info, 0, j0 + j + 1);
        }
        dinv[j] = Ar<T>::scale(nu, q);
        A[j + j * lda] = d;
      }
    };
    T x[RL];
#pragma unroll
    for (int r = 0; r < RL; ++r) x[r] = lane + 32 * r < nb ? A[lane + 32 * r] : Ar<T>::zero();
    finish(0, x);
    for (int j = 0; j + 1 < nb; ++j) {
      __syncthreads();
      const T lk = lbuf[j & 1][j + 1];
#pragma unroll
      for (int r = 0; r < RL; ++r) {
        const int i = lane + 32 * r;
        x[r] = i > j && i < nb ? Ar<T>::fms(cbuf[j & 1][i], lk, pub[(j + 1) & 1][i]) : Ar<T>::zero();
      }
      finish(j + 1, x);
    }
  } else {
    T a[PER];
    int ei[PER], ek[PER];
#pragma unroll
    for (int q = 0; q < PER; ++q) {
      // position e from the end of the column-major triangle: column NB - 1 - c has c + 1 elements
      const int e = tid - 32 + NW * q;
      ei[q] = ek[q] = -1;
      a[q] = Ar<T>::zero();
      if (e < NE) {
        int c = (int)((sqrtf(8.f * (float)e + 1.f) - 1.f) * 0.5f);
        while (c * (c + 1) / 2 > e) --c;
        while ((c + 1) * (c + 2) / 2 <= e) ++c;
        const int k = NB - 1 - c, i = k + (e - c * (c + 1) / 2);
        if (i < nb) {
          ei[q] = i;
          ek[q] = k;
          a[q] = A[i + k * lda];
          if (k == 1) pub[1][i] = a[q];
        }
      }
    }
    for (int j = 0; j + 1 < nb; ++j) {
      __syncthreads();
      const T *c = cbuf[j & 1], *l = lbuf[j & 1];
#pragma unroll
      for (int q = 0; q < PER; ++q)
        if (ek[q] >= j + 2) {
          a[q] = Ar<T>::fms(c[ei[q]], l[ek[q]], a[q]);
          if (ek[q] == j + 2) pub[(j + 2) & 1][ei[q]] = a[q];
        }
    }
  }
}

// ------------------------------------------------- digits of the next product's operands (gint_sgpack.cuh)
// A launch of its own for them took 9 us a panel, as long as the solve before it: the solve's CTAs cut the vectors they
// have just formed, and in the backward substitution, where the left operand is part of the factor and waits for
// nothing, further CTAs of the same launch cut that one.
__device__ __forceinline__ void pack_left(const SgOperand &o, int rb, double (*t)[kPK + 1]) {
  const int tid = threadIdx.x, r0 = rb * kPR;
  grid_wait();  // (the digits' place was read by the product before)
  if (tid < kPT) sg_load_tile(o, tid, r0, 0, t);
  __syncthreads();
  const int r = r0 + (tid >> 3);
  if (tid >= kPT) return;
  const int em = sg_row_exp(t, tid);
  if (r >= o.R) return;
  if ((tid & 7) == 0) o.e[r] = em;
  sg_store_group(o, r, tid & 7, em, [&](int j) { return t[tid >> 3][8 * (tid & 7) + j]; });
}
__device__ __forceinline__ void put(double *t, int i, double x) { t[i] = x; }
__device__ __forceinline__ void put(double *t, int i, double2 x) {
  t[2 * i] = x.x;
  t[2 * i + 1] = x.y;
}
// The exponent of |d|^(-1/2) for a pivot d, from 1 / d.  The update's contraction runs over pivots: W = L D has
// their scale in full and L has none, so that a row's largest element may hide the others' low bits (sg's digits are
// relative to it).  W |d|^(-1/2) against L |d|^(1/2), rounded to powers of two, are of the size of a Cholesky factor's rows: below the
// square root of the matrix diagonal, whatever the pivots.  (Pivots of 1e-8 to 1e-12 under a unit diagonal, n = 160:
// residual over |X| 4e-14 to 5e-12 without it, 4e-16 to 1e-15 with it, as float64 elimination leaves.)
__device__ __forceinline__ int pivot_balance(double dinv) {
  const int e = (__double2hiint(dinv) >> 20) & 0x7ff;
  return e == 0 || e == 0x7ff ? 0 : (e - 1023) >> 1;
}
__device__ __forceinline__ int pivot_balance(double2 dinv) {
  const double a = fabs(dinv.x), b = fabs(dinv.y);
  return pivot_balance(a > b ? a : b);
}
// Vectors v0 .. v0 + SV - 1 of a solve, element i of vector vl: x (before the division by D) and y, to be packed.
//   PANEL: vectors v < nv are rows v of the left operand W and of the right operand L of product 0 and of the left
//   operand L of product 1; the others rows of the right operand W of product 1.  Otherwise all are rows of the right
//   operand of product 0.  (Rows of a complex left operand come in pairs, see SgView.)
template <typename T, int SV, bool PANEL>
__device__ __forceinline__ void pack_vectors(const SgPack &pk, int npk, int v0, int nv, int nv2, int i, int vl, T x, T y,
                                             double (*t)[kPK + 1]) {
  constexpr bool C = sizeof(T) == 16;
  static_assert(SV == 8, "");
  __shared__ int s_e[2 * SV];
  const int tid = threadIdx.x;
  put(t[vl], i, x);
  put(t[SV + vl], i, y);
  __syncthreads();
  if (tid < 2 * SV * 16) {
    int m = 1;
#pragma unroll
    for (int q = 0; q < kPK / 16; ++q) m = max(m, exp_field(t[tid >> 4][(tid & 15) + 16 * q]));
#pragma unroll
    for (int o = 1; o < 16; o <<= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
    if ((tid & 15) == 0) s_e[tid >> 4] = m;
  }
  __syncthreads();
  for (int u = tid; u < 5 * SV * 8; u += blockDim.x) {
    const int slot = u / (SV * 8), l = (u >> 3) & (SV - 1), g = u & 7, v = v0 + l;
    if (v >= nv + nv2) continue;
    int op = -1, r = v, part = -1, src = l;  // operand, its row, row of a complex pair, row of t
    if (PANEL && v >= nv) {
      if (slot == 2) op = 3;
      r = v - nv;
    } else if (slot == 2) {
      op = 1;
      if (PANEL) src = SV + l;
    } else if (PANEL && (C || !(slot & 1 || slot == 4))) {
      op = slot < 2 ? 0 : 2;
      part = C ? (slot < 2 ? slot : slot - 3) : -1;
      r = C ? 2 * v + part : v;
      if (slot >= 2) src = SV + l;
    }
    if (!C && slot == 3 && PANEL && v < nv) {
      op = 2;
      r = v;
      src = SV + l;
    }
    if (op < 0 || op >= npk) continue;
    const SgOperand &o = pk.op[op];
    const double *row = t[src];
    const int em = s_e[src];
    if (g == 0) o.e[r] = em;
    sg_store_group(o, r, g, em, [&](int j) {
      const int k = 8 * g + j;
      if (part < 0) return row[k];
      const double z = row[(k & ~1) | ((k ^ part) & 1)];
      return part == 0 && (k & 1) ? -z : z;
    });
  }
}

// ------------------------------------------------------------- unit-triangular multi-vector solves
// Vectors v < nv, element i < nb at X[v vs + i es]; the nb x nb block L (element (i, j) at
// L[i + j ldl]) in shared memory:
//   TRANS = false: L y = x (unit lower; forward), TRANS = true: L^T y = x (backward).
// PANEL (forward only): the panel of the factorisation, W = y (element (v, j) at W[v + j ldw]) and
// x = y / d_j.  Vectors nv .. nv + nv2 - 1 are those of a second array (the right-hand sides).
// A CTA takes SV vectors with one thread per (element, vector), vectors fastest, and eliminates column by
// column (at step j, y_j is final and every later element subtracts its multiple): a warp holds 32 / SV
// elements, so warps whose elements are final drop out and the float64 pipe does little more than the
// triangle's own multiply-adds.
template <typename T>
struct Vecs {
  T *X;
  long long vs, es;
};
template <typename T, int NB, int SV, bool TRANS, bool PANEL>
__global__ void __launch_bounds__(NB * SV) k_trsv(int nb, const T *__restrict__ L, long long ldl, int nv, Vecs<T> X,
                                                  int nv2, Vecs<T> X2, T *__restrict__ W, long long ldw,
                                                  const T *__restrict__ dinv, const __grid_constant__ SgPack pk, int npk,
                                                  int nsolve) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  if ((int)blockIdx.x >= nsolve) {
    pack_left(pk.op[0], (int)blockIdx.x - nsolve, reinterpret_cast<double(*)[kPK + 1]>(smem_raw));
    return;
  }
  T *Ls = reinterpret_cast<T *>(smem_raw);  // Ls[i + j NB] = L(i, j), or L(j, i) for TRANS
  T *xs = Ls + NB * NB;                     // [element][vector]
  const int tid = threadIdx.x, vl = tid % SV, i = tid / SV, v = blockIdx.x * SV + vl;
  grid_wait();
  for (int e = tid; e < NB * NB; e += NB * SV) {
    const int r = e % NB, c = e / NB;
    if (r < nb && c < nb && (TRANS ? r < c : r > c)) Ls[e] = TRANS ? L[c + (long long)r * ldl] : L[r + (long long)c * ldl];
  }
  const bool act = v < nv + nv2 && i < nb;
  T *x = nullptr;
  if (act) x = v < nv ? X.X + v * X.vs + i * X.es : X2.X + (v - nv) * X2.vs + i * X2.es;
  T xi = act ? *x : Ar<T>::zero();
  const T di = PANEL && act ? dinv[i] : Ar<T>::zero();
  if (i == (TRANS ? nb - 1 : 0)) xs[tid] = xi;
  // step j reads element j (final and published after step j - 1) and changes later elements only
  if (!TRANS) {
    for (int j = 0; j + 1 < nb; ++j) {
      __syncthreads();
      if (i > j && i < nb) {
        xi = Ar<T>::fms(Ls[i + j * NB], xs[j * SV + vl], xi);
        if (i == j + 1) xs[tid] = xi;
      }
    }
  } else {
    for (int j = nb - 1; j > 0; --j) {
      __syncthreads();
      if (i < j) {
        xi = Ar<T>::fms(Ls[i + j * NB], xs[j * SV + vl], xi);
        if (i == j - 1) xs[tid] = xi;
      }
    }
  }
  T yi = xi;
  if (act) {
    if (PANEL) {
      W[v + (long long)i * ldw] = xi;
      yi = Ar<T>::mul(xi, di);
    }
    *x = yi;
  }
  if (npk > 0) {
    if (PANEL) {
      const int b = pivot_balance(di);
      xi = Ar<T>::pow2(xi, b);
      yi = Ar<T>::pow2(yi, -b);
    }
    __syncthreads();  // L and the vectors in shared memory have been read
    pack_vectors<T, SV, PANEL>(pk, npk, blockIdx.x * SV, nv, nv2, i, vl, xi, yi,
                               reinterpret_cast<double(*)[kPK + 1]>(smem_raw));
  }
}

template <typename F>
int set_smem(F *f, size_t bytes) {
  return cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes) == cudaSuccess
             ? GINT_OK
             : GINT_ECUDA;
}

// Operand views and C strides of real and complex column-major blocks.
inline SgView left(const double *p, long long sr, long long sk) { return sg_real(p, sr, sk); }
inline SgView left(const double2 *p, long long sr, long long sk) { return sg_cplx_left(p, sr, sk); }
inline SgView right(const double *p, long long sr, long long sk) { return sg_real(p, sr, sk); }
inline SgView right(const double2 *p, long long sr, long long sk) { return sg_cplx_right(p, sr, sk); }
// C (M x N, column-major, leading dimension ldc) -= A B with contraction K (all in elements of T)
template <typename T>
SgProduct update(int mode, int M, int N, int K, SgView A, SgView B, T *C, long long ldc) {
  constexpr int c = sizeof(T) == 16 ? 1 : 0, u = 1 + c;  // reals per element
  SgProduct p{};
  p.M = u * M;
  p.N = N;
  p.K = u * K;
  p.mode = mode;
  p.cs = c;
  p.neg = 1;
  p.beta = 1;
  p.A = A;
  p.B = B;
  p.C = reinterpret_cast<double *>(C);
  p.crh = 2;
  p.crl = 1;
  p.cch = 2 * u * ldc;
  p.ccl = u * ldc;
  return p;
}

template <typename T, int SV, bool TRANS, bool PANEL>
int trsv(int nb, const T *L, long long ldl, int nv, Vecs<T> X, int nv2, Vecs<T> X2, T *W, long long ldw, const T *dinv,
         const SgPack &pk, int npk, cudaStream_t st) {
  constexpr int NB = LdlBlock<T>::NB;
  const size_t smem = (size_t)(NB * NB + NB * SV) * sizeof(T);
  if (set_smem(k_trsv<T, NB, SV, TRANS, PANEL>, smem) != GINT_OK) return GINT_ECUDA;
  const int nsolve = (nv + nv2 + SV - 1) / SV, nleft = !PANEL && npk > 0 ? pk.first[1] : 0;
  return sg_launch(k_trsv<T, NB, SV, TRANS, PANEL>, dim3((unsigned)(nsolve + nleft)), NB * SV, smem, st, nb, L, ldl, nv, X, nv2,
                   X2, W, ldw, dinv, pk, npk, nsolve);
}

}  // namespace

template <typename T>
int ldl_factor_solve(int n, T *A, long long lda, int nrhs, T *B, long long ldb, T *work, int *info, bool spd,
                     const SgWork &ws, cudaStream_t st) {
  constexpr int NB = LdlBlock<T>::NB;
  int rc;
  const long long ldw = (long long)n + nrhs;
  T *W = work, *dinv = work + ldw * NB;
  for (int j0 = 0; j0 < n; j0 += NB) {
    const int nb = std::min(NB, n - j0), m = n - j0 - nb;
    T *A11 = A + j0 + (long long)j0 * lda, *A21 = A11 + nb, *B1 = B + j0;
    if ((rc = sg_launch(k_ldl_diag<T>, dim3(1), kDT, 0, st, nb, A11, lda, j0, spd ? 1 : 0, info, dinv + j0))) return rc;
    // A22 -= W21 L21^T (lower triangle), B2 -= L21 W_B^T
    const SgProduct pr[2] = {
        update<T>(1, m, m, nb, left(W, 1, ldw), right(A21, 1, lda), A21 + (long long)nb * lda, lda),
        update<T>(0, m, nrhs, nb, left(A21, 1, lda), right(W + m, 1, ldw), B1 + nb, ldb)};
    const int np = nrhs > 0 ? 2 : 1;
    SgPack pk{};
    if (m > 0 && (rc = sg_operands(pr, np, ws, &pk))) return rc;
    // panel rows: W = A21 L11^-T, L21 = W D1^-1, and the same for the right-hand sides
    if (m + nrhs > 0 && (rc = trsv<T, 8, false, true>(nb, A11, lda, m, Vecs<T>{A21, 1, lda}, nrhs, Vecs<T>{B1, ldb, 1}, W,
                                                      ldw, dinv + j0, pk, m > 0 ? 2 * np : 0, st)))
      return rc;
    if (m == 0) continue;
    if ((rc = sg_gemm(pr, np, ws, st, true))) return rc;
  }
  // L^T X = Y, last block first, then the rows above
  for (int k0 = ((n - 1) / NB) * NB; k0 >= 0 && nrhs > 0; k0 -= NB) {
    const int nb = std::min(NB, n - k0);
    const T *Lkk = A + k0 + (long long)k0 * lda;
    // rows i < k0: B_i -= sum_k L[k0 + k, i] X[k0 + k]
    const SgProduct pr = update<T>(0, k0, nrhs, nb, left(A + k0, lda, 1), right(B + k0, ldb, 1), B, ldb);
    SgPack pk{};
    if (k0 > 0 && (rc = sg_operands(&pr, 1, ws, &pk))) return rc;
    if ((rc = trsv<T, 8, true, false>(nb, Lkk, lda, nrhs, Vecs<T>{B + k0, ldb, 1}, 0, Vecs<T>{}, nullptr, 0, nullptr, pk,
                                      k0 > 0 ? 2 : 0, st)))
      return rc;
    if (k0 == 0) continue;
    if ((rc = sg_gemm(&pr, 1, ws, st, true))) return rc;
  }
  return GINT_OK;
}

template int ldl_factor_solve<double>(int, double *, long long, int, double *, long long, double *, int *, bool,
                                      const SgWork &, cudaStream_t);
template int ldl_factor_solve<double2>(int, double2 *, long long, int, double2 *, long long, double2 *, int *, bool,
                                       const SgWork &, cudaStream_t);

}  // namespace gla
