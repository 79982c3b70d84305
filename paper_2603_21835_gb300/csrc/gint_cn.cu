// gint_cn.cu -- the dense steps of real-time propagation around the grid passes: the density matrix
// from coefficients and occupations, D = Re(psi diag(f) psi^dagger), one Crank-Nicolson step of the
// coefficients, (S + i dt/2 H) psi(t + dt) = (S - i dt/2 H) psi(t) (paper Sec. 2: the density matrix
// and the time propagation of the coefficients with the overlap matrix), and the energy-density
// matrix E = (S^{-1} H D + D H S^{-1}) / 2.  All in float64 on this library's own kernels
// (gint_sg.cu: float64 products from exact digit products on the tensor cores; gint_la.cu: blocked
// L D L^T and its solves); the density matrix also has a mixed-precision build (float16 three-term split,
// gint_dm.cu).  A context holds every buffer, so the compute calls allocate nothing.
//
// The step solves A X = S psi with A = S + i dt/2 H and returns 2 X - psi, which equals
// A^{-1} (S - i dt/2 H) psi since S - i dt/2 H = 2 S - A: a real-by-complex product replaces the
// complex one, and A is factored as L D L^T (A^T = A) instead of by a general LU.
#include <cuda_runtime.h>

#include <algorithm>

#include "gint.h"
#include "gint_dm.cuh"
#include "gint_la.cuh"
#include "gint_sgpack.cuh"

namespace {

// The steps work in the basis t_i phi_i, t_i the power of two that brings the norm sqrt(S_ii) next to 1 (between
// 2^-1/2 and 2^1/2).  Digit products scale an operand by its rows' largest elements, so a contraction over basis
// functions of very different norms would lose the bits of the small ones, which float64's own exponents keep; scaled
// by powers of two, nothing is rounded, and the results do not depend on such a scaling of the basis at all.  Normalised
// functions have t = 1.
__device__ __forceinline__ int eq_exp(double s) {  // t = 2^-eq_exp
  const int e = (__double2hiint(s) >> 20) & 0x7ff;
  return e == 0 || e == 0x7ff ? 0 : (e - 1023 + 1) >> 1;
}

// F = t S t, or (H not null) the complex t (S + i dt/2 H) t (S, H real symmetric: row- and column-major alike);
// eq[0 .. n) = log2 t, eq[n .. 2 n) = -log2 t
template <typename T>
__global__ void __launch_bounds__(256) k_cn_mat(int n, const double *__restrict__ S, const double *__restrict__ H,
                                                double half_dt, T *__restrict__ F, int *__restrict__ eq) {
  const int i = blockIdx.x * 256 + threadIdx.x;
  if (i >= n) return;
  const int p = eq_exp(S[i + (long long)i * n]);
  if (blockIdx.y == 0) {
    eq[i] = -p;
    eq[n + i] = p;
  }
  for (int j = blockIdx.y; j < n; j += gridDim.y) {
    const long long e = i + (long long)j * n;
    const double s = S[e];
    const int q = -p - eq_exp(S[j + (long long)j * n]);
    if constexpr (sizeof(T) == 16)
      F[e] = make_double2(gla::times_pow2(s, q), gla::times_pow2(half_dt * H[e], q));
    else
      F[e] = gla::times_pow2(s, q);
  }
}
dim3 mat_grid(int n) { return dim3((unsigned)((n + 255) / 256), (unsigned)std::min(n, 16384)); }

// X <- 2 t X - psi (rows of n)
__global__ void k_cn_finish(int n, int k, const double2 *__restrict__ psi, double2 *__restrict__ X,
                            const int *__restrict__ lt) {
  const int i = blockIdx.x * 256 + threadIdx.x;
  if (i >= n) return;
  const double s = __hiloint2double((1023 + 1 + lt[i]) << 20, 0);
  for (int c = blockIdx.y; c < k; c += gridDim.y) {
    const long long e = i + (long long)c * n;
    const double2 x = X[e], p = psi[e];
    X[e] = make_double2(s * x.x - p.x, s * x.y - p.y);
  }
}

// E = (t X + (t X)^T) / 2 (n x n; X column-major)
__global__ void k_sym_half(int n, const double *__restrict__ X, const int *__restrict__ lt, double *__restrict__ E) {
  const int i = blockIdx.x * 256 + threadIdx.x;
  if (i >= n) return;
  const int li = lt[i];
  for (int j = blockIdx.y; j < n; j += gridDim.y)
    E[i + (long long)j * n] = 0.5 * (gla::times_pow2(X[i + (long long)j * n], li) + gla::times_pow2(X[j + (long long)i * n], lt[j]));
}

}  // namespace

struct gint_cn {
  int n = 0, nocc = 0, device = 0;
  double2 *A = nullptr;        // n x n: the factor (complex), or two real n x n matrices (gint_edm)
  double2 *work = nullptr;     // the factorisation's panel workspace (gla::ldl_work)
  gla::SgWork sg{};            // scratch of the float64 products
  int *eq = nullptr;           // 2 n: the basis scaling of the call (k_cn_mat)
  int *info = nullptr;
  void *dmw = nullptr;         // tensor-core density-matrix build: packed operands and scales
  unsigned *status = nullptr;  // its device error word
};

extern "C" {

int gint_cn_destroy(gint_cn *c) {
  if (!c) return GINT_OK;
  cudaSetDevice(c->device);
  cudaFree(c->A);
  cudaFree(c->work);
  cudaFree(c->sg.buf);
  cudaFree(c->eq);
  cudaFree(c->info);
  cudaFree(c->dmw);
  cudaFree(c->status);
  delete c;
  return GINT_OK;
}

int gint_cn_create(int n, int nocc, gint_cn **out) {
  if (!out || n <= 0 || nocc <= 0) return GINT_EINVAL;
  *out = nullptr;
  gint_cn *c = new gint_cn;
  c->n = n;
  c->nocc = nocc;
  cudaGetDevice(&c->device);
  const size_t nn = (size_t)n * n;
  // panels of the step (complex, nocc right-hand sides) and of the energy-density matrix (real, n)
  const size_t work = std::max(gla::ldl_work<double2>(n, nocc) * sizeof(double2), gla::ldl_work<double>(n, n) * sizeof(double));
  // products: S psi and H D (right rows: 2 nocc or n), the density matrix (contraction 2 nocc), the panels
  c->sg.bytes = std::max({gla::sg_bytes(n + std::max((long long)n, 2LL * nocc), n), gla::sg_bytes(2LL * n, 2LL * nocc),
                          gla::sg_bytes(gla::ldl_rows<double2>(n, nocc), 64), gla::sg_bytes(gla::ldl_rows<double>(n, n), 64)});
  if (cudaDeviceGetAttribute(&c->sg.num_sms, cudaDevAttrMultiProcessorCount, c->device) != cudaSuccess ||
      cudaMalloc(&c->A, nn * sizeof(double2)) != cudaSuccess || cudaMalloc(&c->work, work) != cudaSuccess ||
      cudaMalloc(&c->sg.buf, c->sg.bytes) != cudaSuccess || cudaMalloc(&c->eq, 2 * (size_t)n * sizeof(int)) != cudaSuccess ||
      cudaMalloc(&c->info, sizeof(int)) != cudaSuccess || cudaMalloc(&c->dmw, gint_dm_tc_bytes(n, nocc)) != cudaSuccess ||
      cudaMalloc(&c->status, sizeof(unsigned)) != cudaSuccess ||
      cudaMemset(c->info, 0, sizeof(int)) != cudaSuccess || cudaMemset(c->status, 0, sizeof(unsigned)) != cudaSuccess) {
    cudaGetLastError();
    gint_cn_destroy(c);
    return GINT_ENOMEM;
  }
  c->sg.status = c->status;
  *out = c;
  return GINT_OK;
}

int gint_cn_step(gint_cn *c, const double *S, const double *H, double dt, const double *psi, double *psi_out,
                 void *stream) {
  if (!c || !S || !H || !psi || !psi_out || psi == psi_out) return GINT_EINVAL;
  cudaStream_t st = (cudaStream_t)stream;
  const int n = c->n, k = c->nocc;
  const long long nn = (long long)n * n;
  double2 *X = reinterpret_cast<double2 *>(psi_out);
  if (cudaMemsetAsync(c->info, 0, sizeof(int), st) != cudaSuccess) return GINT_ECUDA;
  k_cn_mat<double2><<<mat_grid(n), 256, 0, st>>>(n, S, H, 0.5 * dt, c->A, c->eq);
  if (cudaGetLastError() != cudaSuccess) return GINT_ECUDA;
  // X = (t S t) (psi / t) as one real product: column 2 c + part of the interleaved complex arrays
  gla::SgProduct p{};
  p.M = p.K = n;
  p.N = 2 * k;
  p.A = gla::sg_real(S, 1, n);
  p.B = gla::SgView{psi, 2LL * n, 1, 4, 2, 0, nullptr};
  p.A.rp = p.A.kp = c->eq;
  p.B.kp = c->eq + n;
  p.C = psi_out;
  p.crh = 4;
  p.crl = 2;
  p.cch = 2LL * n;
  p.ccl = 1;
  int rc = gla::sg_gemm(&p, 1, c->sg, st);
  if (rc) return rc;
  if ((rc = gla::ldl_factor_solve<double2>(n, c->A, n, k, X, n, c->work, c->info, false, c->sg, st))) return rc;
  k_cn_finish<<<dim3((unsigned)((n + 255) / 256), (unsigned)std::min(k, 16384)), 256, 0, st>>>(
      n, k, reinterpret_cast<const double2 *>(psi), X, c->eq);
  return cudaGetLastError() == cudaSuccess ? GINT_OK : GINT_ECUDA;
}

int gint_dm_build(gint_cn *c, const double *psi, const double *f, double *D, void *stream) {
  if (!c || !psi || !f || !D) return GINT_EINVAL;
  const int n = c->n;
  // D = A B^T over k = 2 s + (real, imaginary part): A_ik = f_s psi_is, B_ik = psi_is (real views), with the power of
  // two next to |f_s|^(1/2) moved from A to B: the row maxima that the digits are relative to are then at most
  // about D_ii^(1/2), so a function that lives in states of small occupation keeps its bits;
  // the lower triangle is computed and mirrored, so D is symmetric bit for bit
  gla::SgProduct p{};
  p.M = p.N = n;
  p.K = 2 * c->nocc;
  p.mode = 2;
  p.A = gla::SgView{psi, 4, 2, 2LL * n, 1, 0, f, 1};
  p.B = gla::SgView{psi, 4, 2, 2LL * n, 1, 0, f, 2};
  p.C = D;
  p.crh = 2;
  p.crl = 1;
  p.cch = 2LL * n;
  p.ccl = n;
  return gla::sg_gemm(&p, 1, c->sg, (cudaStream_t)stream);
}

int gint_dm_build_f16x3(gint_cn *c, const double *psi, const double *f, double *D, void *stream) {
  if (!c || !psi || !f || !D) return GINT_EINVAL;
  return gint_dm_tc(c->n, c->nocc, psi, f, D, c->dmw, c->status, (cudaStream_t)stream);
}

int gint_edm(gint_cn *c, const double *S, const double *H, const double *D, double *E, void *stream) {
  if (!c || !S || !H || !D || !E) return GINT_EINVAL;
  cudaStream_t st = (cudaStream_t)stream;
  const int n = c->n;
  // the complex n x n buffer holds two real n x n matrices: F (the factor of S) and X
  double *F = reinterpret_cast<double *>(c->A), *X = F + (size_t)n * n;
  if (cudaMemsetAsync(c->info, 0, sizeof(int), st) != cudaSuccess) return GINT_ECUDA;
  k_cn_mat<double><<<mat_grid(n), 256, 0, st>>>(n, S, nullptr, 0.0, F, c->eq);
  if (cudaGetLastError() != cudaSuccess) return GINT_ECUDA;
  // X = (t H t) (D / t), then X <- (t S t)^{-1} X (t S t = L D L^T), E = (t X + (t X)^T) / 2
  gla::SgProduct p{};
  p.M = p.N = p.K = n;
  p.A = gla::sg_real(H, 1, n);
  p.B = gla::sg_real(D, n, 1);
  p.A.rp = p.A.kp = c->eq;
  p.B.kp = c->eq + n;
  p.C = X;
  p.crh = 2;
  p.crl = 1;
  p.cch = 2LL * n;
  p.ccl = n;
  int rc = gla::sg_gemm(&p, 1, c->sg, st);
  if (rc) return rc;
  if ((rc = gla::ldl_factor_solve<double>(n, F, n, n, X, n, reinterpret_cast<double *>(c->work), c->info, true, c->sg, st)))
    return rc;
  k_sym_half<<<mat_grid(n), 256, 0, st>>>(n, X, c->eq, E);
  return cudaGetLastError() == cudaSuccess ? GINT_OK : GINT_ECUDA;
}

int gint_cn_info(gint_cn *c, int *info) {
  if (!c || !info) return GINT_EINVAL;
  unsigned st = 0;
  if (cudaMemcpy(info, c->info, sizeof(int), cudaMemcpyDeviceToHost) != cudaSuccess ||
      cudaMemcpy(&st, c->status, sizeof(unsigned), cudaMemcpyDeviceToHost) != cudaSuccess)
    return GINT_ECUDA;
  if (st != 0) {
    cudaMemset(c->status, 0, sizeof(unsigned));
    return GINT_ETIMEDOUT;
  }
  return GINT_OK;
}

}  // extern "C"
