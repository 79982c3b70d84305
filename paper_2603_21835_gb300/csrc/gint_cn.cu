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

namespace {

// A = S + i dt/2 H (S, H real symmetric: row- and column-major alike)
__global__ void k_cn_mat(long long nn, const double *__restrict__ S, const double *__restrict__ H, double half_dt,
                         double2 *__restrict__ A) {
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < nn; e += (long long)gridDim.x * blockDim.x)
    A[e] = make_double2(S[e], half_dt * H[e]);
}

// X <- 2 X - psi
__global__ void k_cn_finish(long long m, const double2 *__restrict__ psi, double2 *__restrict__ X) {
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < m; e += (long long)gridDim.x * blockDim.x) {
    const double2 x = X[e], p = psi[e];
    X[e] = make_double2(2.0 * x.x - p.x, 2.0 * x.y - p.y);
  }
}

// E = (X + X^T) / 2 (n x n)
__global__ void k_sym_half(int n, const double *__restrict__ X, double *__restrict__ E) {
  const long long nn = (long long)n * n;
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < nn; e += (long long)gridDim.x * blockDim.x) {
    const long long i = e / n, j = e - i * n;
    E[e] = 0.5 * (X[e] + X[j * n + i]);
  }
}

unsigned blocks_for(long long n) { return (unsigned)std::min<long long>((n + 255) / 256, 4096); }

}  // namespace

struct gint_cn {
  int n = 0, nocc = 0, device = 0;
  double2 *A = nullptr;        // n x n: the factor (complex), or two real n x n matrices (gint_edm)
  double2 *work = nullptr;     // the factorisation's panel workspace (gla::ldl_work)
  gla::SgWork sg{};            // scratch of the float64 products
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
      cudaMalloc(&c->sg.buf, c->sg.bytes) != cudaSuccess ||
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
  k_cn_mat<<<blocks_for(nn), 256, 0, st>>>(nn, S, H, 0.5 * dt, c->A);
  if (cudaGetLastError() != cudaSuccess) return GINT_ECUDA;
  // X = S psi as one real product: column 2 c + part of the interleaved complex arrays
  gla::SgProduct p{};
  p.M = p.K = n;
  p.N = 2 * k;
  p.A = gla::sg_real(S, 1, n);
  p.B = gla::SgView{psi, 2LL * n, 1, 4, 2, 0, nullptr};
  p.C = psi_out;
  p.crh = 4;
  p.crl = 2;
  p.cch = 2LL * n;
  p.ccl = 1;
  int rc = gla::sg_gemm(&p, 1, c->sg, st);
  if (rc) return rc;
  if ((rc = gla::ldl_factor_solve<double2>(n, c->A, n, k, X, n, c->work, c->info, false, c->sg, st))) return rc;
  k_cn_finish<<<blocks_for((long long)n * k), 256, 0, st>>>((long long)n * k, reinterpret_cast<const double2 *>(psi), X);
  return cudaGetLastError() == cudaSuccess ? GINT_OK : GINT_ECUDA;
}

int gint_dm_build(gint_cn *c, const double *psi, const double *f, double *D, void *stream) {
  if (!c || !psi || !f || !D) return GINT_EINVAL;
  const int n = c->n;
  // D = A B^T over k = 2 s + (real, imaginary part): A_ik = f_s psi_is, B_ik = psi_is (real views);
  // the lower triangle is computed and mirrored, so D is symmetric bit for bit
  gla::SgProduct p{};
  p.M = p.N = n;
  p.K = 2 * c->nocc;
  p.mode = 2;
  p.A = gla::SgView{psi, 4, 2, 2LL * n, 1, 0, f};
  p.B = gla::SgView{psi, 4, 2, 2LL * n, 1, 0, nullptr};
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
  if (cudaMemsetAsync(c->info, 0, sizeof(int), st) != cudaSuccess ||
      cudaMemcpyAsync(F, S, (size_t)n * n * sizeof(double), cudaMemcpyDeviceToDevice, st) != cudaSuccess)
    return GINT_ECUDA;
  // X = H D, then X <- S^{-1} X (S = L D L^T), E = (X + X^T) / 2
  gla::SgProduct p{};
  p.M = p.N = p.K = n;
  p.A = gla::sg_real(H, 1, n);
  p.B = gla::sg_real(D, n, 1);
  p.C = X;
  p.crh = 2;
  p.crl = 1;
  p.cch = 2LL * n;
  p.ccl = n;
  int rc = gla::sg_gemm(&p, 1, c->sg, st);
  if (rc) return rc;
  if ((rc = gla::ldl_factor_solve<double>(n, F, n, n, X, n, reinterpret_cast<double *>(c->work), c->info, true, c->sg, st)))
    return rc;
  k_sym_half<<<blocks_for((long long)n * n), 256, 0, st>>>(n, X, E);
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
