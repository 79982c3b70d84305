// gint_internal.cuh -- device-side data structures and orbital evaluation shared by the
// libgint kernels.
//
// Orbital evaluation follows Eq. 1 of the paper (phi = f_{I l zeta}(r) Y_lm(r^)), periodised
// over lattice images at the Gamma point (Eq. 2 with k = 0).  Radials are cubic Hermite
// interpolants of tabulated (f, f') samples; Y_lm are real, orthonormal, no Condon-Shortley
// sign, l <= 2, m ordered 0, +1, -1, +2, -2.  A grid point within 1e-12 Bohr of an atom
// takes the r -> 0 limit (s: f(0) Y00; p gradient: f'(0) sqrt(3/4pi) e_m; the rest 0).
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "gint.h"

#define GINT_MAX_SPECIES 8
#define GINT_MAX_RADIAL 64
#define GINT_MAX_ORB_ATOM 32      // orbitals of one atom
#define GINT_MAX_ATOMS_BRICK 64   // distinct atoms covering one brick (coverage masks are 64-bit)
#define GINT_BI 4                 // brick extent along grid axis 1
#define GINT_BJ 4                 // ... axis 2
#define GINT_BK 8                 // ... axis 3 (contiguous in memory)
#define GINT_BPTS (GINT_BI * GINT_BJ * GINT_BK)  // 128 points = one tcgen05 M tile

struct GRadial {
  int l, npts, off, pad;  // off: first knot of this radial in the packed tables
  double dr, inv_dr, rc, rc2;
  float idr_hi, idr_lo, rc_f, dr_f;  // float32 images: 1/dr as hi + lo, rc, dr
};

struct GSpecies {
  int nrad, rad0, norb, porb;  // porb: orbitals padded to a multiple of 8 (tensor-core layouts)
  int shape;                   // (ns, np, nd) code 1 + ns + 8 np + 64 nd when the radials are l-sorted and
                               // share one knot grid (same npts and dr); 0 otherwise
  float rcut2f;                // rcut2 rounded to float32 (coarse support test of the float32 kernels)
  int ioff, kslot;             // shaped species: interleaved float32 table [knot][kslot] of (f, f') at
                               // float2 offset ioff, kslot = radials rounded up to even; 0 otherwise
  double rcut, rcut2;          // largest rc of the species and its square
};
#define GINT_SHAPE(ns, np, nd) (1 + (ns) + 8 * (np) + 64 * (nd))

// Geometry of one system: cell, grid and bricks.
struct GCell {
  double cell[9];   // rows a1, a2, a3
  double inv[9];    // inverse: fractional u = d . inv
  double reach[3];  // |column c of inv| (fractional extent of a unit Cartesian length)
  double w;         // grid weight
  long long ngrid, nbricks;
  int n1, n2, n3;
  int nbi, nbj, nbk;  // bricks per axis
  int natoms, pad;
};

// Species and radial-table metadata (the knot values live in a separate packed array).
// Systems whose GTabs compare equal byte for byte can share one batched launch.
struct GTabs {
  int nspecies, nrad;
  GSpecies sp[GINT_MAX_SPECIES];
  GRadial rad[GINT_MAX_RADIAL];
};

struct GGeom : GCell, GTabs {};

// Neighbour structure of the bricks (device arrays, CSR).
//   bricks  : b_at_off[b] .. b_at_off[b+1]  distinct atoms of brick b ("slots")
//   slots   : s_atom[k], s_col[k] (first column of the atom in the brick's orbital space),
//             s_ent[k] .. s_ent[k+1]  its (atom, image) entries
//   entries : e_shift[e] = tau_I + R (Cartesian, float64, 3 per entry)
//   pairs   : b_pair_off[b] .. : n_a x n_a table of global pair indices (-1: no block)
struct GNbr {
  const long long *b_at_off;
  const int *b_norb;
  const int *s_atom;
  const int *s_col;
  const long long *s_ent;
  const double *e_shift;
  const long long *b_pair_off;
  const int *b_pair;
  const long long *pair_off;  // element offset of each pair block
  const int *atom_species;
};

#define GINT_PI 3.14159265358979323846

__host__ __device__ __forceinline__ void grid_point(const GCell &g, int i, int j, int k, double r[3]) {
  double fi = (double)i / g.n1, fj = (double)j / g.n2, fk = (double)k / g.n3;
#pragma unroll
  for (int c = 0; c < 3; ++c) r[c] = fi * g.cell[c] + fj * g.cell[3 + c] + fk * g.cell[6 + c];
}

// Decode a local point index 0..127 of a brick into grid indices; returns false outside the grid.
// (brick indices fit 32 bits: gint_create refuses grids of 2^31 bricks or more, so the divisions
// are 32-bit ones, several times cheaper on the GPU than 64-bit ones)
__host__ __device__ __forceinline__ bool brick_point(const GCell &g, long long b, int p, int &i, int &j, int &k) {
  const unsigned ub = (unsigned)b, nbk = (unsigned)g.nbk, q = ub / nbk;
  const int bk = (int)(ub - q * nbk);
  const int bj = (int)(q % (unsigned)g.nbj);
  const int bi = (int)(q / (unsigned)g.nbj);
  int pk = p % GINT_BK, pj = (p / GINT_BK) % GINT_BJ, pi = p / (GINT_BK * GINT_BJ);
  i = bi * GINT_BI + pi;
  j = bj * GINT_BJ + pj;
  k = bk * GINT_BK + pk;
  return i < g.n1 && j < g.n2 && k < g.n3;
}

__host__ __device__ __forceinline__ long long grid_index(const GCell &g, int i, int j, int k) {
  return ((long long)i * g.n2 + j) * g.n3 + k;
}

// ------------------------------------------------------------------------------------------
// Radial: cubic Hermite on uniform knots. tab[k] = (f_k, f'_k).
template <typename T>
struct Tab2;
template <>
struct Tab2<double> { typedef double2 type; };
template <>
struct Tab2<float> { typedef float2 type; };

// dtab (may be NULL): f_{k+1} - f_k per knot formed in float64 (for float32 tables; see the handle)
template <typename T>
__device__ __forceinline__ void radial_eval(const typename Tab2<T>::type *__restrict__ tab, const GRadial &R, T r,
                                            T &f, T &df, const float *__restrict__ dtab = nullptr) {
  T x = r * (T)R.inv_dr;
  int i = (int)x;
  if (i >= R.npts - 1) {
    f = 0;
    df = 0;
    return;
  }
  T t = x - (T)i;
  typename Tab2<T>::type a = tab[R.off + i], b = tab[R.off + i + 1];
  T dr = (T)R.dr;
  T g0 = a.y * dr, g1 = b.y * dr;
  T t2 = t * t;
  const T dlt = dtab ? (T)dtab[R.off + i] : b.x - a.x;
  // Hermite basis in nested form: h00 = 1 - t^2 (3 - 2t), h01 = t^2 (3 - 2t),
  // h10 = t (1 - t)^2, h11 = t^2 (t - 1)
  T s = t2 * ((T)3 - (T)2 * t);
  T u = (T)1 - t;
  f = a.x + dlt * s + g0 * t * u * u + g1 * t2 * (t - (T)1);
  // derivatives: dh01 = 6 t (1 - t) = -dh00, dh10 = (1 - t)(1 - 3t), dh11 = t (3t - 2)
  df = (dlt * (T)6 * t * u + g0 * u * ((T)1 - (T)3 * t) + g1 * t * ((T)3 * t - (T)2)) * (T)R.inv_dr;
}

// ------------------------------------------------------------------------------------------
// Real solid-harmonic polynomials evaluated on the unit vector (ux,uy,uz): y[m] and grad y[m].
template <typename T>
__device__ __forceinline__ void ylm_unit(int l, T ux, T uy, T uz, T *y, T (*gy)[3]) {
  if (l == 0) {
    y[0] = (T)(0.28209479177387814347);  // 1/(2 sqrt(pi))
    gy[0][0] = gy[0][1] = gy[0][2] = 0;
  } else if (l == 1) {
    const T c = (T)(0.48860251190291992159);  // sqrt(3/(4pi))
    y[0] = c * uz; gy[0][0] = 0; gy[0][1] = 0; gy[0][2] = c;
    y[1] = c * ux; gy[1][0] = c; gy[1][1] = 0; gy[1][2] = 0;
    y[2] = c * uy; gy[2][0] = 0; gy[2][1] = c; gy[2][2] = 0;
  } else {
    const T c0 = (T)(0.31539156525252000603);  // sqrt(5/(16pi))
    const T c1 = (T)(1.09254843059207907054);  // sqrt(15/(4pi))
    const T c2 = (T)(0.54627421529603953527);  // sqrt(15/(16pi))
    y[0] = c0 * ((T)2 * uz * uz - ux * ux - uy * uy);
    gy[0][0] = -(T)2 * c0 * ux; gy[0][1] = -(T)2 * c0 * uy; gy[0][2] = (T)4 * c0 * uz;
    y[1] = c1 * ux * uz; gy[1][0] = c1 * uz; gy[1][1] = 0; gy[1][2] = c1 * ux;
    y[2] = c1 * uy * uz; gy[2][0] = 0; gy[2][1] = c1 * uz; gy[2][2] = c1 * uy;
    y[3] = c2 * (ux * ux - uy * uy); gy[3][0] = (T)2 * c2 * ux; gy[3][1] = -(T)2 * c2 * uy; gy[3][2] = 0;
    y[4] = c1 * ux * uy; gy[4][0] = c1 * uy; gy[4][1] = c1 * ux; gy[4][2] = 0;
  }
}

template <typename T>
__device__ __forceinline__ T gsqrt(T x);
template <>
__device__ __forceinline__ double gsqrt<double>(double x) { return sqrt(x); }
template <>
__device__ __forceinline__ float gsqrt<float>(float x) { return sqrtf(x); }

// Adds the orbitals of species `sp` at displacement d (one lattice image, |d| < rcut assumed
// by the caller) to phi[0..norb) if PHI and to grad[0..norb)[3] if GRAD.
// grad phi = u (f' Y - l f Y / r) + (f / r) grad_u y(u), with Y = y(u), u = d / r.
template <typename T, bool PHI, bool GRAD>
__device__ __forceinline__ void add_orbitals(const GTabs &g, const typename Tab2<T>::type *__restrict__ tab, int sp,
                                             T dx, T dy, T dz, T *phi, T (*grad)[3],
                                             const float *__restrict__ dtab = nullptr) {
  const GSpecies &S = g.sp[sp];
  T r2 = dx * dx + dy * dy + dz * dz;
  T r = gsqrt<T>(r2);
  bool at0 = r < (T)1e-12;
  T inv_r = at0 ? (T)0 : (T)1 / r;
  T ux = dx * inv_r, uy = dy * inv_r, uz = dz * inv_r;
  int col = 0;
  for (int k = 0; k < S.nrad; ++k) {
    const GRadial &R = g.rad[S.rad0 + k];
    const int l = R.l, nm = 2 * l + 1;
    if (r < (T)R.rc) {
      T f, df;
      radial_eval<T>(tab, R, r, f, df, dtab);
      if (at0) {
        if (PHI && l == 0) phi[col] += f * (T)0.28209479177387814347;
        if (GRAD && l == 1) {
          const T c = (T)0.48860251190291992159 * df;
          grad[col + 0][2] += c;
          grad[col + 1][0] += c;
          grad[col + 2][1] += c;
        }
      } else {
        T y[5], gy[5][3];
        ylm_unit<T>(l, ux, uy, uz, y, gy);
        T a = 0, fr = 0;
        if (GRAD) {
          fr = f * inv_r;
        }
        for (int m = 0; m < nm; ++m) {
          if (PHI) phi[col + m] += f * y[m];
          if (GRAD) {
            a = df * y[m] - (T)l * fr * y[m];
            grad[col + m][0] += a * ux + fr * gy[m][0];
            grad[col + m][1] += a * uy + fr * gy[m][1];
            grad[col + m][2] += a * uz + fr * gy[m][2];
          }
        }
      }
    }
    col += nm;
  }
}

// ------------------------------------------------------------------------------------------
// Float64 evaluators of l-sorted species on one knot grid (NS s, NP p, ND d radials), for the kernels whose time is
// the number of float64 instructions (a warp-wide one occupies the SM's pipe for 16 clocks).  Tables (otab64 of the
// handle): per knot and radial the interpolant a + t (b + t (c + t d)), times the constant of Y_00, of Y_1m or of
// Y_2,+-1 (the other d functions carry their ratio to it); GSpecies::ioff: first table entry, kslot: the radials end
// at different radii.  (Three instructions a radial, two more with its derivative, and no basis: with knot values and
// slopes the basis functions of t took 7 and 13 more an image.)
#define GINT_O64_SHAPES(X) X(2, 2, 1, 13) X(2, 1, 0, 5) X(1, 1, 1, 9) X(1, 1, 0, 4) X(1, 0, 0, 1) X(3, 3, 2, 22)

// 1 / r, r and the knot position of a point with r2 = |d|^2 (below 1e-36 it counts as 1e-36).  end: at or beyond the
// last knot, where the radials are 0 (r2 may lie below the squared support radius and r round up to the radius).
struct Knot64 {
  double y, r, t;
  int i;
  bool end;
};
__device__ __forceinline__ Knot64 knot64(const GRadial &R0, double r2) {
  Knot64 K;
  if (r2 < 1e-36) {  // on the atom: f / r keeps its limit, u = d / r vanishes
    K.y = 1e18;
    K.r = 1e-18;
  } else {
    // one third-order step from the float32 reciprocal root (relative error below 2^-22): y (1 + e / 2 + 3 e^2 / 8)
    // with e = 1 - r2 y^2; r by a Newton step with an exact residual, almost correctly rounded.  Against rsqrt() the
    // evaluation kernels lost a fifth of their time (float64 instructions at 16 cycles each).
    const double y = (double)rsqrtf((float)r2), e = fma(-(r2 * y), y, 1.0);
    K.y = fma(y, e * fma(e, 0.375, 0.5), y);
    K.r = r2 * K.y;
    K.r = fma(fma(-K.r, K.r, r2), 0.5 * K.y, K.r);
  }
  // knot i = floor(r / dr), t in [0, 1] (a point on a knot may take either side)
  const double x = K.r * R0.inv_dr, big = 6755399441055744.0;  // 1.5 2^52
  const double xi = (x - 0.5) + big;  // its low bits: an integer within 1/2 of x - 1/2
  K.i = __double2loint(xi);
  K.t = x - (xi - big);
  K.end = false;
  if (K.i >= R0.npts - 2) {  // (x rounded: above, the multiplication may be fused into x - 0.5 and t)
    const double xr = __dmul_rn(K.r, R0.inv_dr);
    K.i = R0.npts - 2;
    K.t = xr - (double)K.i;
    K.end = K.t >= 1.0;
  }
  return K;
}

// phi[m] += the orbitals at displacement (dx, dy, dz), r2 below the support.
template <int NS, int NP, int ND>
__device__ __forceinline__ void orbitals64(const GTabs &g, const double *__restrict__ tab, const GSpecies &S, double dx,
                                           double dy, double dz, double r2, double *phi) {
  constexpr int NR = NS + NP + ND;
  const Knot64 K = knot64(g.rad[S.rad0], r2);
  if (K.end) return;
  const double t = K.t;
  const double2 *q = reinterpret_cast<const double2 *>(tab) + ((long long)S.ioff + (long long)K.i * NR) * 2;
  double f[NR];
#pragma unroll
  for (int k = 0; k < NR; ++k) {
    const double2 a = __ldg(q + 2 * k), b = __ldg(q + 2 * k + 1);
    f[k] = fma(fma(fma(b.y, t, b.x), t, a.y), t, a.x);
    if (S.kslot && !(K.r < g.rad[S.rad0 + k].rc)) f[k] = 0.0;
  }
  const double ux = dx * K.y, uy = dy * K.y, uz = dz * K.y;
#pragma unroll
  for (int k = 0; k < NS; ++k) phi[k] += f[k];
#pragma unroll
  for (int k = 0; k < NP; ++k) {
    double *o = phi + NS + 3 * k;
    o[0] = fma(f[NS + k], uz, o[0]);
    o[1] = fma(f[NS + k], ux, o[1]);
    o[2] = fma(f[NS + k], uy, o[2]);
  }
  if (ND > 0) {
    const double xx = ux * ux, y0 = fma(2.0 * uz, uz, -fma(uy, uy, xx)), y3 = fma(-uy, uy, xx);
    const double xz = ux * uz, yz = uy * uz, xy = ux * uy;
#pragma unroll
    for (int k = 0; k < ND; ++k) {
      double *o = phi + NS + 3 * NP + 5 * k;
      const double fk = f[NS + NP + k];
      o[0] = fma(fk * 0.28867513459481288225, y0, o[0]);  // sqrt(5/16) / sqrt(15/4)
      o[1] = fma(fk, xz, o[1]);
      o[2] = fma(fk, yz, o[2]);
      o[3] = fma(fk * 0.5, y3, o[3]);
      o[4] = fma(fk, xy, o[4]);
    }
  }
}

// rho += sum_m c_m phi_m and (gx, gy, gz) += sum_m c_m grad phi_m at the displacement, shell by shell:
// phi = R Y(u), grad phi = u (R' - l R / r) Y + (R / r) grad Y with Y the homogeneous polynomial, so a radial needs
// Y and grad Y contracted with its coefficients only.
template <int NS, int NP, int ND>
__device__ __forceinline__ void contract64(const GTabs &g, const double *__restrict__ tab, const GSpecies &S, double dx,
                                           double dy, double dz, double r2, const double *c, double &rho, double &gx,
                                           double &gy, double &gz) {
  constexpr int NR = NS + NP + ND;
  const GRadial &R0 = g.rad[S.rad0];
  const bool at0 = r2 < 1e-24;
  const Knot64 K = knot64(R0, r2);
  if (K.end) return;
  const double t = K.t, idr = R0.inv_dr;
  const double2 *q = reinterpret_cast<const double2 *>(tab) + ((long long)S.ioff + (long long)K.i * NR) * 2;
  const double ux = at0 ? 0.0 : dx * K.y, uy = at0 ? 0.0 : dy * K.y, uz = at0 ? 0.0 : dz * K.y;
  double rad = 0.0;  // coefficient of u
  auto radial = [&](int k, double &R, double &dR) {
    const double2 a = __ldg(q + 2 * k), b = __ldg(q + 2 * k + 1);
    const double h = fma(b.y, t, b.x), g1 = fma(h, t, a.y);
    R = fma(g1, t, a.x);
    dR = fma(fma(b.y, t, h), t, g1) * idr;
    if (S.kslot && !(K.r < g.rad[S.rad0 + k].rc)) R = dR = 0.0;
  };
#pragma unroll
  for (int k = 0; k < NS; ++k) {
    double R, dR;
    radial(k, R, dR);
    rho = fma(c[k], R, rho);
    rad = fma(c[k], dR, rad);
  }
#pragma unroll
  for (int k = 0; k < NP; ++k) {
    const double *o = c + NS + 3 * k;  // z, x, y
    double R, dR;
    radial(NS + k, R, dR);
    const double Rr = at0 ? dR : R * K.y, y = fma(o[0], uz, fma(o[1], ux, o[2] * uy));
    rho = fma(at0 ? 0.0 : R, y, rho);
    rad = fma(dR - Rr, y, rad);
    gx = fma(Rr, o[1], gx);
    gy = fma(Rr, o[2], gy);
    gz = fma(Rr, o[0], gz);
  }
  if (ND > 0) {
    const double xx = ux * ux, y0 = fma(2.0 * uz, uz, -fma(uy, uy, xx)), y3 = fma(-uy, uy, xx);
    const double xz = ux * uz, yz = uy * uz, xy = ux * uy;
#pragma unroll
    for (int k = 0; k < ND; ++k) {
      const double *o = c + NS + 3 * NP + 5 * k;
      double R, dR;
      radial(NS + NP + k, R, dR);
      const double a0 = o[0] * 0.28867513459481288225, a3 = o[3] * 0.5;
      const double y = fma(a0, y0, fma(o[1], xz, fma(o[2], yz, fma(a3, y3, o[4] * xy))));
      const double Rr = at0 ? 0.0 : R * K.y;
      rho = fma(at0 ? 0.0 : R, y, rho);
      rad = fma(fma(-2.0, Rr, dR), y, rad);
      gx = fma(Rr, fma(2.0 * (a3 - a0), ux, fma(o[1], uz, o[4] * uy)), gx);
      gy = fma(Rr, fma(-2.0 * (a3 + a0), uy, fma(o[2], uz, o[4] * ux)), gy);
      gz = fma(Rr, fma(4.0 * a0, uz, fma(o[1], ux, o[2] * uy)), gz);
    }
  }
  gx = fma(rad, ux, gx);
  gy = fma(rad, uy, gy);
  gz = fma(rad, uz, gz);
}

// Device error word bits.
#define GINT_ERRBIT_CAPACITY 1u
#define GINT_ERRBIT_SKIN 2u
#define GINT_ERRBIT_INDEX 4u
#define GINT_ERRBIT_TIMEOUT 8u
