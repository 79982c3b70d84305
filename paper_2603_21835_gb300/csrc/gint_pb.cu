// gint_pb.cu -- velocity-gauge nonlocal projector overlaps on atom-centred spherical grids (paper
// Sec. 3.3.2, "Spherical Grid Integration for Nonlocal Potentials"):
//   P_{j mu}^{IJ}(A) = <beta_{I j}| e^{-i A.r} |Phi_{J mu}> = int beta_{I j}(r - tau_I) e^{-i A.r} Phi_{J mu}(r) dr
// for every projector atom I and every atom J whose orbitals reach I's projectors (Phi: the orbital
// summed over the lattice images of J, Gamma point).  The integral runs on a grid centred on tau_I:
// r = tau_I + x, x = r_k e_a, with 140 Gauss-Legendre radial nodes on [0, rc_beta] (weight r^2) and an
// angular rule of degree 17.  The paper uses the 110-point Lebedev-Laikov rule; its table is not
// available here, so a product rule of the same degree stands in: 9 Gauss-Legendre nodes in
// cos(theta) times 18 equally spaced azimuths (162 points).
//
// GPU organisation.  Everything is float64, which this GPU runs at 2 multiply-adds per clock and SM: a
// warp-wide float64 instruction occupies the SM's pipe for 16 clocks, and the kernel's time is the number of
// those instructions.  So what does not depend on the pair is formed once per call (k_pb_phase: quadrature
// weight times projector radial times the phase e^{-i A.x} of the point relative to tau_I; e^{-i A.tau_I}
// multiplies the sums at the end), the orbital tables hold the interpolant's polynomial coefficients times the Y_lm
// constants, and points outside an image's support cost the distance test only.  A warp takes 2 neighbouring rays
// times 16 neighbouring radial nodes at a time, a compact patch that is mostly all inside or all outside
// (32 rays of one radius, a band around the whole sphere, are rarely either), and 81 such ray pairs fill whole
// warps where 162 rays leave the last of six with two.  k_psibeta: a CTA of 3 warps (four share an SM: one's
// set-up and sums overlap the others' points; one CTA of 9 warps took 5.33 ms where this takes 4.77) works on a
// pair and a group of its ray pairs; k_pb_sum adds the groups' sums in order (no atomics).
// Inside the support 151 float64 additions, multiplications and fused ones are executed per point (12.7 of the 42.1
// million points below), outside a float32 test for the patch.
// Bound: the float64 pipe (0.88 of its cycles active).  64-atom Si, 1,856 pairs x 22,680 points: 22.9 ms
// (one CTA a pair and one thread a ray, every point evaluated in full) -> 4.62 ms.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <vector>

#include "gint_handle.cuh"

namespace {

constexpr int kPbTheta = 9, kPbPhi = 18, kPbRays = kPbTheta * kPbPhi, kPbNr = 140;
constexpr int kPbWarps = 3, kPbThreads = 32 * kPbWarps;
constexpr int kPbRayPairs = kPbRays / 2, kPbSeg = 16;  // a warp's patch: 2 rays x 16 radial nodes
constexpr int kPbMaxOrb = 16;  // orbitals of the neighbour atom (accumulators held in registers)
constexpr int kPbImages = 32;  // images of a pair staged in shared memory
constexpr int kPbGroup = 2;    // projector radials per pass over the points
constexpr double kPi = 3.14159265358979323846;
static_assert(kPbRays % 2 == 0 && kPbRayPairs % 9 == 0, "ray pairs in ninths");

__constant__ double c_ang[kPbRays][4];  // unit vector and weight (weights sum to 4 pi)
__constant__ double c_rad[kPbNr][2];    // node in (0, 1) and weight of the rule on [0, 1]

struct GPb {
  double A[3];
  const int *pI, *pJ;
  const long long *poff;
  const int *img_off;
  const double *img;  // image positions tau_J + R of the pair's neighbour atom
  const double *pos;
  const int *species;
  const double2 *tab, *ptab;  // orbital and projector tables, (f, f') per knot
  const double *otab;         // orbital tables of orbitals64
  double2 *phase;             // [projector radial][ray][node]: weight x radial x e^{-i A.x}
  const int *order;           // pairs of this launch
  double *part;               // [group][complex element]
  long long nelems;
  int ngroups;                // CTAs per pair
};

// Gauss-Legendre nodes and weights on [-1, 1] (Newton iteration on P_n from the three-term
// recurrence; initial guesses cos(pi (i + 3/4) / (n + 1/2))).
void gauss_legendre(int n, std::vector<double> &x, std::vector<double> &w) {
  x.assign(n, 0.0);
  w.assign(n, 0.0);
  for (int i = 0; i < n; ++i) {
    double z = std::cos(kPi * (i + 0.75) / (n + 0.5)), dp = 0.0;
    for (int it = 0; it < 100; ++it) {
      double p0 = 1.0, p1 = z;
      for (int k = 2; k <= n; ++k) {
        const double p2 = ((2.0 * k - 1.0) * z * p1 - (k - 1.0) * p0) / k;
        p0 = p1;
        p1 = p2;
      }
      dp = n * (z * p1 - p0) / (z * z - 1.0);  // P_n'
      const double dz = p1 / dp;
      z -= dz;
      if (std::fabs(dz) < 1e-16) break;
    }
    double p0 = 1.0, p1 = z;
    for (int k = 2; k <= n; ++k) {
      const double p2 = ((2.0 * k - 1.0) * z * p1 - (k - 1.0) * p0) / k;
      p0 = p1;
      p1 = p2;
    }
    dp = n * (z * p1 - p0) / (z * z - 1.0);
    x[i] = z;
    w[i] = 2.0 / ((1.0 - z * z) * dp * dp);
  }
}

// One thread per (projector radial, ray, node).
__global__ void __launch_bounds__(256) k_pb_phase(const __grid_constant__ GTabs prj, const __grid_constant__ GPb P) {
  const int u = blockIdx.x * 256 + threadIdx.x, rad = blockIdx.y;
  if (u >= kPbRays * kPbNr) return;
  const int a = u / kPbNr, k = u - a * kPbNr;
  double rcb = 0.0;
  for (int s = 0; s < prj.nspecies; ++s)
    if (rad >= prj.sp[s].rad0 && rad < prj.sp[s].rad0 + prj.sp[s].nrad) rcb = prj.sp[s].rcut;
  const GRadial &R = prj.rad[rad];
  const double r = rcb * c_rad[k][0], wk = rcb * c_rad[k][1] * r * r;
  double f = 0.0, df;
  if (r < R.rc) radial_eval<double>(P.ptab, R, r, f, df);
  double s, c;
  sincos(-r * (P.A[0] * c_ang[a][0] + P.A[1] * c_ang[a][1] + P.A[2] * c_ang[a][2]), &s, &c);
  f *= wk;
  P.phase[((long long)rad * kPbRays + a) * kPbNr + k] = make_double2(f * c, f * s);
}

// v[0 .. 2 H) over the lanes that differ in bit `bit`: the lane whose bit is clear keeps the sums of the first
// H, the other those of the second H.
template <int H>
__device__ __forceinline__ void halve(double *v, int bit) {
  const bool up = threadIdx.x & bit;
#pragma unroll
  for (int i = 0; i < H; ++i) {
    const double keep = up ? v[i + H] : v[i], send = up ? v[i] : v[i + H];
    v[i] = keep + __shfl_xor_sync(0xffffffffu, send, bit);
  }
}

// One pair (blockIdx.x) and group of ray pairs (blockIdx.y).  NO orbitals of J; NS = NP = ND = 0: the general
// evaluator (any radial order and knot grids), NO = kPbMaxOrb.
template <int NS, int NP, int ND, int NO>
__global__ void __launch_bounds__(kPbThreads, 4) k_psibeta(const __grid_constant__ GTabs orb,
                                                           const __grid_constant__ GTabs prj,
                                                           const __grid_constant__ GPb P) {
  constexpr int NV = 2 * kPbMaxOrb;  // (orbital, re / im) of one projector radial, padded
  // after the reduction over a ray's 16 lanes a lane holds 2 of the 32 sums of each radial; here their sums over
  // the warp's rays with the angular factors w_a Y_lm(e_a)
  __shared__ double tot[kPbGroup][5][2][kPbThreads];
  __shared__ double rk[kPbNr], sim[3 * kPbImages];  // radial nodes; tau_I - image of J
  __shared__ float rkf[kPbNr], simf[3 * kPbImages];
  const int p = P.order[blockIdx.x], I = P.pI[p], J = P.pJ[p];
  const GSpecies &SJ = orb.sp[P.species[J]];
  const GSpecies &SB = prj.sp[P.species[I]];
  const int noJ = SJ.norb, warp = threadIdx.x >> 5, lane = threadIdx.x & 31, kg = lane & (kPbSeg - 1);
  for (int k = threadIdx.x; k < kPbNr; k += kPbThreads) {
    rk[k] = SB.rcut * c_rad[k][0];
    rkf[k] = (float)rk[k];
  }
  const double tx = P.pos[3 * I], ty = P.pos[3 * I + 1], tz = P.pos[3 * I + 2];
  const int i0 = P.img_off[p], i1 = P.img_off[p + 1];
  const bool staged = i1 - i0 <= kPbImages;
  if (staged)
    for (int u = threadIdx.x; u < 3 * (i1 - i0); u += kPbThreads) {
      sim[u] = P.pos[3 * I + u % 3] - P.img[3 * i0 + u];
      simf[u] = (float)sim[u];
    }
  // float32 coordinates of at most rc_phi + 2 rc_beta, a few roundings each: r^2 is off by less than 1e-6 of their
  // square
  const double ext = SJ.rcut + 2.0 * SB.rcut;
  const float lim2 = (float)(SJ.rcut2 + 4e-6 * ext * ext);
  __syncthreads();
  const int np = kPbRayPairs / P.ngroups, rp0 = blockIdx.y * np;
  double *o = P.part + 2 * (blockIdx.y * P.nelems + P.poff[p]);
  int col = 0;  // first projector function of the pass
  for (int g0 = 0; g0 < SB.nrad; g0 += kPbGroup) {
    const int ng = min(kPbGroup, SB.nrad - g0);
    for (int i = 0; i < kPbGroup * 10; ++i) (&tot[0][0][0][0])[i * kPbThreads + threadIdx.x] = 0.0;
    for (int rp = rp0 + warp; rp < rp0 + np; rp += kPbWarps) {
      const int a = 2 * rp + (lane >> 4);
      const double ex = c_ang[a][0], ey = c_ang[a][1], ez = c_ang[a][2];
      const float exf = (float)ex, eyf = (float)ey, ezf = (float)ez;
      double acc[kPbGroup][NV];
#pragma unroll
      for (int g = 0; g < kPbGroup; ++g)
#pragma unroll
        for (int m = 0; m < NV; ++m) acc[g][m] = 0.0;
      const double2 *ph = P.phase + ((long long)(SB.rad0 + g0) * kPbRays + a) * kPbNr;
      for (int k = kg; k < (kPbNr + kPbSeg - 1) / kPbSeg * kPbSeg; k += kPbSeg) {
        const bool pt = k < kPbNr;
        const double r = pt ? rk[k] : 0.0;
        const float rf = pt ? rkf[k] : 0.f;
        double phi[NO];
#pragma unroll
        for (int m = 0; m < NO; ++m) phi[m] = 0.0;
        bool any = false;
        for (int q = i0; q < i1; ++q) {
          // screened in float32 for the whole patch: a point beyond lim2 (four times the bound on the float32
          // error of r^2 outside the support) is outside
          double ox, oy, oz;  // tau_I - image
          if (staged) {
            const float fx = fmaf(rf, exf, simf[3 * (q - i0)]), fy = fmaf(rf, eyf, simf[3 * (q - i0) + 1]),
                        fz = fmaf(rf, ezf, simf[3 * (q - i0) + 2]);
            if (!__any_sync(0xffffffffu, pt && fx * fx + fy * fy + fz * fz < lim2)) continue;
            ox = sim[3 * (q - i0)], oy = sim[3 * (q - i0) + 1], oz = sim[3 * (q - i0) + 2];
          } else {
            ox = tx - P.img[3 * q], oy = ty - P.img[3 * q + 1], oz = tz - P.img[3 * q + 2];
          }
          const double dx = fma(r, ex, ox), dy = fma(r, ey, oy), dz = fma(r, ez, oz);
          const double r2 = fma(dz, dz, fma(dy, dy, dx * dx));
          if (pt && r2 < SJ.rcut2) {
            any = true;
            if constexpr (NS + NP + ND > 0)
              orbitals64<NS, NP, ND>(orb, P.otab, SJ, dx, dy, dz, r2, phi);
            else
              add_orbitals<double, true, false>(orb, P.tab, P.species[J], dx, dy, dz, phi, nullptr);
          }
        }
        if (!__any_sync(0xffffffffu, any)) continue;
#pragma unroll
        for (int g = 0; g < kPbGroup; ++g) {
          if (g >= ng) break;
          const double2 w = pt ? __ldg(ph + (long long)g * kPbRays * kPbNr + k) : make_double2(0.0, 0.0);
#pragma unroll
          for (int m = 0; m < NO; ++m) {
            acc[g][2 * m] = fma(w.x, phi[m], acc[g][2 * m]);
            acc[g][2 * m + 1] = fma(w.y, phi[m], acc[g][2 * m + 1]);
          }
        }
      }
#pragma unroll
      for (int g = 0; g < kPbGroup; ++g) {
        if (g >= ng) break;
        halve<16>(acc[g], 8);
        halve<8>(acc[g], 4);
        halve<4>(acc[g], 2);
        halve<2>(acc[g], 1);
        double y[5], gy[5][3];
        const int l = prj.rad[SB.rad0 + g0 + g].l;
        ylm_unit<double>(l, ex, ey, ez, y, gy);
#pragma unroll
        for (int mm = 0; mm < 5; ++mm)
          if (mm < 2 * l + 1) {
            const double f = c_ang[a][3] * y[mm];
            double *t = &tot[g][mm][0][threadIdx.x];
            t[0] = fma(f, acc[g][0], t[0]);
            t[kPbThreads] = fma(f, acc[g][1], t[kPbThreads]);
          }
      }
    }
    // the halvings left sums 2 kg, 2 kg + 1 (orbital, re / im) in the lanes kg of either half
    __syncthreads();
    for (int g = 0; g < ng; ++g) {
      const int nm = 2 * prj.rad[SB.rad0 + g0 + g].l + 1;
      for (int u = threadIdx.x; u < 2 * nm * noJ; u += kPbThreads) {
        const int mm = u / (2 * noJ), e = u - mm * 2 * noJ;
        const double *t = &tot[g][mm][e & 1][e >> 1];
        double v = 0.0;
        for (int w = 0; w < 2 * kPbWarps; ++w) v += t[w * kPbSeg];
        o[2 * col * noJ + u] = v;  // (projector col + mm, orbital e / 2, re / im)
      }
      col += nm;
    }
    __syncthreads();
  }
}

// out = e^{-i A.tau_I} times the sum of the groups' parts.
__global__ void __launch_bounds__(128) k_pb_sum(const __grid_constant__ GPb P, double2 *__restrict__ out) {
  const int p = blockIdx.x, I = P.pI[p];
  const double2 *part = reinterpret_cast<const double2 *>(P.part);
  double s, c;
  sincos(-(P.A[0] * P.pos[3 * I] + P.A[1] * P.pos[3 * I + 1] + P.A[2] * P.pos[3 * I + 2]), &s, &c);
  for (long long e = P.poff[p] + threadIdx.x; e < P.poff[p + 1]; e += blockDim.x) {
    double re = 0.0, im = 0.0;
    for (int g = 0; g < P.ngroups; ++g) {
      const double2 v = part[g * P.nelems + e];
      re += v.x;
      im += v.y;
    }
    out[e] = make_double2(re * c - im * s, re * s + im * c);
  }
}

// Orbital shapes (s, p, d radials) with a compiled evaluator, and their orbitals.
#define GINT_PB_SHAPES(X) X(2, 2, 1, 13) X(2, 1, 0, 5) X(1, 1, 1, 9) X(1, 1, 0, 4) X(1, 0, 0, 1)

template <typename T>
void pfree(T *&p) {
  if (p) cudaFree(p);
  p = nullptr;
}

template <typename T>
int upload(T **dst, const std::vector<T> &src) {
  if (cudaMalloc(dst, std::max<size_t>(src.size(), 1) * sizeof(T)) != cudaSuccess) {
    cudaGetLastError();
    return GINT_ENOMEM;
  }
  if (!src.empty() && cudaMemcpy(*dst, src.data(), src.size() * sizeof(T), cudaMemcpyHostToDevice) != cudaSuccess)
    return GINT_ECUDA;
  return GINT_OK;
}

}  // namespace

void gint_pb_free(gint_handle *h) {
  pfree(h->pb_tab64);
  pfree(h->pb_I);
  pfree(h->pb_J);
  pfree(h->pb_off);
  pfree(h->pb_img_off);
  pfree(h->pb_img);
  pfree(h->pb_order);
  pfree(h->pb_phase);
  pfree(h->pb_part);
  h->pb_ready = false;
  h->pb_npairs = 0;
  h->pb_nelems = 0;
  h->pb_bytes = 0;
  h->pb_pairs_host.clear();
  h->pb_off_host.clear();
}

int gint_pb_set(gint_handle *h, int nspecies, const gint_species *proj) {
  const GGeom &g = h->geom;
  if (nspecies != g.nspecies || !proj) return GINT_EINVAL;
  for (int s = 0; s < nspecies; ++s)
    if (g.sp[s].norb > kPbMaxOrb) return GINT_EUNSUPPORTED;  // neighbour orbitals held in registers
  GTabs t{};
  std::vector<double2> tab;
  int r = 0;
  t.nspecies = nspecies;
  for (int s = 0; s < nspecies; ++s) {
    const gint_species &S = proj[s];
    if (S.nradial < 0 || (S.nradial > 0 && !S.radial)) return GINT_EINVAL;
    GSpecies &GS = t.sp[s];
    GS.nrad = S.nradial;
    GS.rad0 = r;
    for (int k = 0; k < S.nradial; ++k, ++r) {
      const gint_radial &R = S.radial[k];
      if (r >= GINT_MAX_RADIAL) return GINT_EINVAL;
      if (R.l < 0 || R.l > 2 || R.npts < 2 || !(R.dr > 0) || !(R.rc > 0) || !R.f || !R.df) return GINT_EINVAL;
      if (R.rc > (R.npts - 1) * R.dr * (1 + 1e-12)) return GINT_EINVAL;
      GRadial &GR = t.rad[r];
      GR.l = R.l;
      GR.npts = R.npts;
      GR.off = (int)tab.size();
      GR.dr = R.dr;
      GR.inv_dr = 1.0 / R.dr;
      GR.rc = R.rc;
      GR.rc2 = R.rc * R.rc;
      for (int i = 0; i < R.npts; ++i) tab.push_back(make_double2(R.f[i], R.df[i]));
      GS.norb += 2 * R.l + 1;
      GS.rcut = std::max(GS.rcut, R.rc);
    }
    GS.rcut2 = GS.rcut * GS.rcut;
  }
  t.nrad = r;
  // pairs (I, J): the images of J whose orbitals reach I's projector sphere
  const int na = g.natoms;
  std::vector<int> pI, pJ, img_off(1, 0);
  std::vector<long long> poff(1, 0);
  std::vector<double> img;
  for (int I = 0; I < na; ++I) {
    const GSpecies &SB = t.sp[h->species_host[I]];
    if (SB.nrad == 0) continue;
    for (int J = 0; J < na; ++J) {
      const GSpecies &SJ = g.sp[h->species_host[J]];
      const double reach = SB.rcut + SJ.rcut;
      double d0[3], u[3];
      for (int c = 0; c < 3; ++c) d0[c] = h->pos_host[3 * J + c] - h->pos_host[3 * I + c];
      for (int c = 0; c < 3; ++c) u[c] = d0[0] * g.inv[0 * 3 + c] + d0[1] * g.inv[1 * 3 + c] + d0[2] * g.inv[2 * 3 + c];
      int lo[3], hi[3];
      for (int c = 0; c < 3; ++c) {
        lo[c] = (int)std::ceil(-u[c] - reach * g.reach[c]);
        hi[c] = (int)std::floor(-u[c] + reach * g.reach[c]);
      }
      const size_t before = img.size();
      for (int n0 = lo[0]; n0 <= hi[0]; ++n0)
        for (int n1 = lo[1]; n1 <= hi[1]; ++n1)
          for (int n2 = lo[2]; n2 <= hi[2]; ++n2) {
            double d[3];
            for (int c = 0; c < 3; ++c) d[c] = d0[c] + n0 * g.cell[c] + n1 * g.cell[3 + c] + n2 * g.cell[6 + c];
            if (d[0] * d[0] + d[1] * d[1] + d[2] * d[2] < reach * reach)
              for (int c = 0; c < 3; ++c) img.push_back(h->pos_host[3 * I + c] + d[c]);
          }
      if (img.size() == before) continue;
      pI.push_back(I);
      pJ.push_back(J);
      img_off.push_back((int)(img.size() / 3));
      poff.push_back(poff.back() + (long long)SB.norb * SJ.norb);
    }
  }
  // quadrature: radial Gauss-Legendre on [0, 1]; angular product rule of degree 17
  std::vector<double> x, w;
  gauss_legendre(kPbNr, x, w);
  double rad[kPbNr][2];
  for (int k = 0; k < kPbNr; ++k) {
    rad[k][0] = 0.5 * (x[k] + 1.0);
    rad[k][1] = 0.5 * w[k];
  }
  gauss_legendre(kPbTheta, x, w);
  double ang[kPbRays][4];
  for (int i = 0; i < kPbTheta; ++i)
    for (int j = 0; j < kPbPhi; ++j) {
      const double ct = x[i], st = std::sqrt(1.0 - ct * ct), ph = 2.0 * kPi * j / kPbPhi;
      double *e = ang[i * kPbPhi + j];
      e[0] = st * std::cos(ph);
      e[1] = st * std::sin(ph);
      e[2] = ct;
      e[3] = w[i] * 2.0 * kPi / kPbPhi;
    }
  if (cudaMemcpyToSymbol(c_rad, rad, sizeof(rad)) != cudaSuccess ||
      cudaMemcpyToSymbol(c_ang, ang, sizeof(ang)) != cudaSuccess) {
    cudaGetLastError();
    return GINT_ECUDA;
  }
  // shapes without a compiled kernel take the general one
  std::vector<int> shape(g.nspecies, 0);
  for (int s = 0; s < g.nspecies; ++s) switch (h->tabs64.sp[s].shape) {
#define CASE_PB(ns, np, nd, no) case GINT_SHAPE(ns, np, nd):
      GINT_PB_SHAPES(CASE_PB)
#undef CASE_PB
      shape[s] = h->tabs64.sp[s].shape;
      break;
      default: break;
    }
  // pairs in launch order: by the shape of J
  std::vector<int> order(pI.size());
  for (size_t q = 0; q < order.size(); ++q) order[q] = (int)q;
  std::stable_sort(order.begin(), order.end(), [&](int x, int y) {
    return shape[h->species_host[pJ[x]]] < shape[h->species_host[pJ[y]]];
  });
  gint_pb_free(h);
  int rc;
  const int npair = (int)pI.size();
  // ray groups per pair (CTAs): enough CTAs for a few waves, no more (each group costs a reduction of its sums)
  h->pb_groups = npair < 4 * h->num_sms ? 9 : npair < 64 * h->num_sms ? 3 : 1;
  const size_t phase = (size_t)std::max(1, t.nrad) * kPbRays * kPbNr, part = (size_t)h->pb_groups * poff.back();
  if ((rc = upload(&h->pb_tab64, tab)) || (rc = upload(&h->pb_I, pI)) || (rc = upload(&h->pb_J, pJ)) ||
      (rc = upload(&h->pb_off, poff)) || (rc = upload(&h->pb_img_off, img_off)) || (rc = upload(&h->pb_img, img)) ||
      (rc = upload(&h->pb_order, order))) {
    gint_pb_free(h);
    return rc;
  }
  if (cudaMalloc(&h->pb_phase, phase * sizeof(double2)) != cudaSuccess ||
      cudaMalloc(&h->pb_part, std::max<size_t>(part, 1) * sizeof(double2)) != cudaSuccess) {
    cudaGetLastError();
    gint_pb_free(h);
    return GINT_ENOMEM;
  }
  h->pb_tabs = t;
  h->pb_shape.clear();
  h->pb_first.clear();
  for (int q = 0; q < npair; ++q) {
    const int sh = shape[h->species_host[pJ[order[q]]]];
    if (q == 0 || sh != h->pb_shape.back()) {
      h->pb_shape.push_back(sh);
      h->pb_first.push_back(q);
    }
  }
  h->pb_first.push_back(npair);
  h->pb_npairs = npair;
  h->pb_nelems = poff.back();
  h->pb_pairs_host.resize(2 * pI.size());
  for (size_t q = 0; q < pI.size(); ++q) {
    h->pb_pairs_host[2 * q] = pI[q];
    h->pb_pairs_host[2 * q + 1] = pJ[q];
  }
  h->pb_off_host = poff;
  h->pb_bytes = (long long)(tab.size() * sizeof(double2) + (3 * pI.size() + img_off.size()) * sizeof(int) +
                            poff.size() * sizeof(long long) + img.size() * sizeof(double) +
                            (phase + part) * sizeof(double2));
  h->pb_ready = true;
  return GINT_OK;
}

int gint_pb_run(gint_handle *h, const double A[3], double *out, cudaStream_t st) {
  if (!h->pb_ready) return GINT_EINVAL;
  if (h->pb_npairs == 0) return GINT_OK;
  GPb P{};
  for (int c = 0; c < 3; ++c) P.A[c] = A[c];
  P.pI = h->pb_I;
  P.pJ = h->pb_J;
  P.poff = h->pb_off;
  P.img_off = h->pb_img_off;
  P.img = h->pb_img;
  P.pos = h->pos_dev;
  P.species = h->species_dev;
  P.tab = h->tab64;
  P.ptab = h->pb_tab64;
  P.otab = h->otab64;
  P.phase = h->pb_phase;
  P.part = reinterpret_cast<double *>(h->pb_part);
  P.nelems = h->pb_nelems;
  P.ngroups = h->pb_groups;
  if (h->pb_tabs.nrad == 0) return GINT_OK;
  k_pb_phase<<<dim3((kPbRays * kPbNr + 255) / 256, (unsigned)h->pb_tabs.nrad), 256, 0, st>>>(h->pb_tabs, P);
  for (size_t q = 0; q < h->pb_shape.size(); ++q) {
    P.order = h->pb_order + h->pb_first[q];
    const dim3 grid((unsigned)(h->pb_first[q + 1] - h->pb_first[q]), (unsigned)h->pb_groups);
    switch (h->pb_shape[q]) {
#define CASE_PB(ns, np, nd, no)                                                                        \
  case GINT_SHAPE(ns, np, nd): k_psibeta<ns, np, nd, no><<<grid, kPbThreads, 0, st>>>(h->tabs64, h->pb_tabs, P); break;
      GINT_PB_SHAPES(CASE_PB)
#undef CASE_PB
      default: k_psibeta<0, 0, 0, kPbMaxOrb><<<grid, kPbThreads, 0, st>>>(h->tabs64, h->pb_tabs, P);
    }
  }
  k_pb_sum<<<(unsigned)h->pb_npairs, 128, 0, st>>>(P, reinterpret_cast<double2 *>(out));
  return cudaGetLastError() == cudaSuccess ? GINT_OK : GINT_ECUDA;
}
