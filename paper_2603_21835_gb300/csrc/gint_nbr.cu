// gint_nbr.cu -- device builder of the grid-brick -> atom neighbour lists (the paper's
// BigGrid neighbour relation managed by GintInfo, Sec. 3.3.1 and Fig. 2).
//
// The grid is cut into bricks of 4 x 4 x 8 points.  An (atom, lattice image) entry belongs
// to a brick when at least one of the brick's grid points lies strictly inside the atom's
// support sphere (exact per-point test, float64).  Entries of one atom form a "slot": its
// orbitals occupy one set of columns in the brick (periodic images folded, Gamma point).  In the
// unfolded layout (the per-R twin of a folded handle) every entry is a slot of its own, in the same
// order (atom, then lattice vector (n1, n2, n3) ascending).
// Each brick also gets an n_a x n_a table of global pair indices for its slots.
//
// Float64 runs at 2 operations per clock and SM here (a warp-wide one occupies the pipe for 16 clocks), so the
// kernels keep it for what needs it: atoms are screened in float32 fractional coordinates and the few near a
// brick compacted before their image ranges are formed in float64; a brick's points are float32 offsets from its
// centre; and the exact float64 test runs for points in a thin shell around a support sphere only.  The counting
// pass leaves each brick's entries in a list, from which the filling pass writes its arrays.  64-atom Si, 96^3
// (6,912 bricks): count 312 -> 48 us, fill 477 -> 11 us, work count 192 -> 50 us, scan 40 -> 16 us.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>

#include "gint_handle.cuh"

namespace {

constexpr int kListCap = (int)(kNbrListBytes / sizeof(int4));  // entries of a brick kept by the counting pass; longer bricks are visited again

// Geometry of a full brick, formed on the host.
struct GBrickGeo {
  double step[3][3];   // Cartesian step of one grid index (cell row / n)
  double mid[3];       // brick centre relative to its first point
  double rad;          // bounding radius (bricks cut off at the grid's upper faces use it too)
  float stepf[3][3];
  float flim[GINT_MAX_SPECIES][3];    // float32 screen of |fractional distance| per species and axis
  float in2[GINT_MAX_SPECIES], out2[GINT_MAX_SPECIES];  // shell around rc^2 (see warp_image_hits)
};

__device__ __forceinline__ void brick_box(const GGeom &g, long long b, int lo[3], int hi[3]) {
  const unsigned ub = (unsigned)b, nbk = (unsigned)g.nbk, q = ub / nbk;  // brick indices fit 32 bits
  const int bk = (int)(ub - q * nbk), bj = (int)(q % (unsigned)g.nbj), bi = (int)(q / (unsigned)g.nbj);
  lo[0] = bi * GINT_BI; hi[0] = min(lo[0] + GINT_BI, g.n1);
  lo[1] = bj * GINT_BJ; hi[1] = min(lo[1] + GINT_BJ, g.n2);
  lo[2] = bk * GINT_BK; hi[2] = min(lo[2] + GINT_BK, g.n3);
}

// Centre of a brick (of the full brick, also where the grid cuts it off).
__device__ __forceinline__ double brick_mid(const GBrickGeo &G, const int lo[3], int d) {
  return G.mid[d] + (lo[0] * G.step[0][d] + lo[1] * G.step[1][d] + lo[2] * G.step[2][d]);
}

// Image range of atom I around a brick sphere (centre c, radius rad); fixed arithmetic so
// that the counting and filling passes take identical decisions.
__device__ __noinline__ void image_range(const GGeom &g, const double *pos, int I, double rc, const double c[3],
                                         double rad, int nlo[3], int nhi[3]) {
  double d0[3], u[3];
  for (int d = 0; d < 3; ++d) d0[d] = c[d] - pos[3 * I + d];
  for (int d = 0; d < 3; ++d) u[d] = d0[0] * g.inv[0 * 3 + d] + d0[1] * g.inv[1 * 3 + d] + d0[2] * g.inv[2 * 3 + d];
  for (int d = 0; d < 3; ++d) {
    double reach = (rc + rad) * g.reach[d];
    nlo[d] = (int)ceil(u[d] - reach);
    nhi[d] = (int)floor(u[d] + reach);
  }
}

// A brick's grid points relative to its centre as float32, four per lane: point q = lane + 32 k, k = 0..3, is
// (q / 32, q / 8 mod 4, q mod 8) of the 4 x 4 x 8 box; in: whether the grid has it.
struct BrickPts {
  float x[4], y[4], z[4];
  bool in[4];
};
__device__ __forceinline__ void brick_points(const GBrickGeo &G, const int lo[3], const int hi[3], int lane, BrickPts &P) {
  const int dj = (lane >> 3) & 3, dk = lane & 7;
  const float fj = (float)dj - 0.5f * (GINT_BJ - 1), fk = (float)dk - 0.5f * (GINT_BK - 1);
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const float fi = (float)k - 0.5f * (GINT_BI - 1);
    P.x[k] = fi * G.stepf[0][0] + fj * G.stepf[1][0] + fk * G.stepf[2][0];
    P.y[k] = fi * G.stepf[0][1] + fj * G.stepf[1][1] + fk * G.stepf[2][1];
    P.z[k] = fi * G.stepf[0][2] + fj * G.stepf[1][2] + fk * G.stepf[2][2];
    P.in[k] = lo[0] + k < hi[0] && lo[1] + dj < hi[1] && lo[2] + dk < hi[2];
  }
}

// The float64 test: does grid point (i, j, k) lie strictly inside the sphere of squared radius rc2 around T?  Not
// inlined: the compiler would hoist the point's float64 divisions out of the loops that rarely need it.
__device__ __noinline__ bool point_inside(const GGeom &g, int i, int j, int k, const double *T, double rc2) {
  double p[3];
  grid_point(g, i, j, k, p);
  return (p[0] - T[0]) * (p[0] - T[0]) + (p[1] - T[1]) * (p[1] - T[1]) + (p[2] - T[2]) * (p[2] - T[2]) < rc2;
}

// Does the image at T of an atom with support radius rc cover any grid point of the brick (some point strictly
// inside the sphere, float64)?  All 32 lanes take part, each testing its four points; tx, ty, tz: T - c in float32,
// in2 / out2 the species' shell, src the lane that holds T.  A float32 squared distance relative to the brick
// centre decides every point outside a shell |r^2 - rc^2| < m around the sphere; a point inside the shell is
// decided by the float64 test itself (same expression as a per-point loop), so the answer equals the float64
// one.  Bound used for m: with |p - c| <= rad and |T - c| < rc + rad (the caller's bounding-sphere test), T - c is
// off by 2^-24 (rc + rad), a point's offset by five roundings of terms below rad, 3e-7 rad, and their difference
// by one more rounding, so the float32 r^2 is off by less than 2.5e-7 (2 rc + 4 rad)^2 + 2.4e-7 r^2; m is sixteen
// times the first term plus four times the second.  Warp-uniform result.
__device__ bool warp_image_hits(const GGeom &g, const BrickPts &P, float tx, float ty, float tz, float in2, float out2,
                                const double T[3], double rc, int src, const int lo[3], int lane) {
  bool hit = false, shell = false;
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const float dx = P.x[k] - tx, dy = P.y[k] - ty, dz = P.z[k] - tz;
    const float r2 = dx * dx + dy * dy + dz * dz;
    hit |= P.in[k] && r2 < in2;
    shell |= P.in[k] && r2 >= in2 && r2 < out2;
  }
  if (__any_sync(0xffffffffu, hit)) return true;
  if (!__any_sync(0xffffffffu, shell)) return false;
  double Ts[3];
  for (int d = 0; d < 3; ++d) Ts[d] = __shfl_sync(0xffffffffu, T[d], src);
  const double rcs = __shfl_sync(0xffffffffu, rc, src), rc2 = rcs * rcs;
  for (int k = 0; k < 4; ++k) {
    const float dx = P.x[k] - tx, dy = P.y[k] - ty, dz = P.z[k] - tz;
    const float r2 = dx * dx + dy * dy + dz * dz;
    if (P.in[k] && r2 >= in2 && r2 < out2)
      hit |= point_inside(g, lo[0] + k, lo[1] + ((lane >> 3) & 3), lo[2] + (lane & 7), Ts, rc2);
  }
  return __any_sync(0xffffffffu, hit);
}

// The lattice images near brick b of the warp's atoms (I: the lane's atom, -1 for none), one candidate at a
// time: every image in the atom's image range whose bounding-sphere test passes (centre distance below rc + rad)
// is tested against the brick's points by the whole warp, in lane order and, within a lane, in the order
// n0, n1, n2 ascending.  visit(src, T, n, hit) runs in every lane (src: the lane whose atom the image belongs to,
// whose T and n are that image's).
template <typename Visit>
__device__ void warp_atom_images(const GGeom &g, const GBrickGeo &G, const double *pos, const int *species, int I,
                                 int lane, const int lo[3], const double c[3], const BrickPts &P, Visit visit) {
  const bool va = I >= 0;
  const int sp = va ? species[I] : 0;
  const double rc = va ? g.sp[sp].rcut : 0.0;
  const float in2 = G.in2[sp], out2 = G.out2[sp];
  int nlo[3] = {0, 0, 0}, nhi[3] = {-1, -1, -1};
  if (va) image_range(g, pos, I, rc, c, G.rad, nlo, nhi);
  const int s1 = max(0, nhi[1] - nlo[1] + 1), s2 = max(0, nhi[2] - nlo[2] + 1);
  const int nimg = max(0, nhi[0] - nlo[0] + 1) * s1 * s2;
  const double lim2 = (rc + G.rad) * (rc + G.rad);
  int k = 0, n[3] = {0, 0, 0};
  double T[3] = {0.0, 0.0, 0.0};
  float tx = 0.f, ty = 0.f, tz = 0.f;
  auto next = [&]() -> bool {
    while (k < nimg) {
      const int i0 = k / (s1 * s2), r = k - i0 * s1 * s2, i1 = r / s2, i2 = r - i1 * s2;
      ++k;
      n[0] = nlo[0] + i0;
      n[1] = nlo[1] + i1;
      n[2] = nlo[2] + i2;
      for (int d = 0; d < 3; ++d) T[d] = pos[3 * I + d] + n[0] * g.cell[d] + n[1] * g.cell[3 + d] + n[2] * g.cell[6 + d];
      const double D2 = (c[0] - T[0]) * (c[0] - T[0]) + (c[1] - T[1]) * (c[1] - T[1]) + (c[2] - T[2]) * (c[2] - T[2]);
      if (!(D2 >= lim2)) {
        tx = (float)(T[0] - c[0]);
        ty = (float)(T[1] - c[1]);
        tz = (float)(T[2] - c[2]);
        return true;
      }
    }
    return false;
  };
  bool cand = next();
  for (;;) {
    const unsigned m = __ballot_sync(0xffffffffu, cand);
    if (!m) break;
    const int src = __ffs(m) - 1;
    const bool hit = warp_image_hits(g, P, __shfl_sync(0xffffffffu, tx, src), __shfl_sync(0xffffffffu, ty, src),
                                     __shfl_sync(0xffffffffu, tz, src), __shfl_sync(0xffffffffu, in2, src),
                                     __shfl_sync(0xffffffffu, out2, src), T, rc, src, lo, lane);
    visit(src, T, n, hit);
    if (lane == src) cand = next();
  }
}

// The atoms that may have an image near the brick, 32 at a time in ascending order: the float32 fractional
// distance to the nearest lattice translate is within the species' limit on every axis (limits carry 1e-4 of
// slack, far above the float32 errors).  batch(I) runs in every lane (-1: none).  buf: 64 ints of the warp's own.
template <typename Batch>
__device__ void near_atoms(const GGeom &g, const GBrickGeo &G, const float *__restrict__ frac,
                           const int *__restrict__ species, const double c[3], int lane, int *buf, Batch batch) {
  float u[3];
  for (int d = 0; d < 3; ++d) u[d] = (float)(c[0] * g.inv[0 * 3 + d] + c[1] * g.inv[1 * 3 + d] + c[2] * g.inv[2 * 3 + d]);
  int held = 0;
  for (int a0 = 0; a0 < g.natoms; a0 += 32) {
    const int I = a0 + lane;
    bool near = false;
    if (I < g.natoms) {
      const int sp = species[I];
      near = true;
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        const float x = u[d] - frac[3 * I + d];
        near &= fabsf(x - rintf(x)) <= G.flim[sp][d];
      }
    }
    const unsigned m = __ballot_sync(0xffffffffu, near);
    if (near) buf[held + __popc(m & ((1u << lane) - 1u))] = I;
    held += __popc(m);
    __syncwarp();
    if (held >= 32) {
      batch(buf[lane]);
      const int rest = lane + 32 < held ? buf[lane + 32] : 0;
      __syncwarp();
      buf[lane] = rest;
      held -= 32;
      __syncwarp();
    }
  }
  if (held > 0) batch(lane < held ? buf[lane] : -1);
  __syncwarp();
}

// Fractional coordinates as float32 (reduced to [0, 1) first, so that their absolute error is 2^-24).
__global__ void k_frac(GGeom g, const double *__restrict__ pos, float *__restrict__ frac) {
  const int I = blockIdx.x * blockDim.x + threadIdx.x;
  if (I >= g.natoms) return;
  for (int d = 0; d < 3; ++d) {
    const double u = pos[3 * I] * g.inv[d] + pos[3 * I + 1] * g.inv[3 + d] + pos[3 * I + 2] * g.inv[6 + d];
    frac[3 * I + d] = (float)(u - floor(u));
  }
}

__device__ __forceinline__ int warp_excl_scan(int v, int lane) {
  int x = v;
  for (int o = 1; o < 32; o <<= 1) {
    int y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  return x - v;
}

// One warp per brick: number of slots, entries and orbitals, and the brick's first kListCap entries (atom, image) in
// order.
constexpr int kNbrWarps = 4;
__global__ void __launch_bounds__(32 * kNbrWarps) k_brick_count(const __grid_constant__ GGeom g,
                                                               const __grid_constant__ GBrickGeo G, const double *pos,
                                                               const float *frac, const int *species, int unfold, int *n_at,
                                                               int *n_ent, int *n_orb, int4 *list) {
  __shared__ int buf[kNbrWarps][64];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const long long b = (long long)blockIdx.x * kNbrWarps + w;
  if (b >= g.nbricks) return;
  int lo[3], hi[3];
  brick_box(g, b, lo, hi);
  double c[3];
  for (int d = 0; d < 3; ++d) c[d] = brick_mid(G, lo, d);
  BrickPts P;
  brick_points(G, lo, hi, lane, P);
  int at = 0, ent = 0, orb = 0, last = -1;  // warp-uniform; last: the atom of the last entry
  near_atoms(g, G, frac, species, c, lane, buf[w], [&](int I) {
    warp_atom_images(g, G, pos, species, I, lane, lo, c, P, [&](int src, const double *, const int *n, bool hit) {
      if (!hit) return;
      if (lane == src && ent < kListCap) list[b * kListCap + ent] = make_int4(I, n[0], n[1], n[2]);
      ++ent;
      const int J = __shfl_sync(0xffffffffu, I, src);
      if (unfold || J != last) {
        ++at;
        orb += g.sp[species[J]].norb;
        last = J;
      }
    });
  });
  if (lane == 0) {
    n_at[b] = at;
    n_ent[b] = ent;
    n_orb[b] = orb;
  }
}

__device__ __forceinline__ long long warp_incl_scan_ll(long long v, int lane) {
  for (int o = 1; o < 32; o <<= 1) {
    const long long y = __shfl_up_sync(0xffffffffu, v, o);
    if (lane >= o) v += y;
  }
  return v;
}

// Single-CTA exclusive scans of the per-brick counts; also the totals and maxima.
//   out[0] = slots, out[1] = entries, out[2] = pair-table size, out[3] = max orbitals,
//   out[4] = max atoms, out[5] = executed pair work sum_b 128 norb_b^2, out[6] = max entries
// Four consecutive bricks per thread and round (coalesced 16-byte loads), scanned by warp shuffles.
__global__ void __launch_bounds__(1024) k_brick_scan(long long nb, const int *n_at, const int *n_ent, const int *n_orb,
                                                     long long *at_off, long long *ent_off, long long *pair_off,
                                                     long long *out) {
  __shared__ long long ws[3][32], wx_s[32];
  __shared__ int wm[3][32];
  const int t = threadIdx.x, lane = t & 31, w = t >> 5;
  long long carry[3] = {0, 0, 0}, wx = 0;
  int mo = 0, ma = 0, me = 0;
  for (long long b0 = 0; b0 < nb; b0 += 4096) {
    const long long b = b0 + 4 * t;
    int a[4], e[4], o[4];
    if (b + 4 <= nb) {
      const int4 x = *reinterpret_cast<const int4 *>(n_at + b), y = *reinterpret_cast<const int4 *>(n_ent + b),
                 z = *reinterpret_cast<const int4 *>(n_orb + b);
      a[0] = x.x, a[1] = x.y, a[2] = x.z, a[3] = x.w;
      e[0] = y.x, e[1] = y.y, e[2] = y.z, e[3] = y.w;
      o[0] = z.x, o[1] = z.y, o[2] = z.z, o[3] = z.w;
    } else {
      for (int k = 0; k < 4; ++k) {
        const bool in = b + k < nb;
        a[k] = in ? n_at[b + k] : 0;
        e[k] = in ? n_ent[b + k] : 0;
        o[k] = in ? n_orb[b + k] : 0;
      }
    }
    long long s[3] = {0, 0, 0};
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      s[0] += a[k];
      s[1] += e[k];
      s[2] += (long long)a[k] * a[k];
      wx += (long long)o[k] * o[k];
      mo = max(mo, o[k]);
      ma = max(ma, a[k]);
      me = max(me, e[k]);
    }
    long long inc[3];
    for (int q = 0; q < 3; ++q) {
      inc[q] = warp_incl_scan_ll(s[q], lane);
      if (lane == 31) ws[q][w] = inc[q];
    }
    __syncthreads();
    if (w < 3) ws[w][lane] = warp_incl_scan_ll(ws[w][lane], lane);
    __syncthreads();
    long long x[3], tot[3];
    for (int q = 0; q < 3; ++q) {
      x[q] = carry[q] + (w > 0 ? ws[q][w - 1] : 0) + inc[q] - s[q];
      tot[q] = ws[q][31];
      carry[q] += tot[q];
    }
#pragma unroll
    for (int k = 0; k < 4; ++k)
      if (b + k < nb) {
        at_off[b + k] = x[0];
        ent_off[b + k] = x[1];
        pair_off[b + k] = x[2];
        x[0] += a[k];
        x[1] += e[k];
        x[2] += (long long)a[k] * a[k];
      }
    __syncthreads();  // ws is rewritten in the next round
  }
  for (int q = 16; q > 0; q >>= 1) {
    wx += __shfl_xor_sync(0xffffffffu, wx, q);
    mo = max(mo, __shfl_xor_sync(0xffffffffu, mo, q));
    ma = max(ma, __shfl_xor_sync(0xffffffffu, ma, q));
    me = max(me, __shfl_xor_sync(0xffffffffu, me, q));
  }
  if (lane == 0) {
    wx_s[w] = wx;
    wm[0][w] = mo;
    wm[1][w] = ma;
    wm[2][w] = me;
  }
  __syncthreads();
  if (t == 0) {
    for (int i = 1; i < 32; ++i) {
      wx += wx_s[i];
      mo = max(mo, wm[0][i]);
      ma = max(ma, wm[1][i]);
      me = max(me, wm[2][i]);
    }
    out[0] = carry[0]; out[1] = carry[1]; out[2] = carry[2]; out[3] = mo; out[4] = ma; out[5] = wx * GINT_BPTS; out[6] = me;
    at_off[nb] = carry[0]; ent_off[nb] = carry[1]; pair_off[nb] = carry[2];
  }
}

// One warp per brick: writes slots (atom, column, first entry) and entries (image shifts), 32 entries at a time,
// from the counting pass's list; a brick with more entries than that holds visits its images again, in the
// same order.
__global__ void __launch_bounds__(32 * kNbrWarps)
    k_brick_fill(const __grid_constant__ GGeom g, const __grid_constant__ GBrickGeo G, const double *pos, const float *frac,
                 const int *species, int unfold, const long long *at_off, const long long *ent_off, const int4 *list,
                 int *s_atom, int *s_col, long long *s_ent, double *e_shift, unsigned *err) {
  __shared__ int buf[kNbrWarps][64];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const long long b = (long long)blockIdx.x * kNbrWarps + w;
  if (b >= g.nbricks) return;
  long long slot = at_off[b], ent = ent_off[b];
  const long long slot_end = at_off[b + 1], ent_end = ent_off[b + 1];
  int col = 0, last = -1;
  const int ne = (int)(ent_end - ent);
  if (ne <= kListCap) {
    for (int e0 = 0; e0 < ne; e0 += 32) {
      const int k = e0 + lane;
      const int4 x = k < ne ? list[b * kListCap + k] : make_int4(-1, 0, 0, 0);
      int prev = __shfl_up_sync(0xffffffffu, x.x, 1);
      if (lane == 0) prev = last;
      const bool first = k < ne && (unfold || x.x != prev);
      const int no = first ? g.sp[species[x.x]].norb : 0;
      const int sl = warp_excl_scan(first, lane), cl = warp_excl_scan(no, lane);
      if (first && slot + sl < slot_end) {
        s_atom[slot + sl] = x.x;
        s_col[slot + sl] = col + cl;
        s_ent[slot + sl] = ent + k;
      }
      if (k < ne)
        for (int d = 0; d < 3; ++d)
          e_shift[3 * (ent + k) + d] = pos[3 * x.x + d] + x.y * g.cell[d] + x.z * g.cell[3 + d] + x.w * g.cell[6 + d];
      slot += __shfl_sync(0xffffffffu, sl + (int)first, 31);
      col += __shfl_sync(0xffffffffu, cl + no, 31);
      last = __shfl_sync(0xffffffffu, x.x, 31);
    }
    if (lane == 0 && slot != slot_end) atomicOr(err, GINT_ERRBIT_INDEX);
    return;
  }
  int lo[3], hi[3];
  brick_box(g, b, lo, hi);
  double c[3];
  for (int d = 0; d < 3; ++d) c[d] = brick_mid(G, lo, d);
  BrickPts P;
  brick_points(G, lo, hi, lane, P);
  near_atoms(g, G, frac, species, c, lane, buf[w], [&](int I) {
    warp_atom_images(g, G, pos, species, I, lane, lo, c, P, [&](int src, const double *T, const int *, bool hit) {
      if (!hit) return;
      const int J = __shfl_sync(0xffffffffu, I, src);
      if (unfold || J != last) {
        if (lane == src && slot < slot_end) {
          s_atom[slot] = J;
          s_col[slot] = col;
          s_ent[slot] = ent;
        }
        ++slot;
        col += g.sp[species[J]].norb;
        last = J;
      }
      if (lane == src && ent < ent_end)
        for (int d = 0; d < 3; ++d) e_shift[3 * ent + d] = T[d];
      ++ent;
    });
  });
  if (lane == 0 && (slot != slot_end || ent != ent_end)) atomicOr(err, GINT_ERRBIT_INDEX);
}

// Minimum distance over lattice images between atoms I and J.
__device__ double min_image_dist(const GGeom &g, const double *pos, int I, int J, double limit) {
  double d0[3], u[3];
  for (int d = 0; d < 3; ++d) d0[d] = pos[3 * J + d] - pos[3 * I + d];
  for (int d = 0; d < 3; ++d) u[d] = d0[0] * g.inv[0 * 3 + d] + d0[1] * g.inv[1 * 3 + d] + d0[2] * g.inv[2 * 3 + d];
  double best = 1e300;
  int nlo[3], nhi[3];
  for (int d = 0; d < 3; ++d) {
    nlo[d] = (int)ceil(-u[d] - limit * g.reach[d]);
    nhi[d] = (int)floor(-u[d] + limit * g.reach[d]);
  }
  for (int n0 = nlo[0]; n0 <= nhi[0]; ++n0)
    for (int n1 = nlo[1]; n1 <= nhi[1]; ++n1)
      for (int n2 = nlo[2]; n2 <= nhi[2]; ++n2) {
        double x[3];
        for (int d = 0; d < 3; ++d) x[d] = d0[d] + n0 * g.cell[d] + n1 * g.cell[3 + d] + n2 * g.cell[6 + d];
        best = fmin(best, sqrt(x[0] * x[0] + x[1] * x[1] + x[2] * x[2]));
      }
  return best;
}

// One warp per brick: pair table of its slots; flags pairs that overlap but have no block.
__global__ void k_brick_pairs(GGeom g, const double *pos, const int *species, const long long *at_off,
                              const int *s_atom, const long long *bp_off, const int *pair_row, const int *pair_col,
                              int *b_pair, unsigned *err) {
  const int lane = threadIdx.x & 31;
  const long long b = (long long)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  if (b >= g.nbricks) return;
  const long long s0 = at_off[b];
  const int na = (int)(at_off[b + 1] - s0);
  for (int e = lane; e < na * na; e += 32) {
    int I = s_atom[s0 + e / na], J = s_atom[s0 + e % na];
    int lo = pair_row[I], hi = pair_row[I + 1] - 1, found = -1;
    while (lo <= hi) {
      int mid = (lo + hi) >> 1;
      int v = pair_col[mid];
      if (v == J) { found = mid; break; }
      if (v < J) lo = mid + 1; else hi = mid - 1;
    }
    if (found < 0) {
      double lim = g.sp[species[I]].rcut + g.sp[species[J]].rcut;
      if (min_image_dist(g, pos, I, J, lim) < lim) atomicOr(err, GINT_ERRBIT_SKIN);
    }
    b_pair[bp_off[b] + e] = found;
  }
}

// Exact algorithmic work: W = sum_g n_g^2 with n_g the orbitals covering point g.  One thread per point of a brick,
// a few CTAs per SM walking the bricks (one atomic per CTA: one per brick, all on one address, took most of the
// kernel's time).  The brick's entries and the slots' screening bounds (at most kCwE
// entries and kCwS slots; larger bricks take the plain float64 loop) are staged in shared memory,
// the entries as float32 offsets from the brick centre, and each (point, entry)
// distance is screened in float32 as in warp_image_hits, the float64 test deciding points in the
// thin shell around the sphere: the same coverage, so the same W, as the per-entry float64 loop.
constexpr int kCwE = 256, kCwS = 64;
__global__ void __launch_bounds__(GINT_BPTS) k_count_work(const __grid_constant__ GGeom g, const __grid_constant__ GBrickGeo G,
                                                         const long long *at_off, const int *s_atom, const long long *s_ent,
                                                         const double *e_shift, const int *species, double *W) {
  const int p = threadIdx.x;
  __shared__ float ex[kCwE], ey[kCwE], ez[kCwE], sin2[kCwS], sout2[kCwS];
  __shared__ int se[kCwS + 1], sno[kCwS];
  __shared__ double sc[3];
  long long acc = 0;
  for (long long b = blockIdx.x; b < g.nbricks; b += gridDim.x) {
    int lo[3], hi[3];
    brick_box(g, b, lo, hi);
    if (p < 3) sc[p] = G.mid[p] + (lo[0] * G.step[0][p] + lo[1] * G.step[1][p] + lo[2] * G.step[2][p]);
    const long long s0 = at_off[b], s1 = at_off[b + 1];
    const long long E0 = s1 > s0 ? s_ent[s0] : 0, E1 = s1 > s0 ? s_ent[s1] : 0;
    const int ns = (int)(s1 - s0);
    const bool staged = E1 - E0 <= kCwE && ns <= kCwS;
    __syncthreads();
    if (staged) {
      for (int e = p; e < (int)(E1 - E0); e += GINT_BPTS) {
        ex[e] = (float)(e_shift[3 * (E0 + e)] - sc[0]);
        ey[e] = (float)(e_shift[3 * (E0 + e) + 1] - sc[1]);
        ez[e] = (float)(e_shift[3 * (E0 + e) + 2] - sc[2]);
      }
      for (int s = p; s < ns; s += GINT_BPTS) {
        const int sp = species[s_atom[s0 + s]];
        sin2[s] = G.in2[sp];
        sout2[s] = G.out2[sp];
        sno[s] = g.sp[sp].norb;
        se[s] = (int)(s_ent[s0 + s] - E0);
      }
      if (p == 0) se[ns] = (int)(E1 - E0);
    }
    __syncthreads();
    const int di = p >> 5, dj = (p >> 3) & 3, dk = p & 7;  // as brick_point
    const int i = lo[0] + di, j = lo[1] + dj, k = lo[2] + dk;
    int n = 0;
    if (i < hi[0] && j < hi[1] && k < hi[2]) {
      auto inside = [&](long long e, double rc2) { return point_inside(g, i, j, k, e_shift + 3 * e, rc2); };
      if (staged) {
        const float fi = (float)di - 0.5f * (GINT_BI - 1), fj = (float)dj - 0.5f * (GINT_BJ - 1), fk = (float)dk - 0.5f * (GINT_BK - 1);
        const float px = fi * G.stepf[0][0] + fj * G.stepf[1][0] + fk * G.stepf[2][0];
        const float py = fi * G.stepf[0][1] + fj * G.stepf[1][1] + fk * G.stepf[2][1];
        const float pz = fi * G.stepf[0][2] + fj * G.stepf[1][2] + fk * G.stepf[2][2];
        for (int s = 0; s < ns; ++s) {
          const float in2 = sin2[s], out2 = sout2[s];
          bool cov = false;
          for (int e = se[s]; e < se[s + 1] && !cov; ++e) {
            const float dx = px - ex[e], dy = py - ey[e], dz = pz - ez[e];
            const float r2 = dx * dx + dy * dy + dz * dz;
            if (r2 < in2)
              cov = true;
            else if (r2 < out2)
              cov = inside(E0 + e, g.sp[species[s_atom[s0 + s]]].rcut2);
          }
          if (cov) n += sno[s];
        }
      } else {
        for (long long s = s0; s < s1; ++s) {
          const GSpecies &S = g.sp[species[s_atom[s]]];
          bool cov = false;
          for (long long e = s_ent[s]; e < s_ent[s + 1] && !cov; ++e) cov = inside(e, S.rcut2);
          if (cov) n += S.norb;
        }
      }
    }
    acc += n * n;
    __syncthreads();  // the staged arrays are rewritten for the next brick
  }
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
  __shared__ long long red[GINT_BPTS / 32];
  if ((p & 31) == 0) red[p >> 5] = acc;
  __syncthreads();
  if (p == 0) {
    long long t = 0;
    for (int w = 0; w < GINT_BPTS / 32; ++w) t += red[w];
    if (t) atomicAdd(W, (double)t);  // integers below 2^53: exact in any order
  }
}

GBrickGeo brick_geo(const GGeom &g) {
  GBrickGeo G{};
  const int n[3] = {g.n1, g.n2, g.n3}, e[3] = {GINT_BI, GINT_BJ, GINT_BK};
  for (int a = 0; a < 3; ++a)
    for (int d = 0; d < 3; ++d) {
      G.step[a][d] = g.cell[3 * a + d] / n[a];
      G.stepf[a][d] = (float)G.step[a][d];
      G.mid[d] += 0.5 * (e[a] - 1) * G.step[a][d];
    }
  // the farthest point of a parallelepiped lattice from its centre is a corner
  for (int corner = 0; corner < 4; ++corner) {
    double r2 = 0;
    for (int d = 0; d < 3; ++d) {
      const double x = 0.5 * ((e[0] - 1) * G.step[0][d] + ((corner & 1) ? 1 : -1) * (e[1] - 1) * G.step[1][d] +
                              ((corner & 2) ? 1 : -1) * (e[2] - 1) * G.step[2][d]);
      r2 += x * x;
    }
    G.rad = std::max(G.rad, std::sqrt(r2));
  }
  G.rad = G.rad * (1.0 + 1e-9) + 1e-12;
  for (int s = 0; s < g.nspecies; ++s) {
    const double rc = g.sp[s].rcut, ext = 2.0 * rc + 4.0 * G.rad, m = 4e-6 * ext * ext + 1e-6 * g.sp[s].rcut2;
    G.in2[s] = (float)(g.sp[s].rcut2 - m);
    G.out2[s] = (float)(g.sp[s].rcut2 + m);
    for (int d = 0; d < 3; ++d) G.flim[s][d] = (float)((rc + G.rad) * g.reach[d] * (1.0 + 1e-4) + 1e-4);
  }
  return G;
}

}  // namespace

#define NBR_CHECK(x)                      \
  do {                                    \
    cudaError_t e_ = (x);                 \
    if (e_ != cudaSuccess) return GINT_ECUDA; \
  } while (0)

// Builds the neighbour structure for the current positions (h->pos_dev).  Synchronous.
int gint_build_neighbours(gint_handle *h, cudaStream_t st) {
  GGeom &g = h->geom;
  const long long nb = g.nbricks;
  const unsigned nblk = (unsigned)((nb + kNbrWarps - 1) / kNbrWarps);
  const GBrickGeo G = brick_geo(g);
  // the lists lie in the tiles' scratch buffer, whose contents no call keeps (a buffer of their own was 1 KB a brick)
  const int hrc = gint_tc_reserve_hs(h, nb * kNbrListBytes);
  if (hrc) return hrc;
  int4 *const b_list = reinterpret_cast<int4 *>(h->hs);
  k_frac<<<(unsigned)((g.natoms + 127) / 128), 128, 0, st>>>(g, h->pos_dev, h->frac_dev);
  k_brick_count<<<nblk, 32 * kNbrWarps, 0, st>>>(g, G, h->pos_dev, h->frac_dev, h->species_dev, h->unfold ? 1 : 0, h->n_at,
                                                 h->n_ent, h->n_orb, b_list);
  NBR_CHECK(cudaGetLastError());
  k_brick_scan<<<1, 1024, 0, st>>>(nb, h->n_at, h->n_ent, h->n_orb, h->b_at_off, h->b_ent_off, h->b_pair_off,
                                   h->scan_out);
  NBR_CHECK(cudaGetLastError());
  long long tot[7];
  NBR_CHECK(cudaMemcpyAsync(tot, h->scan_out, sizeof(tot), cudaMemcpyDeviceToHost, st));
  NBR_CHECK(cudaStreamSynchronize(st));
  h->nslots = tot[0];
  h->nent = tot[1];
  h->npairtab = tot[2];
  h->max_brick_orb = (int)tot[3];
  h->max_brick_atoms = (int)tot[4];
  h->W_exec = (double)tot[5];
  h->max_brick_ent = (int)tot[6];
  h->folded = h->nent != h->nslots;  // some slot holds several images
  if (h->max_brick_atoms > GINT_MAX_ATOMS_BRICK) return GINT_ECAPACITY;
  int rc = gint_reserve_nbr(h);
  if (rc) return rc;
  NBR_CHECK(cudaMemsetAsync(h->err_word, 0, sizeof(unsigned), st));
  k_brick_fill<<<nblk, 32 * kNbrWarps, 0, st>>>(g, G, h->pos_dev, h->frac_dev, h->species_dev, h->unfold ? 1 : 0, h->b_at_off,
                                                h->b_ent_off, b_list, h->s_atom, h->s_col, h->s_ent, h->e_shift,
                                                h->err_word);
  NBR_CHECK(cudaGetLastError());
  // sentinel: s_ent[nslots] = nent
  NBR_CHECK(cudaMemcpyAsync(h->s_ent + h->nslots, h->b_ent_off + nb, sizeof(long long), cudaMemcpyDeviceToDevice, st));
  k_brick_pairs<<<nblk, 32 * kNbrWarps, 0, st>>>(g, h->pos_dev, h->species_dev, h->b_at_off, h->s_atom, h->b_pair_off,
                                           h->pair_row_dev, h->pair_col_dev, h->b_pair, h->err_word);
  NBR_CHECK(cudaGetLastError());
  NBR_CHECK(cudaMemsetAsync(h->scal, 0, sizeof(double), st));
  int sms = 0;
  NBR_CHECK(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, h->device));
  k_count_work<<<(unsigned)std::min<long long>(nb, 12LL * sms), GINT_BPTS, 0, st>>>(g, G, h->b_at_off, h->s_atom, h->s_ent, h->e_shift, h->species_dev,
                                                   h->scal);
  NBR_CHECK(cudaGetLastError());
  unsigned err = 0;
  double W = 0;
  NBR_CHECK(cudaMemcpyAsync(&err, h->err_word, sizeof(unsigned), cudaMemcpyDeviceToHost, st));
  NBR_CHECK(cudaMemcpyAsync(&W, h->scal, sizeof(double), cudaMemcpyDeviceToHost, st));
  NBR_CHECK(cudaStreamSynchronize(st));
  h->W = W;
  if (err & GINT_ERRBIT_INDEX) return GINT_EDEVICE;
  if (err & GINT_ERRBIT_SKIN) return GINT_ESKIN;
  return GINT_OK;
}
