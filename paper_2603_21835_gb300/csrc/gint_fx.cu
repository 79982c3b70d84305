// gint_fx.cu -- the float64 density, force and local-Hamiltonian passes (paper Sec. 3.3.1) with their brick
// contractions on the tensor cores, as exact digit products (gint_sgdev.cuh, the arithmetic of gint_sg.cu).
//
// The contraction of a brick (128 points, NP orbitals) takes 128 NP^2 multiply-adds; at the CUDA cores' 2 float64
// ones per clock and SM that is nine tenths of a pass (8-atom Si, 864 bricks: density 2.2 ms, local H 1.8 ms, forces
// 4.3 ms).  Here the CUDA cores evaluate the orbitals only, and the contractions run as 36 float16 digit products:
// 0.52, 0.60 and 0.98 ms.  Left are the evaluations, bound by the float64 pipe (16 cycles a warp instruction and SM),
// and the scratch round trip through L2.  Per 152 bricks: k_fx_eval 52 (density) and 63 us (local H), k_fx_mma 28 to
// 36 us, k_fx_grad 76 us.  Errors against extended precision on that system (Frobenius norm, mean of five geometries),
// CUDA cores -> here: rho 6.9e-16 -> 6.1e-16, H 1.7e-15 -> 9.1e-16, F 2.0e-15 -> 1.9e-15.
//
//   k_fx_dmax, k_fx_ddigits   D rows' exponents and digits, per pair in 8 x 8 core matrices (a row on one scale in
//               all its pairs: a brick without the pair that sets it may have far less of it, see kMaxGap)
//   k_fx_eval   one CTA per brick: orbitals (float64) and their digits into scratch
//     density: rows = points (scale: the point's largest orbital), contraction = orbitals
//     local H: rows = orbitals (scale: the orbital's largest value in the brick, with and without w V),
//              contraction = points
//   k_fx_mma    one CTA per brick, warp roles as k_sg_mma: Y = P D by 64 columns (D's digits gathered by cp.async,
//               whole 16-byte rows of core matrices), rho = rowsum(P Y) or Y itself for the forces; or the
//               128 x 64 tiles of (w V P)^T P at and above the diagonal, added to H in float64 (atomics, as the
//               CUDA-core path; the lower blocks are mirrored at the end)
//   k_fx_grad   one CTA per brick: per atom grad phi contracted with Y (contract64), forces and rho
//
// A launch takes as many bricks as the scratch (the handle's local-H scratch buffer) holds, one per SM.  Systems
// whose bricks have more than kFxMaxCol padded orbitals, or whose scratch could not be allocated, keep the
// CUDA-core kernels.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstring>

#include "gint_handle.cuh"
#include "gint_ptx.cuh"
#include "gint_sg.cuh"
#include "gint_sgdev.cuh"

namespace {
using namespace gptx;
using namespace sgdev;

constexpr int kFxMaxCol = 512;   // padded orbitals of a brick
constexpr int kFxMaxAtoms = 64;
constexpr int kSlices = 4, kEvalT = 128 * kSlices;  // evaluation and gradient kernels: 128 points x slices of slots
constexpr int kDrainWarps = 16, kMmaWarp = 16, kLoadWarp = 17, kGatherWarp = 18, kGatherWarps = 2;
constexpr int kFxThreads = 32 * (kGatherWarp + kGatherWarps);
constexpr uint32_t kFxSmem = kStages * kStage;
constexpr long long kWaitNs = 2000000000LL;
constexpr size_t kHead = 5120;   // per brick: exponents of the rows (A at 0, B at 2048)

// Scratch of one brick: [kHead | P float64, 128 per column | A digits | B digits or Y].
struct FxLayout {
  int np;  // widest brick of the handle (padded columns, multiple of 16)
  size_t p64, a, b, size;
};
__host__ __device__ inline FxLayout fx_layout(int np) {
  FxLayout L{};
  L.np = np;
  const size_t n16 = (np + 15) / 16, mt = (np + 127) / 128, nt = (np + 63) / 64;
  L.p64 = kHead;
  L.a = L.p64 + n16 * 16 * 128 * 8;
  const size_t arho = n16 * kABytes, ah = mt * 8 * kABytes;
  L.b = L.a + (arho > ah ? arho : ah);
  const size_t bh = nt * 8 * kBBytes, y = nt * 64 * 128 * 8;
  L.size = L.b + (bh > y ? bh : y);
  return L;
}

enum { kRho = 0, kY = 1, kH = 2 };

// An orbital's digits are relative to the largest at the point, D's to its row's largest: orbitals of very different
// size (unnormalised bases) would run against each other in the two operands of Y = D P.  Density and forces therefore
// work with P 2^-q (tables that carry the factor) and D 2^q under the contraction index, 2^q the power of two next to
// the orbital's largest radial value: nothing is rounded, and results do not depend on such a scaling of the basis.
struct FxScale {
  signed char q[GINT_MAX_SPECIES][GINT_MAX_ORB_ATOM];  // 0: species without a compiled shape
};
// Columns whose row of D reaches more than 2^kMaxGap beyond what the brick has of it are summed in float64 (digits
// keep 2^-58 of the row's maximum per term, a float64 chain 2^-53 of its own terms).
constexpr int kMaxGap = 4;
constexpr int kLookGap = 1 << 16;                                    // in the second half of eD
constexpr int kPlain = 1 << 20, kPlainInf = kPlain, kPlainGap = kPlain + 1;  // in FxShared::eB

struct FxArgs {
  GCell c;
  GNbr nb;
  const double *otab, *otabq;  // tables of orbitals64, and times 2^-q
  const double2 *tab;        // radial tables (general evaluator)
  const double *D, *V;
  double *rho, *F, *H;
  const unsigned char *Dd;   // D digits
  const int *eD, *atom_off;  // exponents of D's rows by orbital, then those with kLookGap; first orbital of each atom
  int norb;
  const long long *tile_off;
  unsigned char *scr;
  FxLayout L;
  unsigned *err;
  long long b0;              // first brick of the launch
  FxScale q;
  bool upper;                // the density alone reads the pairs I <= J
};

// ------------------------------------------------------------------------------------------- D digits
struct FxD {
  const double *D;
  const int *pair_I, *pair_J, *pair_T, *species;
  const long long *pair_off, *tile_off;
  const int *atom_off;
  int *eD;
  unsigned char *Dd;
  int npairs, norb;
  FxScale q;
  bool upper;  // the density alone reads the pairs I <= J (the others are their transposes), as every precision does
};
// Element (i, j) of pair p at D[ri i + rj j].
__device__ __forceinline__ const double *d_block(const FxD &P, int p, int nI, int nJ, int &ri, int &rj) {
  const bool t = P.upper && P.pair_I[p] > P.pair_J[p];
  ri = t ? 1 : nJ;
  rj = t ? nI : 1;
  return P.D + P.pair_off[t ? P.pair_T[p] : p];
}
// One warp per pair, one lane per row: the row's largest exponent.
__global__ void __launch_bounds__(256) k_fx_dmax(const __grid_constant__ GTabs g, FxD P) {
  const int p = blockIdx.x * 8 + (threadIdx.x >> 5), i = threadIdx.x & 31;
  if (p >= P.npairs) return;
  const int I = P.pair_I[p], J = P.pair_J[p], nI = g.sp[P.species[I]].norb, nJ = g.sp[P.species[J]].norb;
  if (i >= nI) return;
  int ri, rj, m = 1;
  const double *D = d_block(P, p, nI, nJ, ri, rj);
  const signed char *q = P.q.q[P.species[J]];
  for (int j = 0; j < nJ; ++j) m = max(m, exp_field(times_pow2(D[i * ri + j * rj], q[j])));
  atomicMax(P.eD + P.atom_off[I] + i, m);
  if (I == J) P.eD[P.norb + P.atom_off[I] + i] = m;
}
// One warp per pair, units of (row, 8 columns); core matrix (row group, column group): 1 KB, digit s at 128 s.
__global__ void __launch_bounds__(256) k_fx_ddigits(const __grid_constant__ GTabs g, FxD P) {
  const int p = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (p >= P.npairs) return;
  const int I = P.pair_I[p], J = P.pair_J[p];
  const GSpecies &SI = g.sp[P.species[I]], &SJ = g.sp[P.species[J]];
  const int nI = SI.norb, nJ = SJ.norb, gJ = SJ.porb >> 3;
  const signed char *q = P.q.q[P.species[J]];
  int ri, rj;
  const double *D = d_block(P, p, nI, nJ, ri, rj);
  unsigned char *dst = P.Dd + P.tile_off[p] * 16;
  if (I == J && lane < nI) {  // (rows whose maximum lies far above the own block's: k_fx_mma looks at the brick's part)
    const int o = P.atom_off[I] + lane, e = P.eD[o];
    P.eD[P.norb + o] = e < kNonFinite && e - P.eD[P.norb + o] > kMaxGap ? e | kLookGap : e;
  }
  for (int u = lane; u < SI.porb * gJ; u += 32) {
    const int i = u / gJ, kg = u - i * gJ;
    const int em = i < nI ? P.eD[P.atom_off[I] + i] : 1;
    store_digits([&](int j) { return i < nI && 8 * kg + j < nJ ? times_pow2(D[i * ri + (8 * kg + j) * rj], q[8 * kg + j]) : 0.0; },
                 em, dst + (size_t)((i >> 3) * gJ + kg) * 1024 + (i & 7) * 16, 128);
  }
}

// ----------------------------------------------------------------------------------------- brick slots
// The brick's slots: atom, species, first column (columns padded to 8 per atom, contiguous), entries.
struct Slots {
  int atom[kFxMaxAtoms], sp[kFxMaxAtoms], col[kFxMaxAtoms + 1];
  long long e0[kFxMaxAtoms + 1];
  int na, np;  // np: columns
};
__device__ __forceinline__ void load_slots(const GTabs &g, const GNbr &nb, long long b, Slots &S) {
  const long long s0 = nb.b_at_off[b];
  const int na = (int)(nb.b_at_off[b + 1] - s0);
  for (int a = threadIdx.x; a < na; a += blockDim.x) {
    S.atom[a] = nb.s_atom[s0 + a];
    S.sp[a] = nb.atom_species[S.atom[a]];
    S.e0[a] = nb.s_ent[s0 + a];
    if (a == na - 1) S.e0[na] = nb.s_ent[s0 + na];
  }
  __syncthreads();
  if (threadIdx.x < 32) {
    int run = 0;
    for (int a0 = 0; a0 < na; a0 += 32) {
      const int a = a0 + threadIdx.x, po = a < na ? g.sp[S.sp[a]].porb : 0;
      int x = po;
      for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, x, o);
        if ((int)threadIdx.x >= o) x += y;
      }
      if (a < na) S.col[a] = run + x - po;
      run += __shfl_sync(0xffffffffu, x, 31);
    }
    if (threadIdx.x == 0) {
      S.col[na] = run;
      S.na = na;
      S.np = run;
    }
  }
  __syncthreads();
}
// Grid index of point p of the brick; false outside the grid.
__device__ __forceinline__ bool fx_index(const FxArgs &P, long long b, int p, long long &gidx) {
  int i, j, k;
  const bool valid = brick_point(P.c, b, p, i, j, k);
  gidx = valid ? grid_index(P.c, i, j, k) : 0;
  return valid;
}
// Fractions i / n1, j / n2, k / n3 of the brick's 4 + 4 + 8 index values (one division each for the whole CTA), and a
// point's position from them, in grid_point's order.
__device__ __forceinline__ void fx_fractions(const FxArgs &P, long long b, double *fr) {
  if (threadIdx.x < GINT_BI + GINT_BJ + GINT_BK) {
    const int t = threadIdx.x, ax = t < GINT_BI ? 0 : t < GINT_BI + GINT_BJ ? 1 : 2;
    const unsigned nbk = (unsigned)P.c.nbk, q = (unsigned)b / nbk;
    const int bk = (int)((unsigned)b - q * nbk), bj = (int)(q % (unsigned)P.c.nbj), bi = (int)(q / (unsigned)P.c.nbj);
    const int i = ax == 0 ? bi * GINT_BI + t : ax == 1 ? bj * GINT_BJ + t - GINT_BI : bk * GINT_BK + t - GINT_BI - GINT_BJ;
    fr[t] = (double)i / (ax == 0 ? P.c.n1 : ax == 1 ? P.c.n2 : P.c.n3);
  }
}
__device__ __forceinline__ void fx_position(const FxArgs &P, const double *fr, int p, double r[3]) {
  const double fi = fr[p >> 5], fj = fr[GINT_BI + ((p >> 3) & 3)], fk = fr[GINT_BI + GINT_BJ + (p & 7)];
#pragma unroll
  for (int d = 0; d < 3; ++d) r[d] = fi * P.c.cell[d] + fj * P.c.cell[3 + d] + fk * P.c.cell[6 + d];
}

// ----------------------------------------------------------------------------------------- evaluation
// Orbitals of slot a at the thread's point into column-major P64 (rows 0 .. porb, padding zero); returns the
// largest exponent field.
template <int NS, int NP, int ND, int NO, bool RHO>
__device__ __forceinline__ int eval_slot(const GTabs &g, const FxArgs &P, const Slots &S, int a, const double r[3], bool valid,
                                         double *out) {
  const GSpecies &G = g.sp[S.sp[a]];
  double v[NO];
#pragma unroll
  for (int i = 0; i < NO; ++i) v[i] = 0.0;
  if (valid)
    for (long long e = S.e0[a]; e < S.e0[a + 1]; ++e) {
      const double dx = r[0] - P.nb.e_shift[3 * e], dy = r[1] - P.nb.e_shift[3 * e + 1], dz = r[2] - P.nb.e_shift[3 * e + 2];
      const double r2 = fma(dz, dz, fma(dy, dy, dx * dx));
      if (r2 < G.rcut2) {
        if constexpr (NS + NP + ND > 0)
          orbitals64<NS, NP, ND>(g, RHO ? P.otabq : P.otab, G, dx, dy, dz, r2, v);
        else
          add_orbitals<double, true, false>(g, P.tab, S.sp[a], dx, dy, dz, v, nullptr);
      }
    }
  int em = 1;
  constexpr int PO = (NO + 7) / 8 * 8;
  const int po = NS + NP + ND > 0 ? PO : G.porb;
#pragma unroll
  for (int i = 0; i < PO; ++i)
    if (i < po) {
      const double x = i < NO ? v[i < NO ? i : 0] : 0.0;
      out[i * 128] = x;
      em = max(em, exp_field(x));
    }
  return em;
}

template <bool RHO>
__global__ void __launch_bounds__(kEvalT) k_fx_eval(const __grid_constant__ GTabs g, const __grid_constant__ FxArgs P) {
  __shared__ Slots S;
  __shared__ int s_e[128];
  __shared__ double s_fr[16];
  __shared__ double s_wv[128];
  const long long b = P.b0 + blockIdx.x;
  const int t = threadIdx.x, p = t & 127, q = t >> 7;
  grid_wait();
  unsigned char *scr = P.scr + blockIdx.x * P.L.size;
  double *P64 = reinterpret_cast<double *>(scr + P.L.p64);
  int *eA = reinterpret_cast<int *>(scr), *eB = reinterpret_cast<int *>(scr + 2048);
  if (t < 128) s_e[t] = 1;
  fx_fractions(P, b, s_fr);
  load_slots(g, P.nb, b, S);
  const int na = S.na, np = S.np;
  if (na == 0) return;
  double r[3];
  long long gidx;
  const bool valid = fx_index(P, b, p, gidx);
  fx_position(P, s_fr, p, r);
  if (!RHO && q == 0) s_wv[p] = valid ? P.c.w * P.V[gidx] : 0.0;
  int em = 1;
  for (int a = q; a < na; a += kSlices) {
    double *out = P64 + (long long)S.col[a] * 128 + p;
    switch (g.sp[S.sp[a]].shape) {
#define CASE_E(ns, np_, nd, no) \
  case GINT_SHAPE(ns, np_, nd): em = max(em, eval_slot<ns, np_, nd, no, RHO>(g, P, S, a, r, valid, out)); break;
      GINT_O64_SHAPES(CASE_E)
#undef CASE_E
      default: em = max(em, eval_slot<0, 0, 0, GINT_MAX_ORB_ATOM, RHO>(g, P, S, a, r, valid, out));
    }
  }
  const int n16 = (np + 15) & ~15;
  for (int c = np + q; c < n16; c += kSlices) P64[c * 128 + p] = 0.0;
  if (RHO) atomicMax(&s_e[p], em);
  __syncthreads();
  if (RHO) {
    const int e = s_e[p];
    if (q == 0) eA[p] = e;
    for (int G = q; G < n16 / 8; G += kSlices)
      store_digits([&](int j) { return P64[(8 * G + j) * 128 + p]; }, e,
                   scr + P.L.a + (size_t)(G >> 1) * kABytes + (p >> 3) * 256 + (G & 1) * 128 + (p & 7) * 16, kTM * kCK * 2);
  } else {
    const int warp = t >> 5, lane = t & 31;
    for (int n = warp; n < n16; n += kEvalT / 32) {  // row exponents of w V phi and phi
      int ma = 1, mb = 1;
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const double x = P64[n * 128 + lane + 32 * k];
        ma = max(ma, exp_field(x * s_wv[lane + 32 * k]));
        mb = max(mb, exp_field(x));
      }
      for (int o = 16; o > 0; o >>= 1) {
        ma = max(ma, __shfl_xor_sync(0xffffffffu, ma, o));
        mb = max(mb, __shfl_xor_sync(0xffffffffu, mb, o));
      }
      if (lane == 0) {
        eA[n] = ma;
        eB[n] = mb;
      }
    }
    __syncthreads();
    for (int u = t; u < n16 * 16; u += kEvalT) {  // eight rows fastest, then the 16 groups of 8 points
      const int n = (u & 7) | ((u >> 7) << 3), G = (u >> 3) & 15;
      const double *x = P64 + n * 128 + 8 * G;
      store_digits([&](int j) { return x[j] * s_wv[8 * G + j]; }, eA[n],
                   scr + P.L.a + (size_t)((n >> 7) * 8 + (G >> 1)) * kABytes + ((n & 127) >> 3) * 256 + (G & 1) * 128 + (n & 7) * 16,
                   kTM * kCK * 2);
      store_digits([&](int j) { return x[j]; }, eB[n],
                   scr + P.L.b + (size_t)((n >> 6) * 8 + (G >> 1)) * kBBytes + ((n & 63) >> 3) * 256 + (G & 1) * 128 + (n & 7) * 16,
                   kTN * kCK * 2);
    }
  }
  asm volatile("fence.proxy.async;" ::: "memory");  // the digits are read by bulk copies
}

// ------------------------------------------------------------------------------------------- products
struct FxShared {
  uint64_t full[kStages], empty[kStages], accfull[2], accfree[2];
  uint32_t tmem;
  Slots S;
  unsigned char grp_slot[kFxMaxCol / 8];  // slot of each 8 columns
  short col_orb[kFxMaxCol];   // orbital of its atom, -1: padding
  int eB[kFxMaxCol];
  // density: D's core matrix of (column group, column group), local H: the block offset of (slot, slot); -1: none
  int tab[kFxMaxCol / 8 * (kFxMaxCol / 8)];
  double rho[3][128];
};
__device__ __forceinline__ void cp_async16(void *dst, const void *src, bool in) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(smem_u32(dst)), "l"(src), "r"(in ? 16 : 0) : "memory");
}

// Element (i, j) of slots (a, c)' block at D[ri i + rj j]; null: no pair.
__device__ __forceinline__ const double *slot_block(const GTabs &g, const FxArgs &P, const Slots &S, long long b, int a, int c,
                                                    int &ri, int &rj) {
  const bool t = P.upper && S.atom[a] > S.atom[c];
  const int pr = P.nb.b_pair[P.nb.b_pair_off[b] + (t ? c * S.na + a : a * S.na + c)];
  ri = t ? 1 : g.sp[S.sp[c]].norb;
  rj = t ? g.sp[S.sp[a]].norb : 1;
  return pr < 0 ? nullptr : P.D + P.nb.pair_off[pr];
}
// Largest exponent of D 2^q in the brick's part of row i of slot a's atom.
__device__ __noinline__ int fx_brick_row(const GTabs &g, const FxArgs &P, const Slots &S, long long b, int a, int i) {
  int m = 1;
  for (int c = 0; c < S.na; ++c) {
    int ri, rj;
    const double *D = slot_block(g, P, S, b, a, c, ri, rj);
    if (!D) continue;
    for (int j = 0; j < g.sp[S.sp[c]].norb; ++j) m = max(m, exp_field(times_pow2(D[i * ri + j * rj], P.q.q[S.sp[c]][j])));
  }
  return m;
}
// Sums without digits, where a row holds an infinity or a NaN: over the atoms that reach one of the point's 32
// (the CUDA-core path's slabs, whose rule decides which results a non-finite input reaches).
__device__ __forceinline__ bool fx_reaches(const GTabs &g, const Slots &S, const double *P64, int a, int slab) {
  const int no = g.sp[S.sp[a]].norb;
  for (int i = 0; i < no; ++i)
    for (int p = 0; p < 32; ++p)
      if (P64[(S.col[a] + i) * 128 + 32 * slab + p] != 0.0) return true;
  return false;
}
__device__ __noinline__ double fx_plain_y(const GTabs &g, const FxArgs &P, const FxShared &sh, long long b, const double *P64,
                                          int n, int p) {
  const int na = sh.S.na, c = sh.grp_slot[n >> 3], i = sh.col_orb[n];
  const bool finite = sh.eB[n] == kPlainGap;  // (an atom that does not reach adds zeros)
  double y = 0.0;
  if (!finite && !fx_reaches(g, sh.S, P64, c, p >> 5)) return y;
  for (int a = 0; a < na; ++a) {
    int ri, rj;
    const double *D = slot_block(g, P, sh.S, b, c, a, ri, rj);
    if (!D || (!finite && !fx_reaches(g, sh.S, P64, a, p >> 5))) continue;
    for (int j = 0; j < g.sp[sh.S.sp[a]].norb; ++j)
      y = fma(D[i * ri + j * rj], times_pow2(P64[(sh.S.col[a] + j) * 128 + p], P.q.q[sh.S.sp[a]][j]), y);
  }
  return y;
}
__device__ __noinline__ double fx_plain_h(const GTabs &g, const FxArgs &P, const FxShared &sh, long long b, const double *P64,
                                          int m, int n) {
  double h = 0.0;
  for (int slab = 0; slab < 4; ++slab) {
    if (!fx_reaches(g, sh.S, P64, sh.grp_slot[m >> 3], slab) || !fx_reaches(g, sh.S, P64, sh.grp_slot[n >> 3], slab)) continue;
    for (int p = 32 * slab; p < 32 * slab + 32; ++p) {
      int i, j, k;
      if (brick_point(P.c, b, p, i, j, k))
        h = fma(P.c.w * P.V[grid_index(P.c, i, j, k)] * P64[m * 128 + p], P64[n * 128 + p], h);
    }
  }
  return h;
}
template <int MODE>
__global__ void __launch_bounds__(kFxThreads, 1) k_fx_mma(const __grid_constant__ GTabs g, const __grid_constant__ FxArgs P) {
  extern __shared__ __align__(1024) unsigned char smem[];
  __shared__ FxShared sh;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const long long b = P.b0 + blockIdx.x;
  if (tid == 0) {
    for (int s = 0; s < kStages; ++s) {
      mbar_init(&sh.full[s], MODE == kH ? 1 : 1 + kGatherWarps);
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
  load_slots(g, P.nb, b, sh.S);
  const int na = sh.S.na, np = sh.S.np;
  grid_wait();
  // column tables
  for (int G = tid; G < np / 8; G += kFxThreads) {
    int a = 0;
    while (sh.S.col[a + 1] <= 8 * G) ++a;
    sh.grp_slot[G] = (unsigned char)a;
    const int no = g.sp[sh.S.sp[a]].norb;
    for (int k = 0; k < 8; ++k) {
      const int i = 8 * G + k - sh.S.col[a];
      sh.col_orb[8 * G + k] = (short)(i < no ? i : -1);
    }
  }
  const int ng8 = np / 8;
  if (MODE == kH)
    for (int e = tid; e < na * na; e += kFxThreads) {
      const int p = P.nb.b_pair[P.nb.b_pair_off[b] + e];
      sh.tab[e] = p < 0 ? -1 : (int)P.nb.pair_off[p];
    }
  unsigned char *scr = P.scr + blockIdx.x * P.L.size;
  const double *P64 = reinterpret_cast<const double *>(scr + P.L.p64);
  const int *eA = reinterpret_cast<const int *>(scr);
  if (MODE == kH)
    for (int c = tid; c < np; c += kFxThreads) sh.eB[c] = reinterpret_cast<const int *>(scr + 2048)[c];
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (MODE != kH) {
    // the row's exponent (density: that of Y 2^q, to meet P 2^-q), or why the column is summed in float64: an infinity or
    // a NaN, or the brick's part of the row too far below its maximum (looked at only where the own atom's block, which
    // every brick of the atom has, is)
    for (int c = tid; c < np; c += kFxThreads) {
      const int a = sh.grp_slot[c >> 3], i = sh.col_orb[c];
      int e = i < 0 ? 1 : P.eD[P.norb + P.atom_off[sh.S.atom[a]] + i];
      const bool gap = e >= kLookGap && e - kLookGap - fx_brick_row(g, P, sh.S, b, a, i) > kMaxGap;
      e &= kLookGap - 1;
      sh.eB[c] = gap ? kPlainGap : e == kNonFinite ? kPlainInf : MODE == kRho && i >= 0 ? e + P.q.q[sh.S.sp[a]][i] : e;
    }
    for (int e = tid; e < ng8 * ng8; e += kFxThreads) {
      const int n = e / ng8, k = e - n * ng8, sn = sh.grp_slot[n], sk = sh.grp_slot[k];
      const int p = P.nb.b_pair[P.nb.b_pair_off[b] + sn * na + sk];
      const int gk = (sh.S.col[sk + 1] - sh.S.col[sk]) >> 3;
      sh.tab[e] = p < 0 ? -1 : (int)(P.tile_off[p] >> 6) + (n - (sh.S.col[sn] >> 3)) * gk + (k - (sh.S.col[sk] >> 3));
    }
    __syncthreads();
  }
  const uint32_t tmem = sh.tmem;
  unsigned *err = P.err;
  const int nt = (np + 63) / 64, mt = MODE == kH ? (np + 127) / 128 : 1;
  const int nq = MODE == kH ? 8 : (np + 15) / 16;
  // tiles (m, n) in order; local H: those at and above the diagonal
  auto next_tile = [&](int &m, int &n) {
    if (++n == nt) {
      ++m;
      n = MODE == kH ? 2 * m : 0;
    }
    return m < mt;
  };

  if (warp == kLoadWarp) {
    int gl = 0;
    bool ok = na > 0;
    for (int m = 0, n = 0; ok && m < mt; next_tile(m, n))
      for (int c = 0; c < nq && ok; ++c, ++gl) {
        const int s = gl % kStages;
        if (gl >= kStages)
          ok = __all_sync(0xffffffffu, mbar_wait(&sh.empty[s], (uint32_t)(gl / kStages - 1) & 1u, err, GINT_ERRBIT_TIMEOUT, kWaitNs));
        if (!ok) break;
        if (lane == 0) {
          mbar_arrive_tx(&sh.full[s], MODE == kH ? kStage : kABytes);
          bulk_g2s(smem + s * kStage, scr + P.L.a + (size_t)(MODE == kH ? m * 8 + c : c) * kABytes, kABytes, &sh.full[s]);
          if (MODE == kH)
            bulk_g2s(smem + s * kStage + kABytes, scr + P.L.b + (size_t)(n * 8 + c) * kBBytes, kBBytes, &sh.full[s]);
        }
        __syncwarp();
      }
    for (int c = max(0, gl - kStages); c < gl; ++c)
      mbar_wait(&sh.full[c % kStages], (uint32_t)(c / kStages) & 1u, err, GINT_ERRBIT_TIMEOUT, kWaitNs);
  } else if (warp >= kGatherWarp) {
    if (MODE != kH) {
      // D digits of (64 columns n, 16 orbitals k): thread = (digit, row of 8), two chunks of copies in flight
      const int t = tid - 32 * kGatherWarp, row = t & 7, d = t >> 3;
      int gl = 0;
      bool ok = na > 0;
      auto land = [&](int c) {  // chunk c's copies of this warp are complete
        fence_async_smem();
        __syncwarp();
        if (lane == 0) mbar_arrive(&sh.full[c % kStages]);
      };
      for (int n = 0; n < nt && ok; ++n)
        for (int c = 0; c < nq && ok; ++c, ++gl) {
          const int s = gl % kStages;
          if (gl >= kStages)
            ok = __all_sync(0xffffffffu, mbar_wait(&sh.empty[s], (uint32_t)(gl / kStages - 1) & 1u, err, GINT_ERRBIT_TIMEOUT, kWaitNs));
          if (!ok) break;
          unsigned char *B = smem + s * kStage + kABytes + d * (kTN * kCK * 2) + row * 16;
#pragma unroll
          for (int u = 0; u < 16; ++u) {
            const int ng = 8 * n + (u >> 1), kg = 2 * c + (u & 1);
            const int core = ng < ng8 && kg < ng8 ? sh.tab[ng * ng8 + kg] : -1;
            cp_async16(B + (u >> 1) * 256 + (u & 1) * 128, P.Dd + (size_t)max(core, 0) * 1024 + d * 128 + row * 16, core >= 0);
          }
          asm volatile("cp.async.commit_group;" ::: "memory");
          if (gl >= 2) {
            asm volatile("cp.async.wait_group 2;" ::: "memory");
            land(gl - 2);
          }
        }
      asm volatile("cp.async.wait_group 0;" ::: "memory");
      for (int c = max(0, gl - 2); c < gl; ++c) land(c);
    }
  } else if (warp == kMmaWarp) {
    const uint32_t sbase = smem_u32(smem);
    int gc = 0, gb = 0;
    bool ok = na > 0;
    for (int m = 0, n = 0; ok && m < mt; next_tile(m, n))
      for (int c = 0; c < nq; ++c, ++gc) {
        const int s = gc % kStages, cr = c % kRangeChunks;
        const bool first = cr == 0, last = cr == kRangeChunks - 1 || c == nq - 1;
        if (first) ++gb;
        const uint32_t fpar = (uint32_t)(gb - 2) & 1u;
        ok = mbar_wait(&sh.full[s], (uint32_t)(gc / kStages) & 1u, err, GINT_ERRBIT_TIMEOUT, kWaitNs);
        if (first && gb > 1) ok = ok && mbar_wait(&sh.accfree[0], fpar, err, GINT_ERRBIT_TIMEOUT, kWaitNs);
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
          ok = __all_sync(0xffffffffu, mbar_wait(&sh.accfree[1], fpar, err, GINT_ERRBIT_TIMEOUT, kWaitNs));
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
    if (na > 0) {  // the MMAs issued so far are complete before the tensor memory is given back
      if (!ok && elect_one()) mma_commit(&sh.empty[gc % kStages]);
      __syncwarp();
      const int q = ok ? gc - 1 : gc;
      mbar_wait(&sh.empty[q % kStages], (uint32_t)(q / kStages) & 1u, err, GINT_ERRBIT_TIMEOUT, kWaitNs);
    }
  } else {
    const int c0 = (warp >> 2) * 16, row = (warp & 3) * 32 + lane;
    const uint32_t lbase = tmem + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)c0;
    int gb = 0;
    bool ok = na > 0;
    double racc = 0.0;
    const int nr = (nq + kRangeChunks - 1) / kRangeChunks;
    for (int m = 0, n = 0; ok && m < mt; next_tile(m, n)) {
      Fx x[16];
#pragma unroll
      for (int j = 0; j < 16; ++j) x[j] = Fx{0u, 0u, 0u};
      for (int r = 0; r < nr && ok; ++r, ++gb)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          ok = ok && __all_sync(0xffffffffu, mbar_wait(&sh.accfull[h], (uint32_t)gb & 1u, err, GINT_ERRBIT_TIMEOUT, kWaitNs));
          if (!ok) break;
          tc_fence_after();
          drain_half(lbase, h, x);
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(&sh.accfree[h]);
        }
      if (!ok) break;
      const int jb = 64 * n + c0;  // first column of this warp
      if (jb >= np) continue;
      const int i = 128 * m + row;
      if (MODE == kH) {
        if (i >= np) continue;
        const int ai = sh.grp_slot[i >> 3], li = sh.col_orb[i], ea = eA[i];
        if (li < 0) continue;
        unsigned plain = 0;
#pragma unroll
        for (int j8 = 0; j8 < 16; j8 += 8) {
          if (jb + j8 >= np) break;
          const int aj = sh.grp_slot[(jb + j8) >> 3], no = g.sp[sh.S.sp[aj]].norb, o = sh.tab[ai * na + aj];
          if (o < 0 || aj < ai) continue;
          const int lj0 = jb + j8 - sh.S.col[aj];
          double *const blk = P.H + (long long)o + (long long)li * no + lj0;
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            const int col = jb + j8 + j;
            if (lj0 + j >= no || col < i) continue;  // (an atom may lie across two row tiles: its lower triangle is mirrored)
            const int eb = sh.eB[col];
            if (max(ea, eb) == kNonFinite)
              plain |= 1u << (j8 + j);
            else
              atomicAdd(blk + j, fx_to_double(x[j8 + j], ea + eb - 2 * 1022 - 68));
          }
        }
        while (plain) {  // rows with an infinity or a NaN
          const int col = jb + __ffs(plain) - 1, aj = sh.grp_slot[col >> 3];
          plain &= plain - 1;
          atomicAdd(P.H + sh.tab[ai * na + aj] + (long long)li * g.sp[sh.S.sp[aj]].norb + col - sh.S.col[aj],
                    fx_plain_h(g, P, sh, b, P64, i, col));
        }
      } else {
        const int ea = eA[row];
        double *const Y = reinterpret_cast<double *>(scr + P.L.b);
#pragma unroll
        for (int j8 = 0; j8 < 16; j8 += 8) {
          if (jb + j8 >= np) break;
          double pv[8];
          if (MODE == kRho) {
#pragma unroll
            for (int j = 0; j < 8; ++j) pv[j] = P64[(jb + j8 + j) * 128 + row];
          }
          unsigned plain = 0;
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            const int col = jb + j8 + j, eb = sh.eB[col];
            const double v = fx_to_double(x[j8 + j], ea + eb - 2 * 1022 - 68);
            if (MODE == kY)
              Y[col * 128 + row] = v;
            else if (eb < kPlain)
              racc = fma(pv[j], v, racc);
            if (eb >= kPlain) plain |= 1u << j;
          }
          while (plain) {
            const int col = jb + j8 + __ffs(plain) - 1;
            plain &= plain - 1;
            const double v = fx_plain_y(g, P, sh, b, P64, col, row);
            if (MODE == kY)
              Y[col * 128 + row] = v;
            else
              racc = fma(times_pow2(P64[col * 128 + row], P.q.q[sh.S.sp[sh.grp_slot[col >> 3]]][sh.col_orb[col]]), v, racc);
          }
        }
      }
    }
    if (MODE == kRho) {
      if (warp >= 4) sh.rho[(warp >> 2) - 1][row] = racc;
      asm volatile("bar.sync 1, %0;" ::"n"(32 * kDrainWarps) : "memory");
      if (warp < 4) {
        long long gidx;
        if (fx_index(P, b, row, gidx)) P.rho[gidx] = ((racc + sh.rho[0][row]) + sh.rho[1][row]) + sh.rho[2][row];
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == kMmaWarp) tmem_dealloc(tmem, 512);
}

// ------------------------------------------------------------------------------------------- forces
template <int NS, int NP, int ND, int NO>
__device__ __forceinline__ void grad_slot(const GTabs &g, const FxArgs &P, const Slots &S, int a, const double r[3], bool valid,
                                          const double *Y, double &rho, double f[3]) {
  const GSpecies &G = g.sp[S.sp[a]];
  double c[NO];
#pragma unroll
  for (int i = 0; i < NO; ++i) c[i] = i < G.norb ? Y[i * 128] : 0.0;
  if (!valid) return;
  for (long long e = S.e0[a]; e < S.e0[a + 1]; ++e) {
    const double dx = r[0] - P.nb.e_shift[3 * e], dy = r[1] - P.nb.e_shift[3 * e + 1], dz = r[2] - P.nb.e_shift[3 * e + 2];
    const double r2 = fma(dz, dz, fma(dy, dy, dx * dx));
    if (r2 >= G.rcut2) continue;
    if constexpr (NS + NP + ND > 0) {
      contract64<NS, NP, ND>(g, P.otab, G, dx, dy, dz, r2, c, rho, f[0], f[1], f[2]);
    } else {
      double v[NO], gv[NO][3];
      for (int i = 0; i < G.norb; ++i) v[i] = gv[i][0] = gv[i][1] = gv[i][2] = 0.0;
      add_orbitals<double, true, true>(g, P.tab, S.sp[a], dx, dy, dz, v, gv);
      for (int i = 0; i < G.norb; ++i) {
        rho = fma(c[i], v[i], rho);
        for (int d = 0; d < 3; ++d) f[d] = fma(c[i], gv[i][d], f[d]);
      }
    }
  }
}

__global__ void __launch_bounds__(kEvalT) k_fx_grad(const __grid_constant__ GTabs g, const __grid_constant__ FxArgs P) {
  __shared__ Slots S;
  __shared__ double s_rho[kSlices - 1][128], s_fr[16];
  const long long b = P.b0 + blockIdx.x;
  const int t = threadIdx.x, p = t & 127, q = t >> 7, lane = t & 31;
  fx_fractions(P, b, s_fr);
  load_slots(g, P.nb, b, S);
  grid_wait();
  const int na = S.na;
  double r[3], rho = 0.0;
  long long gidx;
  const bool valid = fx_index(P, b, p, gidx);
  fx_position(P, s_fr, p, r);
  const double wv2 = valid ? 2.0 * (P.c.w * P.V[gidx]) : 0.0;
  const double *Y = reinterpret_cast<const double *>(P.scr + blockIdx.x * P.L.size + P.L.b);
  for (int a = q; a < na; a += kSlices) {
    double f[3] = {0.0, 0.0, 0.0};
    const double *y = Y + (long long)S.col[a] * 128 + p;
    switch (g.sp[S.sp[a]].shape) {
#define CASE_G(ns, np_, nd, no) \
  case GINT_SHAPE(ns, np_, nd): grad_slot<ns, np_, nd, no>(g, P, S, a, r, valid, y, rho, f); break;
      GINT_O64_SHAPES(CASE_G)
#undef CASE_G
      default: grad_slot<0, 0, 0, GINT_MAX_ORB_ATOM>(g, P, S, a, r, valid, y, rho, f);
    }
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      f[d] *= wv2;
      for (int o = 16; o > 0; o >>= 1) f[d] += __shfl_xor_sync(0xffffffffu, f[d], o);
    }
    if (lane == 0)
      for (int d = 0; d < 3; ++d) atomicAdd(P.F + 3 * S.atom[a] + d, f[d]);
  }
  if (!P.rho) return;
  if (q > 0) s_rho[q - 1][p] = rho;
  __syncthreads();
  if (q == 0 && valid) P.rho[gidx] = ((rho + s_rho[0][p]) + s_rho[1][p]) + s_rho[2][p];
}

// H_JI = H_IJ^T for the lower pairs, and the lower triangles of the diagonal blocks.
__global__ void __launch_bounds__(256) k_fx_mirror(const __grid_constant__ GTabs g, const int *__restrict__ pair_I,
                                                  const int *__restrict__ pair_J, const int *__restrict__ pair_T,
                                                  const long long *__restrict__ pair_off, const int *__restrict__ species,
                                                  int npairs, double *__restrict__ H) {
  const int p = blockIdx.x * 8 + (threadIdx.x >> 5);
  if (p >= npairs || pair_I[p] < pair_J[p]) return;
  const bool diag = pair_I[p] == pair_J[p];
  const int nI = g.sp[species[pair_I[p]]].norb, nJ = g.sp[species[pair_J[p]]].norb;
  const double *src = H + pair_off[pair_T[p]];
  double *dst = H + pair_off[p];
  for (int e = threadIdx.x & 31; e < nI * nJ; e += 32) {
    const int i = e / nJ, j = e - i * nJ;
    if (!diag || j < i) dst[e] = src[j * nI + i];
  }
}

// D digits at the start of the scratch, then the bricks.
size_t fx_dbytes(const gint_handle *h) { return ((size_t)std::max(h->ntile_elems, 64LL) * 16 + 1023) & ~(size_t)1023; }

int fx_args(gint_handle *h, FxArgs &P) {
  P.c = static_cast<const GCell &>(h->geom);
  P.nb = h->nbr();
  P.otab = h->otab64;
  P.otabq = h->otab64q;
  P.tab = h->tab64;
  P.tile_off = h->tile_off_dev;
  unsigned char *s = reinterpret_cast<unsigned char *>(h->hs);
  P.Dd = s;
  P.scr = s + fx_dbytes(h);
  P.eD = h->fx_eD;
  P.norb = h->norb;
  static_assert(sizeof(P.q.q) == sizeof(h->fx_q), "");
  memcpy(P.q.q, h->fx_q, sizeof(P.q.q));
  P.atom_off = h->atom_off_dev;
  P.L = fx_layout(h->max_brick_porb);
  P.err = h->err_word;
  return GINT_OK;
}

template <typename K>
int big_smem(K *k) {
  return cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kFxSmem) == cudaSuccess ? GINT_OK : GINT_ECUDA;
}

}  // namespace

long long gint_fx_bytes(const gint_handle *h, int bricks) {
  if (h->max_brick_porb > kFxMaxCol || h->max_brick_atoms > kFxMaxAtoms || h->max_brick_porb < 1 ||
      h->nblock > 0x7fffffffLL)
    return 0;
  return (long long)fx_dbytes(h) + (long long)bricks * (long long)fx_layout(h->max_brick_porb).size;
}

int gint_fx_rho(gint_handle *h, const double *D, double *rho, const double *V, double *F, cudaStream_t st) {
  const long long nb = h->geom.nbricks;
  if (nb == 0) return GINT_OK;
  FxArgs P{};
  fx_args(h, P);
  P.D = D;
  P.V = V;
  P.rho = rho;
  P.F = F;
  P.upper = F == nullptr;
  FxD Q{D, h->pair_I_dev, h->pair_col_dev, h->pair_T_dev, h->species_dev, h->pair_off_dev, h->tile_off_dev, h->atom_off_dev,
        h->fx_eD, const_cast<unsigned char *>(P.Dd), h->npairs, h->norb, P.q, F == nullptr};
  if (cudaMemsetAsync(h->fx_eD, 0, 2 * (size_t)h->norb * sizeof(int), st) != cudaSuccess) return GINT_ECUDA;
  const unsigned pg = (unsigned)((h->npairs + 7) / 8);
  k_fx_dmax<<<pg, 256, 0, st>>>(h->tabs64, Q);
  k_fx_ddigits<<<pg, 256, 0, st>>>(h->tabs64, Q);
  int rc;
  if ((rc = F ? big_smem(k_fx_mma<kY>) : big_smem(k_fx_mma<kRho>))) return rc;
  for (long long b0 = 0; b0 < nb; b0 += h->fx_batch) {
    P.b0 = b0;
    const dim3 grid((unsigned)std::min<long long>(h->fx_batch, nb - b0));
    if ((rc = gla::sg_launch(k_fx_eval<true>, grid, kEvalT, 0, st, h->tabs64, P)) ||
        (rc = gla::sg_launch(F ? k_fx_mma<kY> : k_fx_mma<kRho>, grid, kFxThreads, kFxSmem, st, h->tabs64, P)))
      return rc;
    if (F && (rc = gla::sg_launch(k_fx_grad, grid, kEvalT, 0, st, h->tabs64, P))) return rc;
  }
  return cudaGetLastError() == cudaSuccess ? GINT_OK : GINT_ECUDA;
}

int gint_fx_vlocal(gint_handle *h, const double *V, double *H, cudaStream_t st) {
  const long long nb = h->geom.nbricks;
  if (nb == 0) return GINT_OK;
  FxArgs P{};
  fx_args(h, P);
  P.V = V;
  P.H = H;
  int rc;
  if ((rc = big_smem(k_fx_mma<kH>))) return rc;
  for (long long b0 = 0; b0 < nb; b0 += h->fx_batch) {
    P.b0 = b0;
    const dim3 grid((unsigned)std::min<long long>(h->fx_batch, nb - b0));
    if ((rc = gla::sg_launch(k_fx_eval<false>, grid, kEvalT, 0, st, h->tabs64, P)) ||
        (rc = gla::sg_launch(k_fx_mma<kH>, grid, kFxThreads, kFxSmem, st, h->tabs64, P)))
      return rc;
  }
  k_fx_mirror<<<(unsigned)((h->npairs + 7) / 8), 256, 0, st>>>(h->tabs64, h->pair_I_dev, h->pair_col_dev, h->pair_T_dev,
                                                              h->pair_off_dev, h->species_dev, h->npairs, H);
  return cudaGetLastError() == cudaSuccess ? GINT_OK : GINT_ECUDA;
}
