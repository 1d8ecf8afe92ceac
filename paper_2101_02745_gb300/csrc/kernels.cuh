// kernels.cuh -- GB300 (sm_103a) FP64 device code of the particle-in-cell step
// for the neutrino fast flavour instability (Richers, Willcox, Ford & Myers,
// arXiv:2101.02745).  Included by emu.cu and instances.cuh.
//
// A *batch* is a set of independent 1D periodic boxes advanced together; one
// box is a batch of one.  All arrays of a batch are concatenated:
//   particles: box b occupies [poff_b, poff_b + nz_b * ndir_b) of every SoA array;
//              particle (d, i) of box b is poff_b + d * nz_b + i; component k of a
//              matrix array at [k * Ptot + particle]
//   grid:      cell j of box b is column coff_b + j of A[36][NZ] (the full
//              potential), At[32][NZ] (the step's traceless potential) and mom[72][NZ]
//   tables:    direction d of box b is entry doff_b + d of the per-direction tables
//
// Parallel layout.  Work is split into *units* = (one tile of T cells, one
// direction) of one box: box b has ntiles_b * ndir_b units, numbered box after
// box.  A warp works on one unit at a time with lane l on cell
// (tile * T - H + l): lanes H..H+T-1 own the tile's cells, the H lanes on each
// side are halo lanes that supply the neighbour values of the stencil.  The
// shape orders 0-2 (Sec. 2.2.1) reach one cell on each side (H = 1, T = 30),
// the cubic shape two (H = 2, T = 28).  Because
// the particles of one direction (a ring) translate rigidly (one per cell at a
// common offset, Sec. 3.1 and Eq. 4), the particle on cell j is ring entry
// (j - shift_d) mod nz and its stencil neighbours sit on the adjacent lanes:
// deposit (Eq. 5) and interpolation (Eq. 6) are warp-shuffle gathers.  The
// RK stage has no halo lanes (32-cell tiles, the tile ends through shared
// memory); its commutators and stencil sums run on the integer pipe (wide.cuh).
//
// Schedule.  Large boxes run a fixed grid (2 blocks of 8 warps per SM): in the
// deposit the first nw warps split the U units of the batch into equal contiguous
// ranges, in the RK stage the blocks split the (slab, direction) pairs.  Small
// boxes: a block takes a part of one tile's directions.  The deposit's summation
// order (integer sums over a warp's directions and a part's warps, one partial per
// (warp, tile) or part, partials added in order by k_combine) depends only on the
// batch and the grid: no atomics, bitwise reproducible.
#pragma once

#include <cuda_runtime.h>

#include <cstdint>

#include "wide.cuh"

namespace emu_dev {

constexpr int kWarps = 8;
constexpr int kThreads = kWarps * 32;
constexpr int kLanes = 32;
constexpr int kTileMax = 30;       // most cells a warp owns (shape orders 0-2)
constexpr int kNA = 36;            // components of the grid potential (and of a deposit's partial sums)
// Components of the traceless grid potential the step reads: per moment (n,
// f_x, f_y, f_z) the diagonal differences B_11 - B_22, B_22 - B_33 and the
// six off-diagonal reals.  The trace of H commutes with every rho, so
// -i[H, rho] (Eq. 4) depends on H only through these 8 (per moment: 32).
constexpr int kNT = 32;
constexpr int kNC = 8;             // components of one traceless matrix
constexpr int kNM = 72;            // components of the per-species moments
constexpr int kWSlots = 5;         // weight slots per stage row of the direction weight table (the cubic shape's 5)
constexpr int kSlot = kNA * kTileMax; // doubles in one warp's partial sums for one tile
constexpr double kLatticeTol = 1e-6;
constexpr unsigned kFull = 0xffffffffu;
constexpr int kPersistBlocks = 2 * 152;  // default grid: 2 resident blocks on each of GB300's 152 SMs
constexpr int kMaxBlocks = 4 * 152;      // largest grid the autotuner tries
constexpr int kMaxWarps = kMaxBlocks * kWarps;

enum : int { ERR_LATTICE = 1, ERR_NONFINITE = 2, ERR_WEIGHT = 4, ERR_RING = 8, ERR_STEP = 32 };

// Stencil of the shape of order ORDER (Sec. 2.2.1, orders 0-3): a particle on
// lattice site h (the cell containing it) reaches cells h-H .. h+H, weight
// slots 0 .. NW-1; NWS weight arrays are kept from the deposit for the RK stage
// (none for order 0, whose only weight is 1).
template <int ORDER>
struct Sten {
  static_assert(ORDER >= 0 && ORDER <= 3, "shape orders 0..3");
  static constexpr int H = ORDER == 3 ? 2 : 1;
  static constexpr int T = kLanes - 2 * H;
  static constexpr int NW = 2 * H + 1;
  static constexpr int NWS = ORDER == 0 ? 0 : NW;
  static_assert(T <= kTileMax, "a tile's partial sums must fit a slot");
};

// One box of a batch (device copy lives in the workspace).
struct BoxGeo {
  int nz, M, ntiles, use_dirs;
  int coff, toff, doff, ntiles32;  // ntiles32: 32-cell tiles of the RK stage
  int toff32, sw;                  // toff32: first 32-cell tile of the box among all boxes'; sw: 32-cell tiles of a
                                   // slab of the RK stage (1, 2, 4 or 8)
  int64_t P, poff, uoff, uoff32;   // uoff32: first 32-cell unit of the box
  int64_t soff;                    // first tile unit of the box's slabs (sw per slab and direction)
  double Lz, dz, inv_dz, nz_d, dV, c_light;
  double kappa_dV;   // kappa / dV: scale of the grid potential
  double inv_dV;     // 1 / dV: scale of the moments
  double alpha;      // Eq. 9 perturbation strength (init)
  uint64_t seed;     // Eq. 9 random stream (init)
  double cfl_adv, cfl_flavor, kappa;  // Eq. 7
  double n_e;        // net electron density (matter term of Eq. 2, lepton density of Eq. 7)
  // constant parts of the Hamiltonians in the traceless components (H_11 - H_22,
  // H_22 - H_33, off-diagonal reals): (H_vacuum + H_matter) / hbar for neutrinos,
  // (H_vacuum^* - H_matter^*) / hbar for antineutrinos
  double vnu[kNC];
  double vnubar[kNC];
  long long vq[2][kNC];  // the same as operands (wide.cuh): vq 2^(ve - kBiasV), one exponent per group
  int ve[2][4];
};

// Warps that share a part of n directions: no more than directions, but all 8 in
// the smallest boxes (parts of less than 6: few blocks), where they only share the
// sum over warps and the RK stage's conversions.
__host__ __device__ inline int part_warps(int n) { return n < 6 || n > kWarps ? kWarps : n; }

// Kernel view of a batch (passed by value).
struct Batch {
  const BoxGeo* box;   // [nbox]
  const double* dt;    // [nbox] step size of every box
  int nbox;
  int nw;              // warps that split the units
  int NZ, MT, NT;      // total cells, directions, tiles
  int T;               // cells per tile (the shape order's Sten<>::T)
  int64_t U, Ptot;     // total units, particles
  int64_t U32;         // total 32-cell units of the RK stage (shape orders 0-2)
  int nw32;            // warps that split them
  int64_t US;          // total tile units of the RK stage's slabs
  int slabs;           // its work split: 1 = ranges of slabs, 0 = parts of one tile
  int upb;             // directions of a part (slabs 0)
  int dpb;             // deposit: directions of a block's part of a tile; 0: ranges of units per warp
};

struct Parts {
  double *z, *ox, *oy, *oz, *N, *Nbar, *rho, *rhobar, *acc, *stage;
};

// ------------------------------------------------------------ device helpers

// The step kernels are launched with programmatic dependent launch: their
// blocks may be scheduled while the previous kernel of the stream drains.  Each
// calls this first, before any memory access: it returns once the previous
// kernel has completed and its writes are visible (at once without one).
__device__ __forceinline__ void griddep_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

__device__ __forceinline__ int wrapc(int j, int nz) {
  int r = j % nz;
  return r < 0 ? r + nz : r;
}

__device__ __forceinline__ int64_t unit_begin(int64_t w, const Batch& B) {
  return w >= B.nw ? B.U : w * B.U / B.nw;
}
__device__ __forceinline__ int64_t warp_of_unit(int64_t x, const Batch& B) { return ((x + 1) * B.nw - 1) / B.U; }
__device__ __forceinline__ int64_t unit32_begin(int64_t w, const Batch& B) {
  return w >= B.nw32 ? B.U32 : w * B.U32 / B.nw32;
}

// Index of the box containing unit u / cell c / particle p / direction d
// (binary search over the boxes' offsets; all arguments are warp-uniform in
// the step kernels).
__device__ __forceinline__ int box_of_unit(const Batch& B, int64_t u) {
  int lo = 0, hi = B.nbox - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (B.box[mid].uoff <= u) lo = mid; else hi = mid - 1;
  }
  return lo;
}
__device__ __forceinline__ int box_of_unit32(const Batch& B, int64_t u) {
  int lo = 0, hi = B.nbox - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (B.box[mid].uoff32 <= u) lo = mid; else hi = mid - 1;
  }
  return lo;
}
__device__ __forceinline__ int box_of_cell(const Batch& B, int c) {
  int lo = 0, hi = B.nbox - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (B.box[mid].coff <= c) lo = mid; else hi = mid - 1;
  }
  return lo;
}
__device__ __forceinline__ int box_of_particle(const Batch& B, int64_t p) {
  int lo = 0, hi = B.nbox - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (B.box[mid].poff <= p) lo = mid; else hi = mid - 1;
  }
  return lo;
}
__device__ __forceinline__ int box_of_direction(const Batch& B, int d) {
  int lo = 0, hi = B.nbox - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (B.box[mid].doff <= d) lo = mid; else hi = mid - 1;
  }
  return lo;
}

// |d| >= 1/2 (or NaN) from the upper word: the FP64 comparison of the lattice
// test, one more instruction of the FP64 pipe, only behind it.
__device__ __forceinline__ bool half_or_more(double d) { return (__double2hiint(d) & 0x7fffffff) >= 0x3fe00000; }

// The error of a particle at the offset d from its cell's centre: none, off its
// site, or no finite position (an infinite one's image reduction is NaN).
__device__ __forceinline__ int site_error(double d) {
  return fabs(d) <= 0.5 + kLatticeTol ? 0 : isnan(d) ? ERR_NONFINITE : ERR_LATTICE;
}

// Shape weights (Sec. 2.2.1) of order ORDER of a particle at (unwrapped)
// position zs whose lattice site is cell h (hp = h + 1/2): the offset
// d = zs/dz - hp, reduced to the nearest periodic image, lies in [-1/2, 1/2),
// and w[s] is the weight of cell h + s - H, the cardinal B-spline of degree
// ORDER at the cell centre's distance:
//   order 0: 1 on cell h;   order 1: -d_+ , 1 - |d|, d_+ on h-1, h, h+1;
//   order 2: 1/2 (1/2 - d)^2, 3/4 - d^2, 1/2 (1/2 + d)^2, written as
//            1/8 + (d^2 -+ d)/2 and 3/4 - d^2;
//   order 3: from the base cell j0 = h (d >= 0) or h - 1 (d < 0) and
//            f = d - (j0 - h) in [0, 1): (1-f)^3/6, 2/3 - f^2 + f^3/2,
//            2/3 - (1-f)^2 + (1-f)^3/2, f^3/6 on cells j0-1 .. j0+2.
// The image reduction is only needed next to the domain ends, so it sits
// behind the lattice test.  Returns 0, ERR_LATTICE if the particle is off its
// site, or ERR_NONFINITE if its position is not finite (then w is not either,
// but for order 0).
template <int ORDER>
__device__ __forceinline__ int shape_weights(double zs, double hp, double inv_dz, double nz_d,
                                             double (&w)[Sten<ORDER>::NW]) {
  double d = fma(zs, inv_dz, -hp);
  int bad = 0;
  if (half_or_more(d) && !(fabs(d) <= 0.5 + kLatticeTol)) {
    d -= nz_d * rint(d / nz_d);
    bad = site_error(d);
  }
  if constexpr (ORDER == 0) {
    w[0] = 0.0; w[1] = 1.0; w[2] = 0.0;
  } else if constexpr (ORDER == 1) {
    w[0] = fmax(-d, 0.0);
    w[1] = 1.0 - fabs(d);
    w[2] = fmax(d, 0.0);
  } else if constexpr (ORDER == 2) {
    const double d2 = d * d;
    w[1] = 0.75 - d2;
    w[0] = fma(0.5, d2 - d, 0.125);
    w[2] = fma(0.5, d2 + d, 0.125);
  } else {
    const bool up = d >= 0.0;
    const double f = up ? d : 1.0 + d, g = 1.0 - f;
    const double a = g * g * g * (1.0 / 6.0);
    const double bb = fma(f * f, fma(0.5, f, -1.0), 2.0 / 3.0);
    const double c = fma(g * g, fma(0.5, g, -1.0), 2.0 / 3.0);
    const double e = f * f * f * (1.0 / 6.0);
    w[0] = up ? 0.0 : a;
    w[1] = up ? a : bb;
    w[2] = up ? bb : c;
    w[3] = up ? c : e;
    w[4] = up ? e : 0.0;
  }
  return bad;
}

// The lattice test of shape_weights alone, for the particle at zs and the cell
// whose centre is hp (in cells), up to the periodic image.
__device__ __forceinline__ int off_site(double zs, double hp, double inv_dz, double nz_d) {
  double d = fma(zs, inv_dz, -hp);
  if (half_or_more(d) && !(fabs(d) <= 0.5 + kLatticeTol)) {
    d -= nz_d * rint(d / nz_d);
    return site_error(d);
  }
  return 0;
}

// Loads of data that a fused step launch (k_step) writes before it reads
// them (positions, stage states, shape weights, grid potential, lattice
// shifts) must not take the read-only (non-coherent) path, which is only
// valid across launches.  COH = true selects a weak global load instead: it
// may hit in L1, which the acquire fence of every grid barrier invalidates,
// so after a barrier it sees what other blocks wrote before it.  The
// separate kernels keep the read-only path (ldd, ldi) or a plain load (ldp).
__device__ __forceinline__ double ld_weak(const double* p) {
  double v;
  asm volatile("ld.global.f64 %0, [%1];" : "=d"(v) : "l"(p));
  return v;
}
__device__ __forceinline__ int ld_weak(const int* p) {
  int v;
  asm volatile("ld.global.s32 %0, [%1];" : "=r"(v) : "l"(p));
  return v;
}
template <bool COH>
__device__ __forceinline__ double ldd(const double* p) {
  if constexpr (COH) return ld_weak(p);
  else return __ldg(p);
}
template <bool COH>
__device__ __forceinline__ int ldi(const int* p) {
  if constexpr (COH) return ld_weak(p);
  else return __ldg(p);
}
template <bool COH>
__device__ __forceinline__ double ldp(const double* p) {
  if constexpr (COH) return ld_weak(p);
  else return *p;
}

// Element k of an array of rows of P doubles, at row pointer p (P < 2^32: the
// address is one IMAD.WIDE; with a 64-bit P each cost about seven
// instructions, a fifth of the RK stage's).
__device__ __forceinline__ const double* row(const double* p, unsigned P, unsigned k) {
  return (const double*)((const char*)p + (uint64_t)P * (8u * k));
}
__device__ __forceinline__ double* row(double* p, unsigned P, unsigned k) {
  return (double*)((char*)p + (uint64_t)P * (8u * k));
}

// Index of this warp among the warps of a persistent grid: warp i of every
// block comes before warp i + 1 of any block.  Units are split into
// contiguous ranges in this order, so when a batch has fewer units than the
// grid has warps the busy warps spread over all blocks, and so over all SMs
// (GB300's FP64 pipe is shared by the four sub-partitions of an SM), instead
// of filling the first blocks.  The split itself, and so every sum, does not
// depend on this numbering.
__device__ __forceinline__ int64_t logical_warp() {
  return (int64_t)(threadIdx.x >> 5) * gridDim.x + blockIdx.x;
}

// The weights kept by the deposit for the RK stage (order 0: 1 on the own cell).
template <int ORDER, bool COH = false>
__device__ __forceinline__ void load_weights(const double* W, int64_t P, int64_t p, double (&w)[Sten<ORDER>::NW]) {
  if constexpr (ORDER == 0) {
    w[0] = 0.0; w[1] = 1.0; w[2] = 0.0;
  } else {
#pragma unroll
    for (int s = 0; s < Sten<ORDER>::NW; ++s) w[s] = ldp<COH>(W + s * P + p);
  }
}

template <int ORDER>
__device__ __forceinline__ void zero_weights(double (&w)[Sten<ORDER>::NW]) {
#pragma unroll
  for (int s = 0; s < Sten<ORDER>::NW; ++s) w[s] = 0.0;
}

// Interpolation through the stencil (Eq. 6): sum over s of w[s] times the
// value v on the lane of cell h + s - H.  Every lane must call it.
template <int ORDER>
__device__ __forceinline__ double gather(const double (&w)[Sten<ORDER>::NW], double v) {
  if constexpr (ORDER == 0) {
    return v;
  } else {
    constexpr int H = Sten<ORDER>::H, NW = Sten<ORDER>::NW;
    double h = w[NW - 1] * __shfl_down_sync(kFull, v, H);
#pragma unroll
    for (int s = NW - 2; s >= 0; --s) {
      const int o = s - H;
      const double x = o > 0 ? __shfl_down_sync(kFull, v, o) : o < 0 ? __shfl_up_sync(kFull, v, -o) : v;
      h = fma(w[s], x, h);
    }
    return h;
  }
}

// Deposit through the stencil (Eq. 5): a lane's cell receives from the
// particle o lanes to its left the weight that particle gives to cell
// (its site + o), and likewise from the right.  init() shuffles the weights
// once per unit; apply(v) returns the sum over those particles of weight x v.
// Every lane must call both.
template <int ORDER>
struct Spread {
  static constexpr int H = Sten<ORDER>::H;
  double w0, fl[H], fr[H];
  __device__ __forceinline__ void init(const double (&w)[Sten<ORDER>::NW]) {
    w0 = w[H];
#pragma unroll
    for (int o = 1; o <= H; ++o) {
      fl[o - 1] = __shfl_up_sync(kFull, w[H + o], o);
      fr[o - 1] = __shfl_down_sync(kFull, w[H - o], o);
    }
  }
  __device__ __forceinline__ double apply(double v) const {
    if constexpr (ORDER == 0) {
      return v;
    } else {
      double c = fr[H - 1] * __shfl_down_sync(kFull, v, H);
#pragma unroll
      for (int o = H - 1; o >= 1; --o) c = fma(fr[o - 1], __shfl_down_sync(kFull, v, o), c);
      c = fma(w0, v, c);
#pragma unroll
      for (int o = 1; o <= H; ++o) c = fma(fl[o - 1], __shfl_up_sync(kFull, v, o), c);
      return c;
    }
  }
};

// Prefetch into L2 by a whole warp: of `narr` arrays (array(a) the first double
// of array a) the doubles [i0, i0 + n), n <= 32.  One lane takes one 128-byte
// line: at most three per array.  (The bulk form, one cp.async.bulk.prefetch per
// array, is a uniform instruction: a warp whose lanes name different arrays
// runs it once per lane, ~17 instructions each; 57 arrays cost a unit of the
// RK stage a quarter of its 3750 instructions.)
__device__ __forceinline__ void prefetch_line(const double* a) {
  asm volatile("prefetch.global.L2 [%0];" ::"l"(a));
}
template <typename F>
__device__ __forceinline__ void prefetch_l2(int lane, int narr, int64_t i0, int n, F array) {
  for (int t = lane; t < 4 * narr; t += kLanes) {
    const int a = t >> 2, q = t & 3;
    if (q < 3) prefetch_line(array(a) + i0 + min(16 * q, n - 1));
  }
}

// Periodic wrap into [0, Lz).
__device__ __forceinline__ double wrap_z(double z, double Lz) {
  if (z >= Lz) z -= Lz;
  else if (z < 0.0) {
    z += Lz;
    if (z >= Lz) z -= Lz;
  }
  return z;
}

// -i [H, r] (Eq. 4 with H in units of hbar) from the operands of wide.cuh.
// Diagonal outputs are returned HALVED (kd = K_aa / 2).  Off-diagonal outputs
// ko = (Re K12, Im K12, Re K13, Im K13, Re K23, Im K23).
__device__ __forceinline__ void commutator(const emu_wide::Ham& H, const emu_wide::Mat& m, double (&kd)[3],
                                           double (&ko)[6]) {
  namespace w = emu_wide;
  // (exponents from the smallest normal results up; out of range: NaN)
  constexpr int emin = w::kBiasP - 1022;
  auto value = [](double v, int e) { return e - w::kBiasP > 959 ? nan("") : w::scale_nz(v, e - w::kBiasP); };
  const bool inf = w::max_i(w::top(H), w::top(m)) >= w::kExpNonFinite;
  const int e0 = inf ? 1 << 16 : emin;
  double cr, ci;
  int e, ke[3];
  // C = [H, r]; K = -i C  =>  Re K = Im C, Im K = -Re C
  w::commutator_off<0>(H, m, e0, cr, ci, e);
  ko[0] = value(ci, e);
  ko[1] = -value(cr, e);
  w::commutator_off<1>(H, m, e0, cr, ci, e);
  ko[2] = value(ci, e);
  ko[3] = -value(cr, e);
  w::commutator_off<2>(H, m, e0, cr, ci, e);
  ko[4] = value(ci, e);
  ko[5] = -value(cr, e);
  w::commutator_diag(H, m, e0, kd, ke);
#pragma unroll
  for (int k = 0; k < 3; ++k) kd[k] = value(kd[k], ke[k]);
}

// ------------------------------------------------------------------ kernels
//
// Every step kernel is a thin wrapper around a *phase*: the work of one warp
// (deposit, RK stage) or of one block (deposit combination, lattice shifts) in
// a persistent grid.  The separate kernels run one phase per launch; the fused
// step kernel (k_step) runs all phases of a step in one cooperative launch
// with grid barriers between them.  COH = true marks the fused form, whose
// loads of data written earlier in the same launch take the coherent path.

// Per-direction table from each ring's first particle: Omega and v_z = c Omega_z
// ([4][MT]); also checks that every particle of a ring carries its direction.
static __global__ void k_dirtable(Batch B, Parts pt, double* __restrict__ dirtab, int* __restrict__ err) {
  const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= B.Ptot) return;
  const BoxGeo& g = B.box[box_of_particle(B, p)];
  const int d = (int)((p - g.poff) / g.nz);
  const int64_t p0 = g.poff + (int64_t)d * g.nz;
  const double ox = pt.ox[p0], oy = pt.oy[p0], oz = pt.oz[p0];
  if (pt.ox[p] != ox || pt.oy[p] != oy || pt.oz[p] != oz) atomicOr(err, ERR_RING);
  if (p == p0) {
    const int gd = g.doff + d;
    dirtab[gd] = ox;
    dirtab[B.MT + gd] = oy;
    dirtab[2 * B.MT + gd] = oz;
    dirtab[3 * B.MT + gd] = g.c_light * oz;
  }
}

// Lattice shift of every direction for up to 4 position offsets frac[s] * dt_b:
// the cell of the ring's first particle at z + frac[s] dt_b v_z ([nrows][MT]).
// A fifth row (nrows = 5) holds the shift of the next step's first stage: the
// cell of wrap(z + dt_b v_z), the position stage 4 writes, computed exactly as
// the RK stage computes it.  Beside each shift row the ring's shape weights
// (the direction weight table, kWSlots per row): a ring translates rigidly, so
// all its particles sit at its first particle's offset inside their cells.
struct Fracs { double v[4]; };

// Position offset of RK stage s (0-based), in units of dt (Sec. 2.3, classic tableau).
__device__ __forceinline__ double stage_frac(int s) { return s == 0 ? 0.0 : s == 3 ? 1.0 : 0.5; }

__device__ __forceinline__ int lattice_cell(double z0, double frac_dt, double vz, const BoxGeo& g) {
  const double zs = fma(frac_dt, vz, z0);
  return wrapc((int)floor(zs * g.inv_dz), g.nz);
}

// Row `row` of the tables for direction gd: the shift (the cell of the ring's
// first particle at its row position) and, with wtab, that particle's shape
// weights there.  Rows 0-3: z + frac[row] dt_b v_z; row 4: wrap(z + dt_b v_z).
template <bool COH, int ORDER>
__device__ __forceinline__ void shifts_row(const Batch& B, int gd, const double* z, const double* __restrict__ dirtab,
                                           const Fracs& fr, int row, int* shift, double* wtab) {
  const int b = box_of_direction(B, gd);
  const BoxGeo& g = B.box[b];
  const double z0 = ldp<COH>(z + g.poff + (int64_t)(gd - g.doff) * g.nz);
  const double vz = dirtab[3 * B.MT + gd];
  const double dt = B.dt[b];
  const double zs = row < 4 ? fma(fr.v[row] * dt, vz, z0) : wrap_z(fma(dt, vz, z0), g.Lz);
  const int cell = lattice_cell(zs, 0.0, vz, g);
  shift[row * B.MT + gd] = cell;
  if (wtab != nullptr) {   // the ring's weights: its first particle's, at the cell the shift assigns it
    double w[Sten<ORDER>::NW];
    (void)shape_weights<ORDER>(zs, (double)cell + 0.5, g.inv_dz, g.nz_d, w);
#pragma unroll
    for (int q = 0; q < Sten<ORDER>::NWS; ++q) wtab[(row * kWSlots + q) * B.MT + gd] = w[q];
  }
}

template <bool COH, int ORDER>
__device__ __forceinline__ void shifts_phase(const Batch& B, int gd, const double* z, const double* __restrict__ dirtab,
                                             const Fracs& fr, int nrows, int* shift, double* wtab) {
  if (gd >= B.MT) return;
  for (int row = 0; row < nrows && row < 5; ++row) shifts_row<COH, ORDER>(B, gd, z, dirtab, fr, row, shift, wtab);
}

// One thread per (direction, row): the rows' chains run side by side.
template <int ORDER>
__global__ void k_shifts(Batch B, const double* __restrict__ z, const double* __restrict__ dirtab, Fracs fr,
                         int nrows, int* __restrict__ shift, double* __restrict__ wtab) {
  griddep_wait();
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  const int row = t / B.MT, gd = t - row * B.MT;
  if (row >= nrows) return;
  shifts_row<false, ORDER>(B, gd, z, dirtab, fr, row, shift, wtab);
}

// A warp's sums for one tile go to slot (warp + global tile) of the partial
// buffer: unique, because a later warp never returns to an earlier tile.
template <int ORDER, int NA>
__device__ __forceinline__ void flush_tile(const double (&acc)[NA], int64_t gtile, int local_cell, int nz,
                                           int64_t w, int lane, double* __restrict__ partial) {
  constexpr int H = Sten<ORDER>::H, T = Sten<ORDER>::T;
  if (lane >= H && lane < H + T && local_cell < nz) {
    double* slot = partial + (w + gtile) * kSlot + lane - H;
#pragma unroll
    for (int c = 0; c < NA; ++c) slot[c * T] = acc[c];
  }
}

// A value of lane `src` as limbs in every lane.
__device__ __forceinline__ emu_wide::Limbs bcast(emu_wide::Limbs v, int src) {
  return emu_wide::Limbs{__shfl_sync(kFull, v.h, src), __shfl_sync(kFull, v.l, src)};
}
// Limbs of the lane o to the left (o > 0) or right (o < 0).
__device__ __forceinline__ emu_wide::Limbs from_lane(emu_wide::Limbs v, int o) {
  return o > 0 ? emu_wide::Limbs{__shfl_up_sync(kFull, v.h, o), __shfl_up_sync(kFull, v.l, o)}
               : emu_wide::Limbs{__shfl_down_sync(kFull, v.h, -o), __shfl_down_sync(kFull, v.l, -o)};
}
__device__ __forceinline__ int from_lane(int v, int o) {
  return o > 0 ? __shfl_up_sync(kFull, v, o) : __shfl_down_sync(kFull, v, -o);
}

// Limbs of u in every lane: a direction's components in lanes 0-2, there scaled by
// 2^-ko (direction_excess), other numbers up to 1 in the rest (one that is not
// finite counts as an infinite direction).
__device__ __forceinline__ emu_wide::Limbs direction_limbs(double u, int lane, int& ko) {
  emu_wide::Limbs l = emu_wide::unit_limbs(u);
  ko = 0;
  const int m = emu_wide::unit_magnitude(u);
  if (__reduce_add_sync(kFull, lane < 3 || m > emu_wide::kDotLimit ? m : 0) > emu_wide::kDotLimit) {
    ko = max(__reduce_max_sync(kFull, emu_wide::unit_excess(u)), 1);
    if (lane < 3) l = emu_wide::unit_limbs(u, ko);
  }
  return l;
}

// Asynchronous copies of 8 bytes from global to shared memory, by the thread
// that reads them: its copies of all but the last N groups are done after
// cp_async_wait<N>.
__device__ __forceinline__ void cp_async8(double* dst, const double* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src)
               : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}
constexpr int kDepRows = 21;   // doubles of a particle a deposit reads
constexpr int kDepBuf = 2 * kDepRows * kLanes;                                // of one warp's buffers
constexpr int kDepSmem = kWarps * kDepBuf * (int)sizeof(double);              // 86 KB a block

// What a deposit of mode MODE (deposit_phase) sums: SETS fields of COMP
// components with MOM moments each (row (set * MOM + m) * COMP + c), and which
// of a particle's arrays it reads.
template <int MODE>
struct DepMode {
  static constexpr int SETS = MODE == 4 ? 2 : 1, MOM = MODE == 4 ? 2 : 4, COMP = MODE == 5 ? kNC : 9;
  static constexpr int NA = SETS * MOM * COMP;
  static constexpr bool N1 = MODE != 2 && MODE != 3, N2 = MODE != 1 && MODE != 3, RNU = MODE != 2,
                        RNB = MODE != 1 && MODE != 3;
  // components that share the exponent of their sums: single diagonal entries (or
  // their differences), then the real and imaginary part of an off-diagonal
  static constexpr int SINGLE = MODE == 5 ? 2 : 3, GROUPS = SINGLE + 3;
};

// The direction loop of the deposit for one tile: warp lane `lane` of a tile
// of box b (lane l owns cell tile * T - H + l) adds the rings dfirst..dlast-1
// of the tile, in a fixed order, in acc (MODES as deposit_phase), on the integer pipe.
// B is formed in FP64 (20 instructions a particle, against 85-100 for a deposit
// with FP64 sums: at 16 cycles each the FP64 pipe bound it); its spread over the
// stencil and the moments' sums are fixed-point (wide.cuh).  A sum is an
// int64 per lane; the components of one group share the exponent ea of
// their sums, which grows when a direction's contribution asks for it (the
// sums are then shifted).  Sums of n directions have headroom for n contributions
// and round them without a bias (sum_headroom): less error than FP64 sums, whose
// rounding follows the partial sums.  Zero contributions add exactly nothing.
// Bound by latency at four warps a scheduler (issue slots 48 %, FP64 pipe 58 %
// busy): 16384 x 1000 2467 -> 1050 us a stage against FP64 sums (1256 with plain
// loads: cp.async hides their latency), 1024 x 378 74 -> 41 us.
// (buf: this warp's two buffers of kDepRows x 32 doubles in shared memory;
// ring2 0: only one, when no warp takes more than one direction of a tile.)
// phase > 0: the directions in cyclic order from the first multiple of phase (a
// warp's share), so that the warps of neighbouring tiles read the same ring at the
// same time: a tile's 256-byte rows start anywhere in a 128-byte line, and lines
// shared with the neighbours came from DRAM twice (268 bytes a particle for 168;
// 16384 x 1000 1067 -> 1038 us).
template <int MODE, int ORDER, bool COH>
__device__ __forceinline__ void deposit_tile(const Batch& B, int b, int tile, int dfirst, int dlast, int lane,
                                                  const double* z, const double* __restrict__ N,
                                                  const double* __restrict__ Nbar, const double* r_nu,
                                                  const double* r_nb, const double* __restrict__ dirtab,
                                                  const int* shift, const double* wrow, double frac, double* W,
                                                  double* buf, int ring2, int phase,
                                                  int64_t (&acc)[DepMode<MODE>::NA],
                                                  int (&ea)[DepMode<MODE>::SETS * DepMode<MODE>::GROUPS], int& bad) {
  namespace w = emu_wide;
  constexpr int H = Sten<ORDER>::H, T = Sten<ORDER>::T, NW = Sten<ORDER>::NW;
  using D = DepMode<MODE>;
  const BoxGeo& g = B.box[b];
  const int nz = g.nz;
  const unsigned P = (unsigned)B.Ptot;
  const int MT = B.MT;
  const int craw = tile * T - H + lane;
  const int j = wrapc(craw, nz);
  const double hp = (double)j + 0.5;
  const bool own = lane >= H && lane < H + T && craw < nz;
  const double pos_dt = frac * B.dt[b];
  const int dbase = g.doff;
  const int head = w::sum_headroom(dlast - dfirst);
#pragma unroll
  for (int c = 0; c < D::NA; ++c) acc[c] = 0;
#pragma unroll
  for (int q = 0; q < D::SETS * D::GROUPS; ++q) ea[q] = 0;
  // direction d's particle data into buffer d & 1, asynchronously (each lane
  // its own particle's: no exchange between lanes): z, N, Nbar, rho, rhobar
  auto fetch = [&](int d, int k) -> int64_t {
    int i = j - ldi<COH>(shift + dbase + d);
    if (i < 0) i += nz;
    const int64_t p = g.poff + (int64_t)d * nz + i;
    double* dst = buf + (k & ring2) * kDepRows * kLanes + lane;
    cp_async8(dst, z + p);
    if (D::N1) cp_async8(dst + kLanes, N + p);
    if (D::N2) cp_async8(dst + 2 * kLanes, Nbar + p);
#pragma unroll
    for (int k = 0; k < 9; ++k) {
      if (D::RNU) cp_async8(dst + (3 + k) * kLanes, row(r_nu + p, P, k));
      if (D::RNB) cp_async8(dst + (12 + k) * kLanes, row(r_nb + p, P, k));
    }
    cp_async_commit();
    return p;
  };
  const int n = dlast - dfirst;
  int dnext = dfirst;
  if (phase > 0) {   // (no multiple of it among the directions: from dfirst)
    const int o = (phase - dfirst % phase) % phase;
    if (o < n) dnext += o;
  }
  int64_t pnext = fetch(dnext, 0);
  for (int k = 0; k < n; ++k) {
    const int d = dnext;
    dnext = d + 1 < dlast ? d + 1 : dfirst;
    const int gd = dbase + d;
    const int64_t p = pnext;
    if (k + 1 < n && ring2) {
      pnext = fetch(dnext, k + 1);
      cp_async_wait<1>();
    } else {
      cp_async_wait<0>();
    }
    double* x = buf + (k & ring2) * kDepRows * kLanes + lane;
    // Omega, and the ring's weights when every particle takes them: lane q
    // converts one of them
    double u = 0.0;
    if (lane < 3) u = __ldg(dirtab + lane * MT + gd);
    const double zs = fma(pos_dt, __ldg(dirtab + 3 * MT + gd), x[0]);
    double wt[NW];
    int site;          // the lattice test's error
    if (wrow != nullptr) {
      if (ORDER > 0 && lane >= 3 && lane < 3 + NW) u = ldp<COH>(wrow + (lane - 3) * MT + gd);
      site = off_site(zs, hp, __ldg(&g.inv_dz), __ldg(&g.nz_d));
    } else {
      site = shape_weights<ORDER>(zs, hp, __ldg(&g.inv_dz), __ldg(&g.nz_d), wt);
      if ((MODE == 0 || MODE == 5) && W != nullptr && own) {   // the RK stage of these positions reads them back
#pragma unroll
        for (int q = 0; q < Sten<ORDER>::NWS; ++q) *row(W + p, P, q) = wt[q];
      }
    }
    // weights have no exponent: a particle without a finite position counts as
    // one of infinite B, a ring without finite weights as an infinite direction
    if (site != 0) {
      bad |= site;
      if (site & ERR_NONFINITE) {
#pragma unroll 1
        for (int q = 1; q < kDepRows; ++q) x[q * kLanes] = nan("");
      }
    }
    const double n1 = D::N1 ? x[kLanes] : 0.0, n2 = D::N2 ? x[2 * kLanes] : 0.0;
    // component k of the deposited matrix (conj(rhobar) flips the sign of the
    // imaginary components 4, 6, 8)
    auto value = [&](int set, int k) -> double {
      const bool im = k == 4 || k == 6 || k == 8;
      const double a = D::RNU ? x[(3 + k) * kLanes] : 0.0, c = D::RNB ? x[(12 + k) * kLanes] : 0.0;
      if (MODE == 3) return a;
      if (MODE == 1 || (MODE == 4 && set == 0)) return n1 * a;
      if (MODE == 2 || MODE == 4) return n2 * c;
      return fma(im ? n2 : -n2, c, n1 * a);
    };
    w::Limbs wl[NW];   // the weight slot o of the particle that gives it to this lane's cell
    // directions above 1 (not unit vectors) are scaled by 2^-ko
    const int ko = __reduce_max_sync(kFull, w::unit_excess(u)), half = w::sum_half(ko);
    const w::Limbs ul = w::unit_limbs(u, lane < 3 ? ko : 0);
    const w::Factor uf = w::factor(w::join(ul));
    w::Factor om[3];
    int64_t mh[3];   // (order 3 has no registers left for them: it adds the half unit as one every second term)
#pragma unroll
    for (int m = 0; m < 3; ++m) {
      om[m] = w::Factor{__shfl_sync(kFull, uf.h, m), __shfl_sync(kFull, uf.l, m)};
      mh[m] = w::moment_half(om[m]);
    }
    if constexpr (ORDER > 0) {
      if (wrow != nullptr) {
        if ((MODE == 0 || MODE == 5) && W != nullptr && own) {
#pragma unroll
          for (int q = 0; q < NW; ++q) *row(W + p, P, q) = ldp<COH>(wrow + q * MT + gd);
        }
#pragma unroll
        for (int o = 0; o < NW; ++o) wl[o] = bcast(ul, 3 + o);
      } else {
#pragma unroll
        for (int o = 0; o < NW; ++o) {   // from the lane o - H to the left
          wl[o] = w::unit_limbs(wt[o]);
          if (o != H) wl[o] = from_lane(wl[o], o - H);
        }
      }
    }
    double bprev = MODE == 5 ? value(0, 0) : 0.0;   // B of the previous diagonal entry
#pragma unroll
    for (int sq = 0; sq < D::SETS * D::GROUPS; ++sq) {
      const int set = sq / D::GROUPS, q = sq % D::GROUPS, nc = q < D::SINGLE ? 1 : 2;
      const int c0 = q < D::SINGLE ? q : 2 * q - D::SINGLE;   // the group's components c0 .. c0 + nc - 1
      const int r0 = set * D::MOM * D::COMP + c0;             // and the row of its first sum
      double bv[2] = {0.0, 0.0};
      if (MODE == 5 && nc == 1) {
        const double bn = value(0, q + 1);
        bv[0] = bprev - bn;
        bprev = bn;
      } else {
        const int k = c0 + (MODE == 5 ? 1 : 0);
        bv[0] = value(set, k);
        if (nc > 1) bv[1] = value(set, k + 1);
      }
      const int e0 = w::exponent(bv[0]), e1 = nc > 1 ? w::exponent(bv[1]) : 0, e = max(e0, e1);
      w::Limbs bl[2];
      bl[0] = nc > 1 ? w::limbs(bv[0], e0, e) : w::limbs(bv[0], e);
      if (nc > 1) bl[1] = w::limbs(bv[1], e1, e);
      // the spread (Eq. 5): taps at the largest exponent of the contributing particles
      int64_t cv[2];
      int et = e;
      if constexpr (ORDER == 0) {
        for (int c = 0; c < nc; ++c) cv[c] = w::join(bl[c]) >> 2;
      } else {
        int en[NW];
#pragma unroll
        for (int o = 0; o < NW; ++o) {
          en[o] = o == H ? e : from_lane(e, o - H);
          et = max(et, en[o]);
        }
        for (int c = 0; c < nc; ++c) cv[c] = 0;
#pragma unroll
        for (int o = 0; o < NW; ++o) {
          const int dd = et - en[o], df = max(dd - 32, 0);
#pragma unroll
          for (int c = 0; c < nc; ++c) {
            const w::Limbs v = o == H ? bl[c] : from_lane(bl[c], o - H);
            cv[c] += w::align(w::mul(v, wl[o]), dd, df);
          }
        }
      }
      // the sums' exponent
      const int es = ko <= w::kMaxExcess ? et + ko : w::kExpNonFinite;
      if (es + head > ea[sq]) {
        const int sh = es + head - ea[sq], sf = max(sh - 32, 0);
        ea[sq] += sh;
#pragma unroll
        for (int c = 0; c < nc; ++c) {
#pragma unroll
          for (int m = 0; m < D::MOM; ++m) acc[m * D::COMP + r0 + c] = w::align(acc[m * D::COMP + r0 + c], sh, sf);
        }
      }
      const int dd = ea[sq] - es, df = max(dd - 32, 0);
#pragma unroll
      for (int c = 0; c < nc; ++c) {
        const int64_t v = w::align(cv[c], dd, df);
        const w::Factor f = w::factor(ORDER == 3 ? v + (k & 1) : v);
        acc[r0 + c] += w::zeroth_moment(v, ko, half);
#pragma unroll
        for (int m = 1; m < D::MOM; ++m)
          acc[m * D::COMP + r0 + c] = w::moment_add(f, om[m - 1], ORDER == 3 ? w::half_unit() : mh[m - 1], acc[m * D::COMP + r0 + c]);
      }
    }
  }
}

// Exponents of sums that are not finite, lie at an end of the range of doubles or are
// zero (the smallest).
__device__ __forceinline__ bool far_exponent(int ea) { return (unsigned)(ea - 64) > 1966u; }
// A sum acc 2^(ea + 4 - kBiasV) of deposit_tile as a double.
__device__ __forceinline__ double deposit_sum(int64_t acc, int ea) {
  namespace w = emu_wide;
  if (far_exponent(ea) && (acc != 0 || ea >= w::kExpNonFinite))
    return ea >= w::kExpNonFinite ? nan("") : w::scaled(acc, ea + 4 - w::kBiasV);
  return w::scaled_near(acc, ea + 4 - w::kBiasV);
}
// The exponent group of row c.
template <int MODE>
__device__ __forceinline__ constexpr int deposit_group(int c) {
  using D = DepMode<MODE>;
  const int k = c % D::COMP, q = k < D::SINGLE ? k : D::SINGLE + (k - D::SINGLE) / 2;
  return c / (D::MOM * D::COMP) * D::GROUPS + q;
}

// deposit_sum of a tile's sums, with one branch for all of them.
template <int MODE>
__device__ __forceinline__ void deposit_sums(const int64_t (&sum)[DepMode<MODE>::NA],
                                             const int (&ea)[DepMode<MODE>::SETS * DepMode<MODE>::GROUPS],
                                             double (&acc)[DepMode<MODE>::NA]) {
  namespace w = emu_wide;
  using D = DepMode<MODE>;
  int64_t far = 0;
#pragma unroll
  for (int q = 0; q < D::SETS * D::GROUPS; ++q) {
    if (far_exponent(ea[q])) {
      far |= ea[q] >= w::kExpNonFinite;
#pragma unroll
      for (int c = 0; c < D::NA; ++c)
        if (deposit_group<MODE>(c) == q) far |= sum[c];
    }
  }
#pragma unroll
  for (int c = 0; c < D::NA; ++c)
    acc[c] = w::scaled_near(sum[c], w::near(ea[deposit_group<MODE>(c)] + 4 - w::kBiasV));
  if (far != 0) {
#pragma unroll
    for (int c = 0; c < D::NA; ++c) {
      const int e = ea[deposit_group<MODE>(c)];
      acc[c] = e >= w::kExpNonFinite ? nan("") : acc[c] * w::far_factor(e + 4 - w::kBiasV);
    }
  }
}

// Where a part's warp keeps the exponents of its sums (deposit_phase), in 32-bit
// words: two a row, in the 8-byte column of their lane.  The warp's buffer still
// holds particle data there, and each lane reads and writes its own column only:
// no lane's store can pass another's reads.
__host__ __device__ constexpr int part_exponent(int c, int lane) { return 2 * ((c >> 1) * kLanes + lane) + (c & 1); }
__host__ __device__ constexpr bool part_exponents_in_column(int groups) {
  for (int c = 0; c < groups; ++c)
    for (int lane = 0; lane < kLanes; ++lane)
      if (part_exponent(c, lane) / 2 % kLanes != lane) return false;
  return true;
}

// Part q of the deposit's split into blocks (Batch::dpb > 0): box b, tile and
// directions [d0, d1); false past the last one.  first_part: the first part of a tile.
__device__ __forceinline__ bool deposit_part(const Batch& B, int q, int& b, int& tile, int& d0, int& d1) {
  for (b = 0; b < B.nbox; ++b) {
    const BoxGeo& g = B.box[b];
    const int per = (g.M + B.dpb - 1) / B.dpb, all = per * g.ntiles;
    if (q < all) {
      tile = q / per;
      const int i = q - tile * per, len = g.M / per, more = g.M - len * per;   // (the first `more` parts take one more)
      d0 = i * len + min(i, more);
      d1 = d0 + len + (i < more);
      return true;
    }
    q -= all;
  }
  return false;
}
__device__ __forceinline__ int first_part(const Batch& B, const BoxGeo* box, int tile) {
  int q = 0;
  for (const BoxGeo* g = B.box; g < box; ++g) q += (g->M + B.dpb - 1) / B.dpb * g->ntiles;
  return q + tile * ((box->M + B.dpb - 1) / B.dpb);
}

// Deposit (Eq. 5), first phase.  MODE 0: B = N rho - Nbar rhobar^* (the
// combination that enters H, Eq. 2); MODE 1: B = N rho; MODE 2: B = Nbar rhobar;
// MODE 3: B = r_nu (packed matrices given per particle: the adjoint's Gamma);
// MODE 4: the moments the diagnostics read (Eq. 10), both species in one
// pass: rows 0-8 n, 9-17 f_x (from N rho), 18-26 nbar, 27-35 fbar_x (Nbar rhobar);
// MODE 5: MODE 0's B in the traceless components the step reads (kNT rows:
// moment m, component c at row m * kNC + c; c = 0, 1 the diagonal differences
// B_11 - B_22 and B_22 - B_33, c = 2..7 the off-diagonal reals 3..8).
// Warp w walks its units in order (box, tile, direction), summing
// w_pj (1, Omega_p) B_p over directions in registers (lane l owns cell
// tile * T - H + l) and writing one partial per tile it touches; MODES 0 and 5
// also store every particle's weights for the RK stage.  Positions: z + frac dt_b v_z.
// With wrow (the stage's row of the direction weight table k_shifts writes)
// every particle of a ring takes the ring's weights: the ring translates
// rigidly, so its particles share their offset inside the cells (to
// rounding); each particle's position is still checked against its cell.
template <int MODE, int ORDER, bool COH, bool PART>
__device__ __forceinline__ void deposit_phase(const Batch& B, int64_t w, int lane, const double* z,
                                              const double* __restrict__ N, const double* __restrict__ Nbar,
                                              const double* r_nu, const double* r_nb,
                                              const double* __restrict__ dirtab, const int* shift,
                                              const double* wrow, double frac, double* __restrict__ partial,
                                              double* W, int* err, double* buf = nullptr) {
  using D = DepMode<MODE>;
  constexpr int H = Sten<ORDER>::H, T = Sten<ORDER>::T;
  int bad = 0;
  if constexpr (PART) {
    // few units: a block takes a part of one tile's directions, adds its warps'
    // sums (as integers, rounded at their largest exponent: a warp's sum has
    // headroom for its own directions only) and writes one partial
    const int wib = threadIdx.x >> 5;
    const int nwarps = part_warps(B.dpb);                         // (the block's, but in k_step)
    int64_t* sums = (int64_t*)(buf - wib * kDepBuf);              // [warp][row][lane], then the exponents
    constexpr int kE = D::NA * kLanes;                            // doubles before a warp's exponents
    constexpr int NE = D::SETS * D::GROUPS;
    static_assert(D::NA + (NE + 1) / 2 <= kDepBuf / kLanes, "a warp's sums fit its buffers");
    static_assert(part_exponents_in_column(NE), "a lane's exponents lie in its own column");
    int b, tile, d0, d1;
    for (int q = blockIdx.x; deposit_part(B, q, b, tile, d0, d1); q += gridDim.x) {
      const int n = d1 - d0, used = min(n, nwarps);
      if (wib < used) {
        const int len = n / nwarps, more = n - len * nwarps;
        const int w0 = d0 + wib * len + min(wib, more);
        int64_t acc[D::NA];
        int ea[D::SETS * D::GROUPS];
        deposit_tile<MODE, ORDER, COH>(B, b, tile, w0, w0 + len + (wib < more), lane, z, N, Nbar, r_nu, r_nb, dirtab, shift,
                                       wrow, frac, W, buf, 1, 0, acc, ea, bad);
#pragma unroll
        for (int c = 0; c < D::NA; ++c) sums[wib * kDepBuf + c * kLanes + lane] = acc[c];
#pragma unroll
        for (int c = 0; c < NE; ++c) ((int*)(sums + wib * kDepBuf + kE))[part_exponent(c, lane)] = ea[c];
      }
      __syncthreads();
      const int cell = tile * T - H + lane;
      if (wib < nwarps && lane >= H && lane < H + T && cell < B.box[b].nz) {
        for (int c = wib; c < D::NA; c += nwarps) {
          const int* ex = (const int*)(sums + kE) + part_exponent(deposit_group<MODE>(c), lane);
          int top = 0, e[kWarps];
#pragma unroll
          for (int x = 0; x < kWarps; ++x) top = max(top, e[x] = x < used ? ex[x * 2 * kDepBuf] : 0);
          top += 3;   // headroom for 8 warps
          int64_t v = 0;
#pragma unroll
          for (int x = 0; x < kWarps; ++x)
            if (x < used) v += emu_wide::align_round(sums[x * kDepBuf + c * kLanes + lane], top - e[x]);
          partial[(int64_t)q * kSlot + c * T + lane - H] = deposit_sum(v, top);
        }
      }
      __syncthreads();   // (the sums are free for the next part)
    }
    if (bad) atomicOr(err, bad);
    return;
  }
  const int64_t u0 = unit_begin(w, B), u1 = unit_begin(w + 1, B);
  if (u0 >= u1) return;
  const int phase = (int)((B.U + B.nw - 1) / B.nw);
  int b = box_of_unit(B, u0);
  for (int64_t u = u0; u < u1;) {        // one segment per (box, tile) the warp touches
    while (u >= B.box[b].uoff + (int64_t)B.box[b].ntiles * B.box[b].M) ++b;
    const BoxGeo& g = B.box[b];
    const int M = g.M;
    const int tile = (int)((u - g.uoff) / M);
    const int64_t uend = min(u1, g.uoff + (int64_t)(tile + 1) * M);
    const int64_t ubase = g.uoff + (int64_t)tile * M;
    const int dfirst = (int)(u - ubase), dlast = (int)(uend - ubase);
    u = uend;
    int64_t sum[D::NA];
    int ea[D::SETS * D::GROUPS];
    deposit_tile<MODE, ORDER, COH>(B, b, tile, dfirst, dlast, lane, z, N, Nbar, r_nu, r_nb, dirtab, shift, wrow, frac, W,
                                   buf, B.U > B.nw, phase, sum, ea, bad);
    double acc[D::NA];
    deposit_sums<MODE>(sum, ea, acc);
    flush_tile<ORDER>(acc, g.toff + tile, tile * T - H + lane, g.nz, w, lane, partial);
  }
  if (bad) atomicOr(err, bad);
}

// TAB: the rings' weights from the weight row wrow; otherwise each
// particle's own (wrow unused, and the table's code compiled out).
template <int MODE, int ORDER, bool TAB, bool PART>
__global__ void __launch_bounds__(kThreads, 2)
k_deposit(Batch B, const double* __restrict__ z, const double* __restrict__ N, const double* __restrict__ Nbar,
          const double* __restrict__ r_nu, const double* __restrict__ r_nb, const double* __restrict__ dirtab,
          const int* __restrict__ shift, const double* __restrict__ wrow, double frac, double* __restrict__ partial,
          double* __restrict__ W, int* __restrict__ err) {
  extern __shared__ double dep_sm[];   // kDepSmem bytes (half with one buffer)
  griddep_wait();
  deposit_phase<MODE, ORDER, false, PART>(B, logical_warp(), threadIdx.x & 31, z, N, Nbar, r_nu, r_nb, dirtab, shift,
                                    TAB ? wrow : nullptr, frac, partial, W, err, dep_sm + (threadIdx.x >> 5) * (PART || B.U > B.nw ? kDepBuf : kDepBuf / 2));
}

// ------------------------------------------------------- cluster deposit
//
// The step's deposit (MODE 5) by thread-block clusters of CL blocks (8 or 16),
// with no separate combination: cluster c takes the tiles c, c + clusters,
// ... (all boxes' tiles in order).  For each tile the cluster's W =
// CL x kWarps warps split its rings (warp i: rings [i M / W,
// (i + 1) M / W), summed in order in registers as in deposit_phase); the
// warps of each block are added in warp order through shared memory, then the
// blocks in rank order through distributed shared memory, and the potential
// of the tile's cells is written.  The summation order depends only on the
// box and the cluster size, not on the grid: results are bitwise reproducible.
// All blocks of a cluster walk the same tiles, so every block reaches every
// cluster barrier (hardware barriers, as __syncthreads: no spin on memory).
static_assert(kDepBuf >= kNT * kLanes, "a warp's sums of a tile fit its buffers");

__device__ __forceinline__ unsigned cluster_rank() {
  unsigned r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ unsigned cluster_index() {
  unsigned r;
  asm volatile("mov.u32 %0, %%clusterid.x;" : "=r"(r));
  return r;
}
__device__ __forceinline__ unsigned cluster_count() {
  unsigned r;
  asm volatile("mov.u32 %0, %%nclusterid.x;" : "=r"(r));
  return r;
}
// Barrier of all threads of the cluster; shared-memory writes before it are
// visible to every block of the cluster after it.  (The non-.aligned form:
// correct whether or not the threads of a warp arrive together.)
__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
}
// The double at this block's shared address a, read from block `rank` of the cluster.
__device__ __forceinline__ double ld_cluster(const double* a, unsigned rank) {
  const unsigned local = (unsigned)__cvta_generic_to_shared(a);
  unsigned remote;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(remote) : "r"(local), "r"(rank));
  double v;
  asm volatile("ld.shared::cluster.f64 %0, [%1];" : "=d"(v) : "r"(remote) : "memory");
  return v;
}

__device__ __forceinline__ int box_of_tile(const Batch& B, int64_t t) {
  int lo = 0, hi = B.nbox - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (B.box[mid].toff <= t) lo = mid; else hi = mid - 1;
  }
  return lo;
}

// out: the potential ([kNT][NZ], scale kappa / dV of each box); W as k_deposit.
template <int ORDER, bool TAB, int CL>
__global__ void __launch_bounds__(kThreads, 2)
k_deposit_cluster(Batch B, const double* __restrict__ z, const double* __restrict__ N,
                  const double* __restrict__ Nbar, const double* __restrict__ r_nu, const double* __restrict__ r_nb,
                  const double* __restrict__ dirtab, const int* __restrict__ shift, const double* __restrict__ wrow,
                  double frac, double* __restrict__ out, double* __restrict__ W, int* __restrict__ err) {
  griddep_wait();
  // each warp's particle data, then its sums of the tile ([kNT][kLanes])
  extern __shared__ double red[];
  constexpr int H = Sten<ORDER>::H, T = Sten<ORDER>::T;
  constexpr int NE = kNT * kLanes, per = NE / CL, nwc = CL * kWarps;
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
  const unsigned rank = cluster_rank();
  const int gw = (int)rank * kWarps + wib;
  int bad = 0, nonfinite = 0;
  for (int64_t gt = cluster_index(); gt < B.NT; gt += cluster_count()) {
    const int b = box_of_tile(B, gt);
    const BoxGeo& g = B.box[b];
    const int tile = (int)(gt - g.toff);
    const int d0 = (int)((int64_t)gw * g.M / nwc), d1 = (int)((int64_t)(gw + 1) * g.M / nwc);
    int64_t acc[kNT];
    int ea[DepMode<5>::GROUPS];
#pragma unroll
    for (int c = 0; c < kNT; ++c) acc[c] = 0;
#pragma unroll
    for (int c = 0; c < DepMode<5>::GROUPS; ++c) ea[c] = 0;
    if (d0 < d1)
      deposit_tile<5, ORDER, false>(B, b, tile, d0, d1, lane, z, N, Nbar, r_nu, r_nb, dirtab, shift,
                                    TAB ? wrow : nullptr, frac, W, red + wib * kDepBuf, 1, 0, acc, ea, bad);
    double sum[kNT];
    deposit_sums<5>(acc, ea, sum);
#pragma unroll
    for (int c = 0; c < kNT; ++c) red[wib * kDepBuf + c * kLanes + lane] = sum[c];
    __syncthreads();
    for (int e = threadIdx.x; e < NE; e += kThreads) {   // the block's warps, in warp order
      double v = red[e];
#pragma unroll
      for (int i = 1; i < kWarps; ++i) v += red[i * kDepBuf + e];
      red[e] = v;
    }
    cluster_sync();
    if (threadIdx.x < per) {   // the cluster's blocks, in rank order; this block's share of the outputs
      const int e = (int)rank * per + threadIdx.x;
      double v = ld_cluster(red + e, 0);
#pragma unroll
      for (unsigned q = 1; q < CL; ++q) v += ld_cluster(red + e, q);
      const int c = e / kLanes, l = e - c * kLanes, craw = tile * T - H + l;
      if (l >= H && l < H + T && craw < g.nz) {
        v *= g.kappa_dV;
        nonfinite |= !isfinite(v);
        out[(int64_t)c * B.NZ + g.coff + craw] = v;
      }
    }
    cluster_sync();   // the slots are free for the next tile, and no block leaves while read
  }
  if (bad) atomicOr(err, bad);
  if (nonfinite) atomicOr(err, ERR_NONFINITE);
}

// Deposit, second phase: fixed-order sum of the per-warp partials.
// out[c * NZ + coff_b + j] (c < rows) = scale_b * (sum over the warps that own
// units of j's tile), scale_b = kappa_b / dV_b (potential) or 1 / dV_b.  Lane l of a warp
// takes output e0 + l (consecutive cells: coalesced reads of the partials).
// With `split` > 1 (a power of two <= 8), `split` warps of a block take the
// same 32 outputs: warp i adds the partials of warps wf + i, wf + i + split,
// ..., and the first adds the split sums in warp order through shared
// memory.  A warp keeps kCombineILP running sums (its partials taken
// round-robin, then added pairwise) so that many loads are in flight.  The
// order depends only on the batch, the number of warps that split the units
// and `split`, not on the grid of this phase: results are bitwise reproducible.
// The partials are read through L2 (coherent within a fused launch too).
constexpr int kCombineILP = 8;
__device__ __forceinline__ void combine_phase(const Batch& B, const double* partial, double* out, int rows,
                                              int potential, int split, int* err) {
  __shared__ double sums[kWarps][kLanes];
  const int64_t n = (int64_t)rows * B.NZ;
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
  const int grp = wib / split, wi = wib - grp * split;       // output group of this warp, rank within it
  const int groups = kWarps / split;
  int bad = 0;
  // every block runs the same number of rounds (it synchronises inside)
  for (int64_t base = (int64_t)blockIdx.x * groups * kLanes; base < n; base += (int64_t)gridDim.x * groups * kLanes) {
    const int64_t e = base + (int64_t)grp * kLanes + lane;
    double v = 0.0;
    const BoxGeo* g = nullptr;
    if (e < n) {
      const int c = (int)(e / B.NZ), gc = (int)(e - (int64_t)c * B.NZ);
      g = &B.box[box_of_cell(B, gc)];
      const int lc = gc - g->coff;
      const int tile = lc / B.T, k = lc - tile * B.T;
      // the slots of the tile's partials: of the warps that own units of it, or of its parts
      int64_t gtile = g->toff + tile, wf, wl;
      if (B.dpb > 0) {
        wf = first_part(B, g, tile);
        wl = wf + (g->M + B.dpb - 1) / B.dpb - 1;
        gtile = 0;
      } else {
        wf = warp_of_unit(g->uoff + (int64_t)tile * g->M, B);
        wl = warp_of_unit(g->uoff + (int64_t)(tile + 1) * g->M - 1, B);
      }
      const double* src = partial + c * B.T + k;
      double a[kCombineILP] = {};
      int64_t q = wf + wi;
      for (; q + (kCombineILP - 1) * split <= wl; q += kCombineILP * split) {
#pragma unroll
        for (int i = 0; i < kCombineILP; ++i) a[i] += __ldcg(src + (q + i * split + gtile) * kSlot);
      }
      for (; q <= wl; q += split) a[0] += __ldcg(src + (q + gtile) * kSlot);
#pragma unroll
      for (int h = kCombineILP / 2; h >= 1; h /= 2) {   // pairwise: ((a0 + a4) + (a2 + a6)) + ...
#pragma unroll
        for (int i = 0; i < h; ++i) a[i] += a[i + h];
      }
      v = a[0];
    }
    if (split > 1) {
      sums[wib][lane] = v;
      __syncthreads();
      if (wi == 0)
        for (int i = 1; i < split; ++i) v += sums[wib + i][lane];
      __syncthreads();
    }
    if (e < n && wi == 0) {
      v *= potential ? g->kappa_dV : g->inv_dV;
      bad |= !isfinite(v);
      out[e] = v;
    }
  }
  if (bad) atomicOr(err, ERR_NONFINITE);
}

static __global__ void k_combine(Batch B, const double* __restrict__ partial, double* __restrict__ out, int rows,
                          int potential, int split, int* __restrict__ err) {
  griddep_wait();
  combine_phase(B, partial, out, rows, potential, split, err);
}

// The RK4 update (Sec. 2.3) of particle p at stage s: K =
// -i[H, rho], Kbar = -i[Hbar, rhobar] (Eq. 4) from the operand hm of H (Eq. 6,
// Eq. 2; OWNBAR: hb of Hbar, otherwise Hbar = -H^*) and the neutrino source
// matrix r (already loaded; the antineutrinos' source is src_b), then the
// accumulator and next stage state (stage 4: the new state and position, from
// *vz).  S is the stage (2 stands for 2 and 3).  With KEEP the state it stores (the next stage's, or at
// stage 4 the new one), rho and rhobar, is also combined as
// B = n1 rho - n2 rhobar^* into keep[9] (the arithmetic of the deposit, Eq. 5)
// and the new position returned in *zkeep.
// The commutators run on the integer pipe (wide.cuh), the updates as FP64
// multiply-adds: 36 + 31 FP64 instructions a particle instead of 144 (at
// 16 cycles each the FP64 pipe bound the stage).
template <int N>
struct Int {
  static constexpr int value = N;
};

template <int S, bool OWNBAR, bool COH, bool KEEP = false>
__device__ __forceinline__ void rk_update(double Lz, const Parts& pt, const double* src_b, int64_t P_, int64_t p,
                                          int dry, double bdt, double cdt, double dtb,
                                          const double* vz, const emu_wide::Ham& hm, const emu_wide::Ham& hb,
                                          double (&r)[9], double* keep = nullptr, double* zkeep = nullptr,
                                          double n1 = 0.0, double n2 = 0.0) {
  namespace w = emu_wide;
  const unsigned P = (unsigned)P_;
  static_assert(S == 1 || S == 2 || S == 4, "stage 1, 2 (and 3) or 4");
  constexpr bool first = S == 1, last = S == 4;
  // Sums of products have an exponent of at least emin, so that the
  // coefficients that take it (below) stay normal; infinite and NaN inputs
  // raise it to kInfExp, and the coefficients, out of range, then make every
  // result NaN
  constexpr int kInfExp = 1 << 16;
  const int emin0 = w::kBiasP + 1 - w::min_i(w::exponent(bdt), w::exponent(cdt));
  const int htop = w::top(hm);
  // one pass per species: a loop, not unrolled (the commutator's ~600
  // instructions once keep the stage in the instruction cache)
#pragma unroll 1
  for (int which = 0; which < 2; ++which) {
    const w::Ham& h = OWNBAR && which ? hb : hm;
    const w::Mat m = w::mat(r, !OWNBAR && which);
    const int top = w::max_i(w::top(m), OWNBAR && which ? w::top(hb) : htop);
    const int emin = top < w::kExpNonFinite ? emin0 : kInfExp;
    double* __restrict__ yv = (which ? pt.rhobar : pt.rho) + p;
    double* __restrict__ av = row(pt.acc, P, which * 9) + p;
    double* __restrict__ sv = row(pt.stage, P, which * 9) + p;
    double* __restrict__ dst = (!last || dry) ? sv : yv;
    // the accumulator and the step's start of component k
    auto load = [&](int k, double& a, double& y) {
      a = first ? r[k] : ldp<COH>(row(av, P, k));
      y = first ? r[k] : last ? 0.0 : ldp<COH>(row(yv, P, k));
    };
    // its update from K_k = kv 2^e: the coefficients bdt, cdt take the exponent
    auto update = [&](int k, double kv, int e, double a, double y) {
      double nv;   // the state stored: the next stage's, or at stage 4 the new one
      if (last) {
        nv = fma(w::scale_up(bdt, e), kv, a);
      } else {
        *row(av, P, k) = fma(w::scale_up(bdt, e), kv, a);
        nv = fma(w::scale_up(cdt, e), kv, y);
      }
      *row(dst, P, k) = nv;
      if constexpr (KEEP)   // B = n1 rho - n2 rhobar^*: conj(rhobar) flips the sign of the imaginary components
        keep[k] = which == 0 ? n1 * nv : fma((k == 4 || k == 6 || k == 8) ? n2 : -n2, nv, keep[k]);
    };
    // K = -i[H, r]: neutrinos K_12.. = (Im C, -Re C).  Antineutrinos with
    // Hbar = -H^*: conj(rhobar) obeys the neutrinos' equation with the same H,
    // and Kbar = conj(K): (Im C, Re C).  Entry by entry, each with its loads
    // issued before its products and finished before the next: few registers
    // wait, and the products cover the loads' latency.
    const int flip = (which == 1 && !OWNBAR) ? 0 : (int)0x80000000;
    auto off = [&](auto Q) {
      constexpr int q = decltype(Q)::value, k = 3 + 2 * q;
      double a0, a1, y0, y1, cr, ci;
      int e;
      load(k, a0, y0);
      load(k + 1, a1, y1);
      w::commutator_off<q>(h, m, emin, cr, ci, e);
      e = w::min_i(e - w::kBiasP, 3000);
      update(k, ci, e, a0, y0);
      update(k + 1, w::from_words(w::hi_word(cr) ^ flip, w::lo_word(cr)), e, a1, y1);
    };
    off(Int<0>{});
    off(Int<1>{});
    off(Int<2>{});
    {
      double a[3], y[3], kd[3];
      int ke[3];
#pragma unroll
      for (int k = 0; k < 3; ++k) load(k, a[k], y[k]);
      if (which == 0) {   // the other species' source
#pragma unroll
        for (int k = 0; k < 9; ++k) r[k] = ldp<COH>(row(src_b + p, P, k));
      }
      w::commutator_diag(h, m, emin, kd, ke);
#pragma unroll
      for (int k = 0; k < 3; ++k) update(k, kd[k], w::min_i(ke[k] - w::kBiasP + 1, 3000), a[k], y[k]);   // (halved)
    }
  }
  if (last) {
    const double vzv = *vz;   // (a plain load: vz may point at a caller's local value)
    const double zn = wrap_z(fma(dtb, vzv, ldp<COH>(pt.z + p)), Lz);
    if (dry) pt.stage[p] = zn;  // (only to keep the work of the real stage)
    else pt.z[p] = zn;
    if constexpr (KEEP) *zkeep = zn;
  }
}

// Coefficients of K at stage s (Sec. 2.3): bdt in the accumulator, cdt in the
// next stage's state (at least the smallest normal number: rk_update scales
// them by powers of two).
__device__ __forceinline__ void rk_coefficients(int s, double dt, double& bdt, double& cdt) {
  bdt = fmax((s == 1 || s == 4) ? dt / 6.0 : dt / 3.0, 0x1p-1022);
  cdt = fmax(s == 3 ? dt : 0.5 * dt, 0x1p-1022);
}

// H + V and Hbar = -H^* + Vbar with the box's vacuum and matter terms (Eq. 2):
// in the traceless components the diagonal differences and real parts of -H^*
// flip sign, the imaginary parts stay.
__device__ __forceinline__ void add_potentials(const BoxGeo& g, double (&Hm)[kNC], double (&Hb)[kNC]) {
#pragma unroll
  for (int c = 0; c < kNC; ++c) {
    const bool im = (c == 3 || c == 5 || c == 7);
    Hb[c] = (im ? Hm[c] : -Hm[c]) + __ldg(g.vnubar + c);
    Hm[c] += __ldg(g.vnu + c);
  }
}

// rk_update of particle p of box g from H in the traceless components.
template <bool POT, int S, bool COH, bool KEEP = false>
__device__ __forceinline__ void rk_particle(const BoxGeo& g, const Parts& pt, const double* src_b, int64_t P,
                                            int64_t p, int dry, double bdt, double cdt, double dtb,
                                            const double* __restrict__ vz, double (&Hm)[kNC], double (&r)[9],
                                            double* keep = nullptr, double* zkeep = nullptr, double n1 = 0.0,
                                            double n2 = 0.0) {
  if constexpr (POT) {
    double Hb[kNC];
    add_potentials(g, Hm, Hb);
    const emu_wide::Ham hm = emu_wide::ham(Hm), hb = emu_wide::ham(Hb);
    rk_update<S, true, COH, KEEP>(g.Lz, pt, src_b, P, p, dry, bdt, cdt, dtb, vz, hm, hb, r, keep, zkeep, n1, n2);
  } else {
    const emu_wide::Ham hm = emu_wide::ham(Hm);
    rk_update<S, false, COH, KEEP>(g.Lz, pt, src_b, P, p, dry, bdt, cdt, dtb, vz, hm, hm, r, keep, zkeep, n1,
                                   n2);
  }
}

// The commutator's operand from H in the traceless components, given as
// hv[c] 2^(he[c / 2] - kBiasV), |hv| < 2^60.8.
__device__ __forceinline__ emu_wide::Ham operand_ham(const int64_t (&hv)[kNC], const int (&he)[4]) {
  namespace w = emu_wide;
  w::Ham hm;
  hm.d12 = w::Real{w::split(hv[0]), he[0]};
  hm.d13 = w::Real{w::split(hv[0] + hv[1]), he[0]};
  hm.d23 = w::Real{w::split(hv[1]), he[0]};
  hm.a = w::Cplx{w::split(hv[2]), w::split(hv[3]), he[1]};
  hm.b = w::Cplx{w::split(hv[4]), w::split(hv[5]), he[2]};
  hm.c = w::Cplx{w::split(hv[6]), w::split(hv[7]), he[3]};
  return hm;
}

// H + V with the box's potential terms as operands (NEGH: with -H^* instead of H,
// NEGV: with -V^*): added at the larger exponent of each group, two bits of headroom.
// (As doubles 32 FP64 instructions a particle more: 1999 x 251 cubic 124 us a stage, now 115.)
template <bool NEGH, bool NEGV>
__device__ __forceinline__ emu_wide::Ham operand_sum(const int64_t (&hv)[kNC], const int (&he)[4], const long long* vq,
                                                     const int* ve) {
  namespace w = emu_wide;
  int64_t s[kNC];
  int e[4];
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const int ev = __ldg(ve + q);
    e[q] = max(he[q], ev) + 2;
    const int dh = e[q] - he[q], dv = e[q] - ev, fh = max(dh - 32, 0), fv = max(dv - 32, 0);
#pragma unroll
    for (int c = 2 * q; c < 2 * q + 2; ++c) {
      const bool im = c == 3 || c == 5 || c == 7;
      const int64_t a = w::align(hv[c], dh, fh), b = w::align(__ldg(vq + c), dv, fv);
      s[c] = (NEGH && !im ? -a : a) + (NEGV && !im ? -b : b);
    }
  }
  return operand_ham(s, e);
}

// rk_update of particle p of box g from H (hv, he as operand_ham).
template <bool POT, int S, bool COH>
__device__ __forceinline__ void rk_from_H(const BoxGeo& g, const Parts& pt, const double* src_b, int64_t P, int64_t p,
                                          int dry, double bdt, double cdt, double dtb, const double* vz,
                                          const int64_t (&hv)[kNC], const int (&he)[4], double (&r)[9]) {
  if constexpr (POT) {
    const emu_wide::Ham hm = operand_sum<false, false>(hv, he, g.vq[0], g.ve[0]);
    const emu_wide::Ham hb = operand_sum<true, false>(hv, he, g.vq[1], g.ve[1]);
    rk_update<S, true, COH>(g.Lz, pt, src_b, P, p, dry, bdt, cdt, dtb, vz, hm, hb, r);
  } else {
    const emu_wide::Ham hm = operand_ham(hv, he);
    rk_update<S, false, COH>(g.Lz, pt, src_b, P, p, dry, bdt, cdt, dtb, vz, hm, hm, r);
  }
}

// Arrays of the adjoint's first stage kernel (k_adj_a).
struct AdjStage {
  const double *lam, *lamn;   // adjoint of the step's result and of the next stage's state (NULL at stage 4)
  double *out, *gam;          // adjoint of this stage's state (direct terms), and of its H
};

// k_adj_a for particle p: r its neutrino matrix (loaded), H as rk_from_H.  The
// antineutrinos take the neutrinos' operand: with h = H - Vbar^* (H without
// potentials) -K(Hbar, m) = -conj K(h, m^*) and -conj K(rbar, m) = K(rbar^*, m^*).
template <bool POT>
__device__ __forceinline__ void adj_update(const BoxGeo& g, const Parts& pt, int64_t P_, int64_t p, double a, double c,
                                           const AdjStage& x, const int64_t (&hv)[kNC], const int (&he)[4],
                                           double (&r)[9]) {
  namespace w = emu_wide;
  const unsigned P = (unsigned)P_;
  double Gm[9];
  w::Ham h;
  if constexpr (!POT) h = operand_ham(hv, he);
#pragma unroll
  for (int k = 0; k < 9; ++k) Gm[k] = 0.0;
#pragma unroll 1
  for (int which = 0; which < 2; ++which) {
    const double* lam = row(x.lam, P, which * 9) + p;
    const double* ln = row(x.lamn, P, which * 9) + p;
    double* out = row(x.out, P, which * 9) + p;
    double m2[9], kd[3], ko[6];
#pragma unroll
    for (int k = 0; k < 9; ++k) {
      const double f = k < 3 ? 2.0 : 1.0;
      m2[k] = f * a * __ldg(row(lam, P, k));
      if (x.lamn != nullptr) m2[k] = fma(f * c, __ldg(row(ln, P, k)), m2[k]);
    }
    const w::Mat m = w::mat(m2, which);
    if constexpr (POT)
      h = which == 0 ? operand_sum<false, false>(hv, he, g.vq[0], g.ve[0])
                     : operand_sum<false, true>(hv, he, g.vq[1], g.ve[1]);
    commutator(h, m, kd, ko);
#pragma unroll
    for (int k = 0; k < 3; ++k) *row(out, P, k) = -kd[k];
#pragma unroll
    for (int k = 0; k < 6; ++k) *row(out, P, 3 + k) = (k & 1) && which ? ko[k] : -ko[k];
    const double cj = which ? -1.0 : 1.0;
    const double rt[kNC] = {r[0] - r[1], r[1] - r[2], r[3], cj * r[4], r[5], cj * r[6], r[7], cj * r[8]};
    w::Ham rh = w::ham(rt);
    rh.d13 = w::real(r[0] - r[2]);
    if (which == 0) {   // the antineutrinos' matrix
#pragma unroll
      for (int k = 0; k < 9; ++k) r[k] = __ldg(row(pt.rhobar + p, P, k));
    }
    commutator(rh, m, kd, ko);
#pragma unroll
    for (int k = 0; k < 9; ++k) Gm[k] += k < 3 ? kd[k] : ko[k - 3];
  }
#pragma unroll
  for (int k = 0; k < 9; ++k) *row(x.gam + p, P, k) = Gm[k];
}

// Box of tile unit x of the slabs (a pair of a slab and a direction counts as
// its sw tile units).
__device__ __forceinline__ int box_of_slab_unit(const Batch& B, int64_t x) {
  int lo = 0, hi = B.nbox - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (B.box[mid].soff <= x) lo = mid; else hi = mid - 1;
  }
  return lo;
}

// One RK4 stage s (1..4) after the deposit of the stage state: interpolate
// (Eq. 6), H and Hbar = -H^* (Eq. 2, Sec. 2.1), K = -i[H, rho] and
// Kbar = -i[Hbar, rhobar] (Eq. 4), then the classic RK4 update (Sec. 2.3):
//   s = 1: acc = y + dt/6 K,  stage = y + dt/2 K
//   s = 2: acc += dt/3 K,     stage = y + dt/2 K
//   s = 3: acc += dt/3 K,     stage = y + dt K
//   s = 4: y = acc + dt/6 K,  z = wrap(z + dt v_z)   (dry: into the stage buffer instead)
// With POT the constant vacuum and matter terms of the box are added:
// H = H_self + V, Hbar = -H_self^* + Vbar (Eq. 2, Sec. 2.1).  Stages 2-4 read
// their state from stage_src (normally the stage buffer itself, updated in
// place; a separate buffer when the stage states are kept for the adjoint).
//
// Work split.  Batch::slabs 1: a block takes a contiguous range of (slab,
// direction) pairs of the batch (an equal share of their tile units), slab by
// slab; a slab is 1, 2, 4 or 8 (BoxGeo::sw) consecutive 32-cell tiles.  Batch::
// slabs 0 (few units): a block takes a part of one tile's directions (at most
// upb), so that no block does two tiles one after the other while others idle
// (256 x 96: 3 units a block on 256 blocks).  The block converts the slab's (tile's)
// potential once to integer operands
// in shared memory (per cell and moment the 8 traceless components, one
// exponent per cell for the diagonal pair and for each complex component),
// and its warps walk the slab's directions: with sw tiles, warp i takes tile
// i mod sw and every (8 / sw)-th direction, so the warps of a block read
// adjacent pieces of the same rings (sw = 8: 2 KB of every array).  Per unit a
// warp forms G = A0 - Omega . A of its cells, the neighbours' G come from
// shared memory, and the stencil sum is the commutator's operand: everything
// up to the update runs on the integer pipe.  Latency bounds it: four warps a
// scheduler (126 registers), issue slots 45-49 % busy, fixed-latency waits and
// memory the largest stalls, the FP64 pipe (conversions and updates) busiest at
// 56-71 %, HBM at 53 %.  16384 x 1000 5.13 -> 2.64 ms a stage against FP64 arithmetic
// (the FP64 pipe its bound), 1024 x 378 139 -> 73 us.
constexpr int kSlabTiles = 8;                      // most tiles of a slab
constexpr int kRowCells = kLanes + 4;              // cells of a unit, likewise
template <int TILES>                               // of the widest slab
struct SlabTable {
  static constexpr int kSlabCells = TILES * kLanes + 4;   // its cells, two neighbours a side
  int2 a[kNT][kSlabCells];                         // the potential: A0 / 4 as int64, limbs of A_x, A_y, A_z
  int e[4][kSlabCells];                            // exponents: diagonal pair, three complex components
  int2 g[kWarps][kNC][kRowCells];                  // limbs of G of each warp's unit
  const double* pf[64];                            // the arrays a stage reads, for the L2 prefetch
};
constexpr int kSlabSmem = (int)sizeof(SlabTable<kSlabTiles>);
constexpr int kStepSmem = kSlabSmem > kDepSmem ? kSlabSmem : kDepSmem;   // of k_step: either phase's

// The operands of one exponent group of NV / 4 components of the potential at a
// cell: v[k] moment k / (NV / 4), component k % (NV / 4) of the group; put(k,
// operand): A0 / 4 as an int64 (low, high word; dot3's addend), limbs of A_x,
// A_y, A_z.  Returns their exponent.
template <int NV, typename F>
__device__ __forceinline__ int potential_operands(const double (&v)[NV], F put) {
  namespace w = emu_wide;
  int e[NV], top = 0;
#pragma unroll
  for (int k = 0; k < NV; ++k) {
    e[k] = w::exponent(v[k]);
    top = max(top, e[k]);
  }
#pragma unroll
  for (int k = 0; k < NV; ++k) {
    const w::Limbs l = w::limbs(v[k], e[k], top);
    int2 x = make_int2(l.h, l.l);
    if (k < NV / 4) {
      const int64_t q = w::join(l) >> 2;
      x = make_int2((int)q, (int)(q >> 32));
    }
    put(k, x);
  }
  return top;
}

// Potential of cells c0 .. c0 + n - 1 (modulo nz) of box g into the table, by
// the whole block: one (cell, exponent group) per thread and round.
template <bool COH, class Table>
__device__ __forceinline__ void slab_table(Table& t, const double* A, int NZ, const BoxGeo& g, int c0, int n) {
  for (int q = threadIdx.x; q < 4 * n; q += blockDim.x) {
    const int grp = q / n, c = q - grp * n;
    const double* Aj = A + g.coff + wrapc(c0 + c, g.nz) + (int64_t)2 * grp * NZ;
    double v[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) v[k] = ldd<COH>(Aj + (int64_t)((k >> 1) * kNC + (k & 1)) * NZ);
    t.e[grp][c] = potential_operands(
        v, [&](int k, int2 x) { t.a[(k >> 1) * kNC + 2 * grp + (k & 1)][c] = x; });
  }
}

__device__ __forceinline__ emu_wide::Limbs limbs_of(int2 v) { return emu_wide::Limbs{v.x, v.y}; }

// G = A0 - Omega . A from the operands of one component (o: limbs of -Omega;
// directions scaled by 2^-ko: so is G); component c of it at table cell j.
__device__ __forceinline__ int2 operand_G(int2 q, int2 a1, int2 a2, int2 a3, const emu_wide::Limbs (&o)[3], int ko) {
  const int64_t a0 = (int64_t)(((uint64_t)(uint32_t)q.y << 32) | (uint32_t)q.x);
  const emu_wide::Limbs g = emu_wide::split(
      emu_wide::dot3(emu_wide::align(a0, ko, 0), limbs_of(a1), o[0], limbs_of(a2), o[1], limbs_of(a3), o[2]));
  return make_int2(g.h, g.l);
}
template <class Table>
__device__ __forceinline__ int2 table_G(const Table& t, int c, int j, const emu_wide::Limbs (&o)[3], int ko) {
  return operand_G(t.a[c][j], t.a[kNC + c][j], t.a[2 * kNC + c][j], t.a[3 * kNC + c][j], o, ko);
}

template <bool POT, int ORDER, int S, bool COH, class Table>
__device__ __forceinline__ void rk_phase(const Batch& B, const Parts& pt, const double* W, const double* wrow,
                                         const double* __restrict__ dirtab, const int* shift, const double* A,
                                         const double* stage_src, int s, int dry, Table& t,
                                         const AdjStage& adj = {}) {
  namespace w = emu_wide;
  constexpr int H = ORDER == 0 ? 0 : Sten<ORDER>::H, NW = ORDER == 0 ? 1 : Sten<ORDER>::NW;
  constexpr int NWS = Sten<ORDER>::NWS;
  const int lane = threadIdx.x & 31;
  const int wib = __shfl_sync(kFull, (int)(threadIdx.x >> 5), 0);
  const int64_t P = B.Ptot;
  const int MT = B.MT;
  const double* src_r = S <= 1 ? pt.rho : stage_src;
  const double* src_b = S <= 1 ? pt.rhobar : stage_src + 9 * P;
  // the arrays this stage reads per particle
  const int ny = S == 2 || (S == 0 && adj.lamn != nullptr) ? 18 : 0;
  constexpr int nacc = S == 1 ? 0 : 18, nz_ = S == 4 ? 1 : 0;
  const int narr = 18 + ny + nacc + nz_ + (wrow != nullptr ? 0 : NWS);
  __syncthreads();
  for (int a = threadIdx.x; a < narr; a += blockDim.x) {
    const double* arr;
    if (a < 18) arr = a < 9 ? src_r + a * P : src_b + (a - 9) * P;
    else if (a < 18 + nacc) arr = (S == 0 ? adj.lam : pt.acc) + (a - 18) * P;
    else if (S == 0 && a < 18 + nacc + ny) arr = adj.lamn + (a - 18 - nacc) * P;
    else if (a < 18 + nacc + ny) arr = a - 18 - nacc < 9 ? pt.rho + (a - 18 - nacc) * P
                                                         : pt.rhobar + (a - 18 - nacc - 9) * P;
    else if (a < 18 + nacc + ny + nz_) arr = pt.z;
    else arr = W + (a - 18 - nacc - ny - nz_) * P;
    t.pf[a] = arr;
  }
  // slabs: this block's tile units [x, x1), a (slab, direction) pair belonging
  // to the block its first unit falls to; otherwise its parts part, part + grid, ..
  int64_t x = B.slabs ? (int64_t)blockIdx.x * B.US / gridDim.x : 0;
  const int64_t x1 = B.slabs ? ((int64_t)blockIdx.x + 1) * B.US / gridDim.x : 0;
  int part = blockIdx.x;
  int b = B.slabs && x < x1 ? box_of_slab_unit(B, x) : 0;
  while (true) {
    int slab, d0, d1, sw = 1;
    if (B.slabs) {
      if (x >= x1 || b >= B.nbox) break;
      const BoxGeo& g = B.box[b];
      const int M = g.M;
      sw = g.sw;
      const int nslab = (g.ntiles32 + sw - 1) / sw;
      const int64_t q = (x - g.soff + sw - 1) / sw;                             // first pair, box-local
      const int64_t q1 = min((int64_t)nslab * M, (x1 - g.soff + sw - 1) / sw);   // and the end of this block's
      if (q >= q1) {   // (the box's pairs left start in later blocks, or it has none left)
        x = g.soff + (int64_t)nslab * M * sw;
        ++b;
        continue;
      }
      slab = (int)(q / M);
      d0 = (int)(q - (int64_t)slab * M);
      d1 = (int)min((int64_t)M, (int64_t)d0 + (q1 - q));
      x = g.soff + (q + (d1 - d0)) * sw;
    } else {
      int k = part, per = 0;
      for (b = 0; b < B.nbox; ++b) {
        per = (B.box[b].M + B.upb - 1) / B.upb;   // parts of a tile
        const int all = per * B.box[b].ntiles32;
        if (k < all) break;
        k -= all;
      }
      if (b == B.nbox) break;
      part += gridDim.x;
      slab = k / per;
      const int i = k - slab * per, M = B.box[b].M, len = M / per, more = M - len * per;
      d0 = i * len + min(i, more);   // (the first `more` parts take one more)
      d1 = d0 + len + (i < more);
    }
    const BoxGeo& g = B.box[b];
    const int nz = g.nz;
    const int c0 = slab * sw * kLanes;
    const int tile0 = (wib & (sw - 1)) * kLanes;       // this warp's tile within the slab, in cells
    const int n = min(kLanes, nz - c0 - tile0);
    const int dstep = (int)(blockDim.x >> 5) / sw;
    double bdt, cdt;
    const double dtb = B.dt[b];
    rk_coefficients(S == 2 || S == 0 ? s : S, dtb, bdt, cdt);
    const int64_t poff = g.poff;
    const int doff = g.doff;
    const int tc = tile0 + H + lane;                   // table cell of this lane
    // a direction's own numbers, loaded a unit ahead: -Omega in lanes 0-2, the
    // ring's weights (when every particle takes them) in the next NW, the shift
    const bool ring = ORDER > 0 && wrow != nullptr;
    const double* utab = lane < 3 ? dirtab + lane * MT : wrow + (lane - 3) * MT;
    const bool uload = lane < 3 || (ring && lane < 3 + NW);
    auto own_number = [&](int gd) {
      const double v = uload ? ldp<COH>(utab + gd) : 0.0;
      return lane < 3 ? -v : v;
    };
    const int dw = d0 + wib / sw;
    const bool active = lane < n, some = n > 0 && dw < d1;
    double unext = 0.0;
    int shnext = 0;
    if (some) {   // (these loads' latency before the table's)
      unext = own_number(doff + dw);
      shnext = ldi<COH>(shift + doff + dw);
    }
    __syncthreads();   // (the previous slab's table is free, and pf is written)
    slab_table<COH>(t, A, B.NZ, g, c0 - H, min(sw * kLanes, nz - c0) + 2 * H);
    __syncthreads();
    if (!some) continue;
    for (int d = dw; d < d1; d += dstep) {
      const int gd = doff + d;
      const int sh = shnext;
      const double u = unext;
      if (d + dstep < d1) {   // prefetch the next unit's particle data into L2
        unext = own_number(gd + dstep);
        shnext = ldi<COH>(shift + gd + dstep);
        int i0 = c0 + tile0 - shnext;
        if (i0 < 0) i0 += nz;
        const int cnt = min(n, nz - i0);
        const int64_t nb = poff + (int64_t)(d + dstep) * nz + i0;
        for (int x = lane; x < 3 * narr; x += kLanes) {
          const int a = (x * 171) >> 9, l = x - 3 * a;   // x / 3, x % 3 (exact below 256)
          prefetch_line(t.pf[a] + nb + min(16 * l, cnt - 1));
        }
      }
      int i = c0 + tile0 + lane - sh;
      if (i < 0) i += nz;
      const int64_t p = poff + (int64_t)d * nz + (active ? i : 0);
      // the neutrino source matrix and the weights first, so their latency
      // overlaps the interpolation
      double r[9], wd[NW];
#pragma unroll
      for (int k = 0; k < 9; ++k) r[k] = ldp<COH>(row(src_r + p, (unsigned)P, k));
      if (ORDER > 0 && !ring) {
#pragma unroll
        for (int o = 0; o < NW; ++o) wd[o] = ldp<COH>(row(W + p, (unsigned)P, o));
      }
      // (longer directions than unit vectors are scaled by 2^-ko)
      int ko;
      const w::Limbs ul = direction_limbs(u, lane, ko);
      const w::Limbs om[3] = {bcast(ul, 0), bcast(ul, 1), bcast(ul, 2)};
      // G of this lane's cell and of the H cells on each side of the tile
      if (active) {
        if (ko == 0) {
#pragma unroll
          for (int c = 0; c < kNC; ++c) t.g[wib][c][H + lane] = table_G(t, c, tc, om, 0);
        } else {
#pragma unroll 1
          for (int c = 0; c < kNC; ++c) t.g[wib][c][H + lane] = table_G(t, c, tc, om, ko);
        }
      }
      if constexpr (H > 0) {
        if (lane < 2 * H * kNC) {
          const int c = lane & (kNC - 1), h = lane >> 3;
          const int x = h < H ? h : n + h;            // position among the unit's cells
          t.g[wib][c][x] = table_G(t, c, tile0 + x, om, ko);
        }
      }
      w::Limbs wl[NW];
      if constexpr (ORDER > 0) {
#pragma unroll
        for (int o = 0; o < NW; ++o) wl[o] = wrow != nullptr ? bcast(ul, 3 + o) : w::unit_limbs(wd[o]);
      }
      __syncwarp();
      if (active) {
        // interpolation (Eq. 6): per component the taps at the largest exponent
        int64_t hv[kNC];
        int he[4];
#pragma unroll
        for (int grp = 0; grp < 4; ++grp) {
          int e[NW], dd[NW], df[NW];
          he[grp] = 0;
#pragma unroll
          for (int o = 0; o < NW; ++o) {
            e[o] = t.e[grp][tc - H + o];
            he[grp] = max(he[grp], e[o]);
          }
#pragma unroll
          for (int o = 0; o < NW; ++o) {
            dd[o] = he[grp] - e[o];
            df[o] = max(dd[o] - 32, 0);
          }
#pragma unroll
          for (int c = 2 * grp; c < 2 * grp + 2; ++c) {
            if constexpr (ORDER == 0) {
              hv[c] = w::join(limbs_of(t.g[wib][c][lane]));
            } else {
              int64_t v = 0;
#pragma unroll
              for (int o = 0; o < NW; ++o)
                v += w::align(w::mul(limbs_of(t.g[wib][c][lane + o]), wl[o]), dd[o], df[o]);
              hv[c] = v * 4;
            }
          }
        }
        // hv[c] 2^(he + 2 - kBiasV) = H_c, then he + 2 -> he (a particle's own weights
        // need no test: where they are not finite, the deposit's potential is not)
        if (ko != 0) {
#pragma unroll
          for (int grp = 0; grp < 4; ++grp) he[grp] = ko <= w::kMaxExcess ? he[grp] + ko : w::kExpNonFinite;
        }
#pragma unroll
        for (int grp = 0; grp < 4; ++grp) he[grp] += 2;
        if constexpr (S == 0) adj_update<POT>(g, pt, P, p, bdt, cdt, adj, hv, he, r);
        else rk_from_H<POT, S, COH>(g, pt, src_b, P, p, dry, bdt, cdt, dtb, dirtab + 3 * MT + gd, hv, he, r);
      }
      __syncwarp();   // (the unit's G are rewritten by the next)
    }
  }
}

// TILES: of the widest slab (kSlabTiles, or 1 when Batch::slabs is 0: the
// smaller table leaves the SM room for the next kernel's blocks).
template <bool POT, int ORDER, int S, int TILES>
__global__ void __launch_bounds__(kThreads, 2)
k_rk_stage(Batch B, Parts pt, const double* __restrict__ W, const double* __restrict__ wrow,
           const double* __restrict__ dirtab, const int* __restrict__ shift, const double* __restrict__ A,
           const double* stage_src, int s, int dry) {
  extern __shared__ char smem[];
  griddep_wait();
  rk_phase<POT, ORDER, S, false>(B, pt, W, wrow, dirtab, shift, A, stage_src, s, dry, *(SlabTable<TILES>*)smem);
}

// ------------------------------------------------------ interpolation only
//
// H[k * Ptot + p] (Eq. 6 then Eq. 2, 9 packed components) of a single box's
// particles at z + frac dt v_z, each with its own weights, from the potential
// A[36][NZ].  As rk_phase up to H: a block takes a range of (slab of 4 tiles,
// direction) pairs and converts the slab's potential once; the diagonal entries
// have an exponent each.  (18 FP64 instructions a particle for 63 with FP64 G and
// taps: 2048 x 1000 262 -> 116 us.)
struct InterpTable {
  static constexpr int kTiles = 4, kCells = kTiles * kLanes + 4;
  int2 a[kNA][kCells];
  int e[6][kCells];              // exponents: three diagonal entries, three complex components
  int2 g[kWarps][9][kRowCells];
};
constexpr int kInterpSmem = (int)sizeof(InterpTable);

template <int ORDER>
__global__ void __launch_bounds__(kThreads, 2)
k_interpolate(Batch B, const double* __restrict__ z, const double* __restrict__ dirtab,
              const int* __restrict__ shift, const double* __restrict__ A, double frac, double* __restrict__ Hout,
              int* __restrict__ err) {
  namespace w = emu_wide;
  extern __shared__ char smem[];
  InterpTable& t = *(InterpTable*)smem;
  constexpr int H = ORDER == 0 ? 0 : Sten<ORDER>::H, NW = ORDER == 0 ? 1 : Sten<ORDER>::NW;
  const int lane = threadIdx.x & 31, wib = __shfl_sync(kFull, (int)(threadIdx.x >> 5), 0);
  const unsigned P = (unsigned)B.Ptot;
  const int MT = B.MT, NZ = B.NZ;
  const BoxGeo& g = B.box[0];
  const int nz = g.nz, M = g.M, nslab = (g.ntiles32 + InterpTable::kTiles - 1) / InterpTable::kTiles;
  const double pos_dt = frac * B.dt[0];
  const int64_t all = (int64_t)nslab * M, q1 = ((int64_t)blockIdx.x + 1) * all / gridDim.x;
  int bad = 0;
  for (int64_t q = (int64_t)blockIdx.x * all / gridDim.x; q < q1;) {
    const int slab = (int)(q / M), d0 = (int)(q - (int64_t)slab * M), d1 = (int)min((int64_t)M, d0 + (q1 - q));
    q += d1 - d0;
    const int c0 = slab * InterpTable::kTiles * kLanes, ncell = min(InterpTable::kTiles * kLanes, nz - c0) + 2 * H;
    __syncthreads();
    int far = 0;   // whether a cell's exponent takes H to an end of the range of doubles
    for (int x = threadIdx.x; x < 6 * ncell; x += kThreads) {
      const int grp = x / ncell, c = x - grp * ncell;
      const double* Aj = A + wrapc(c0 - H + c, nz);
      int e, some = 0;
      if (grp < 3) {
        double v[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          v[k] = __ldg(Aj + (int64_t)(9 * k + grp) * NZ);
          some |= (__double2hiint(v[k]) & 0x7fffffff) | __double2loint(v[k]);
        }
        e = potential_operands<4>(v, [&](int k, int2 o) { t.a[9 * k + grp][c] = o; });
      } else {
        const int k0 = 2 * grp - 3;
        double v[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) {
          v[k] = __ldg(Aj + (int64_t)(9 * (k >> 1) + k0 + (k & 1)) * NZ);
          some |= (__double2hiint(v[k]) & 0x7fffffff) | __double2loint(v[k]);
        }
        e = potential_operands<8>(v, [&](int k, int2 o) { t.a[9 * (k >> 1) + k0 + (k & 1)][c] = o; });
      }
      t.e[grp][c] = e;
      far |= e > 2000 || (e < 64 && some != 0);
    }
    far = __syncthreads_or(far);
    const int tile0 = (wib & (InterpTable::kTiles - 1)) * kLanes, n = min(kLanes, nz - c0 - tile0);
    if (n <= 0) continue;
    const int j = c0 + tile0 + lane, tc = tile0 + H + lane;
    const bool active = lane < n;
    for (int d = d0 + wib / InterpTable::kTiles; d < d1; d += kWarps / InterpTable::kTiles) {
      const int gd = g.doff + d;
      int i = active ? j - __ldg(shift + gd) : 0;
      if (i < 0) i += nz;
      const int64_t p = (int64_t)d * nz + i;
      const double u = lane < 3 ? -__ldg(dirtab + lane * MT + gd) : 0.0;
      double wt[Sten<ORDER>::NW];
      zero_weights<ORDER>(wt);
      int site = 0;
      if (active)
        site = shape_weights<ORDER>(fma(pos_dt, __ldg(dirtab + 3 * MT + gd), z[p]), (double)j + 0.5, g.inv_dz, g.nz_d,
                                    wt);
      bad |= site;
      int ko;
      const w::Limbs ul = direction_limbs(u, lane, ko);
      const w::Limbs om[3] = {bcast(ul, 0), bcast(ul, 1), bcast(ul, 2)};
      auto G = [&](int c, int x) {
        return operand_G(t.a[c][x], t.a[9 + c][x], t.a[18 + c][x], t.a[27 + c][x], om, ko);
      };
      if (active) {
#pragma unroll
        for (int c = 0; c < 9; ++c) t.g[wib][c][H + lane] = G(c, tc);
      }
      if constexpr (H > 0) {   // the H cells on each side
        for (int x = lane; x < 2 * H * 9; x += kLanes) {
          const int c = x % 9, h = x / 9, at = h < H ? h : n + h;
          t.g[wib][c][at] = G(c, tile0 + at);
        }
      }
      __syncwarp();
      if (active) {
        w::Limbs wl[NW];
#pragma unroll
        for (int o = 0; o < NW; ++o) wl[o] = w::unit_limbs(wt[o]);
#pragma unroll
        for (int grp = 0; grp < 6; ++grp) {
          const int nc = grp < 3 ? 1 : 2, k0 = grp < 3 ? grp : 2 * grp - 3;
          int e[NW], he = 0;
#pragma unroll
          for (int o = 0; o < NW; ++o) {
            e[o] = t.e[grp][tc - H + o];
            he = max(he, e[o]);
          }
          const int k2 = w::near(he + 2 + ko - w::kBiasV);
          const bool inf = he >= w::kExpNonFinite || ko > w::kMaxExcess || (site & ERR_NONFINITE);
#pragma unroll
          for (int c = k0; c < k0 + nc; ++c) {
            int64_t v = 0;
            if constexpr (ORDER == 0) {
              v = w::join(limbs_of(t.g[wib][c][lane]));
            } else {
#pragma unroll
              for (int o = 0; o < NW; ++o)
                v += w::align(w::mul(limbs_of(t.g[wib][c][lane + o]), wl[o]), he - e[o]);
              v *= 4;
            }
            *row(Hout + p, P, c) = inf ? nan("") : w::scaled_near(v, k2);
          }
        }
        if (far) {   // (in place: read back by the thread that wrote them)
#pragma unroll 1
          for (int c = 0; c < 9; ++c) {
            int he = 0;
            for (int o = 0; o < NW; ++o) he = max(he, t.e[c < 3 ? c : (c + 3) / 2][tc - H + o]);
            *row(Hout + p, P, c) *= w::far_factor(he + 2 + ko - w::kBiasV);
          }
        }
      }
      __syncwarp();   // (the unit's G are rewritten by the next)
    }
  }
  if (bad) atomicOr(err, bad);
}

// ------------------------------------------- RK stage with the next deposit
//
// Step form 2: every RK stage also deposits (Eq. 5) the state it has just
// computed, at the positions of the next stage (at stage 4: the first stage of
// the next step), so a step is four (combination, RK stage) launch pairs and
// the separate deposit kernel with its re-read of the state is gone.  Units
// are (32-cell tile, direction), TILE-major: a warp walks directions of one
// tile and sums their deposits in shared memory.  Lane l holds the particle on
// cell tile * 32 + l at the stage's positions; every lane owns its particle
// (the G values left of lane 0 and right of the last lane are formed by 16
// lanes, one component each).  Between two stages a ring moves rigidly by
// delta cells, |delta| <= 1 when dt c < 2 dz (the host runs this form only
// then), so the particles of one unit deposit onto cells
// tile * 32 + delta - 1 .. tile * 32 + n + delta: a warp's sums for one tile
// cover the frame of kFrame cells tile * 32 - 2 .. tile * 32 + 33 and go to
// slot (warp + global 32-cell tile) of the partial buffer (unique, as for
// k_deposit).  k_frame_sum adds the slots of each tile in warp order (the
// tile's frame sums), and the next RK stage adds, for each cell, the frame
// entries of the tiles that reach it in a fixed order: bitwise reproducible
// for a fixed grid.  For the shapes of one cell of reach (orders 0-2).
constexpr int kFrame = kLanes + 4;
constexpr int kSlotF = kNT * kFrame;   // doubles in one warp's frame sums for one tile
constexpr int kFrameSmem = (int)sizeof(double) * kWarps * kSlotF;   // dynamic shared memory of k_rk_deposit

__device__ __forceinline__ int64_t warp_of_unit32(int64_t x, const Batch& B) {
  return ((x + 1) * B.nw32 - 1) / B.U32;
}

// Writes a warp's frame sums to its slot and clears them.
__device__ __forceinline__ void flush_frame(double* acc, double* __restrict__ dst, int lane) {
  __syncwarp();
  for (int k = lane; k < kSlotF; k += kLanes) {
    dst[k] = acc[k];
    acc[k] = 0.0;
  }
  __syncwarp();
}

// The frame entries that add up to the potential at cell x of box g: Fr
// offsets of component row 0 in o[0..4] (-1: none).  A tile's frame covers
// cell tile * 32 - 2 + k for k < (its cells) + 4, modulo nz.  When the box has
// at least three tiles and its last tile at least two cells, only the tile of
// x (entry x - tile * 32 + 2) and, for the two cells at either end of a tile,
// the adjacent tile reach x.  Otherwise (rings of few tiles) the tiles of
// cells x - 2 .. x + 2 are taken in that order, once each, with every entry
// of theirs that covers x.
__device__ __forceinline__ bool frame_fast(const BoxGeo& g) {
  return g.ntiles32 >= 3 && g.nz - (g.ntiles32 - 1) * kLanes >= 2;
}
__device__ __forceinline__ void frame_sources(const BoxGeo& g, int x, int (&o)[5]) {
  const int nz = g.nz, nt = g.ntiles32;
#pragma unroll
  for (int q = 0; q < 5; ++q) o[q] = -1;
  if (frame_fast(g)) {
    const int t = x / kLanes, i = x - t * kLanes, n = min(kLanes, nz - t * kLanes);
    o[0] = (g.toff32 + t) * kSlotF + i + 2;
    if (i < 2) {
      const int tl = t == 0 ? nt - 1 : t - 1;
      o[1] = (g.toff32 + tl) * kSlotF + min(kLanes, nz - tl * kLanes) + 2 + i;
    }
    if (i >= n - 2) {
      const int tr = t == nt - 1 ? 0 : t + 1;
      o[2] = (g.toff32 + tr) * kSlotF + i - n + 2;
    }
    return;
  }
  int cnt = 0;
  int prev[4] = {-1, -1, -1, -1};
#pragma unroll
  for (int d = -2; d <= 2; ++d) {
    const int tau = wrapc(x + d, nz) / kLanes;
    bool seen = false;
#pragma unroll
    for (int q = 0; q < d + 2; ++q) seen |= prev[q] == tau;
    if (d < 2) prev[d + 2] = tau;
    if (seen) continue;
    const int ntau = min(kLanes, nz - tau * kLanes);
    const int base = (g.toff32 + tau) * kSlotF;
    for (int k = wrapc(x - tau * kLanes + 2, nz); k < ntau + 4; k += nz) {
#pragma unroll
      for (int q = 0; q < 5; ++q)
        if (q == cnt) o[q] = base + k;
      ++cnt;
    }
  }
}

// Value of component row r of the potential from its frame entries.
__device__ __forceinline__ double frame_value(const double* __restrict__ Fr, const int (&o)[5], int r) {
  double v = __ldg(Fr + o[0] + r * kFrame);
#pragma unroll
  for (int q = 1; q < 5; ++q)
    if (o[q] >= 0) v += __ldg(Fr + o[q] + r * kFrame);
  return v;
}

// Stage s (1..4) of every box: the RK4 update of k_rk_stage (its commutators
// and update; interpolation in FP64; the potential of a cell is the sum of the frame entries of
// k_frame_sum that cover it, Fr), then the
// deposit of its result at the next stage's positions: the shape weights
// (kept in W for the next stage), B = N rho - Nbar rhobar^* in the traceless
// components (Eq. 5, Eq. 2) and w (1, Omega) B summed per frame cell.
// STAGE 0: no RK update; the deposit of the state in rho, rhobar at the first
// stage's positions (the first launch of a run of steps).  Shift rows: this
// stage's s - 1, the deposit's s (row 4: the next step's first stage).  The
// stage is a template parameter: each instance keeps only its own stage's
// loads live (fewer registers than one kernel for all four).
template <bool POT, int ORDER, int STAGE>
__global__ void __launch_bounds__(kThreads, 2)
k_rk_deposit(Batch B, Parts pt, double* __restrict__ W, const double* __restrict__ dirtab,
             const int* __restrict__ shift, const double* __restrict__ Fr, int dry,
             double* __restrict__ partial, int* __restrict__ err) {
  static_assert(Sten<ORDER>::H == 1, "the frame covers the shapes of one cell of reach");
  static_assert(STAGE >= 0 && STAGE <= 4, "stages 1-4, or 0 for the first deposit");
  constexpr bool DEP_ONLY = STAGE == 0;
  constexpr int s = STAGE;
  constexpr int NW = Sten<ORDER>::NW, NWS = Sten<ORDER>::NWS;
  extern __shared__ double frame_sm[];
  __shared__ double gsm[kWarps][kNC][kLanes];   // G of the unit's cells
  __shared__ double gedge[kWarps][2 * kNC];      // G left of lane 0, right of lane n - 1
  griddep_wait();
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
  double* acc = frame_sm + wib * kSlotF;
  const int64_t w = logical_warp();
  const int64_t u0 = unit32_begin(w, B), u1 = unit32_begin(w + 1, B);
  if (u0 >= u1) return;
  for (int k = lane; k < kSlotF; k += kLanes) acc[k] = 0.0;
  __syncwarp();
  const int64_t P = B.Ptot;
  const int MT = B.MT;
  const bool first = DEP_ONLY || s == 1;
  const double* src_r = first ? pt.rho : pt.stage;
  const double* src_b = first ? pt.rhobar : pt.stage + 9 * P;
  const int* sh_cur = shift + (DEP_ONLY ? 0 : s - 1) * MT;
  const int* sh_next = shift + (DEP_ONLY ? 0 : s) * MT;
  // arrays read per particle, for the L2 prefetch of the next unit: the state
  // (18), y (18, s = 2, 3), acc (18, s >= 2), W (NWS), z, N, Nbar
  const int ny = (!DEP_ONLY && (s == 2 || s == 3)) ? 18 : 0, nacc = (!DEP_ONLY && s >= 2) ? 18 : 0;
  const int nw_ = DEP_ONLY ? 0 : NWS;
  const int narr = 18 + ny + nacc + nw_ + 3;
  int lat = 0, far = 0;
  int b = box_of_unit32(B, u0);
  int bcur = -1;
  double dtb = 0.0, bdt = 0.0, cdt = 0.0;
  int64_t stile = -1;   // global tile whose sums acc holds
  for (int64_t u = u0; u < u1; ++u) {
    while (u >= B.box[b].uoff32 + (int64_t)B.box[b].ntiles32 * B.box[b].M) ++b;
    const BoxGeo& g = B.box[b];
    const int nz = g.nz, M = g.M;
    const int lu = (int)(u - g.uoff32);
    const int tile = lu / M, d = lu - tile * M;
    const int64_t gtile = g.toff32 + tile;
    if (gtile != stile) {
      if (stile >= 0) flush_frame(acc, partial + (w + stile) * kSlotF, lane);
      stile = gtile;
    }
    if (b != bcur) {
      bcur = b;
      dtb = B.dt[b];
      rk_coefficients(s, dtb, bdt, cdt);
    }
    if (u + 1 < u1 && lu + 1 < g.ntiles32 * M) {   // prefetch the next unit of the same box
      const int tn = (lu + 1) / M, dn = lu + 1 - tn * M;
      const int i0 = tn * kLanes - __ldg(sh_cur + g.doff + dn);
      const int cnt = min(kLanes, nz - tn * kLanes);
      if (i0 >= 0 && i0 + cnt <= nz) {
        const int64_t base = g.poff + (int64_t)dn * nz + i0;
        prefetch_l2(lane, narr, base, cnt, [&](int a) {
          const double* arr;
          if (a < 18) arr = a < 9 ? src_r + (int64_t)a * P : src_b + (int64_t)(a - 9) * P;
          else if (a < 18 + ny) arr = a - 18 < 9 ? pt.rho + (int64_t)(a - 18) * P : pt.rhobar + (int64_t)(a - 27) * P;
          else if (a < 18 + ny + nacc) arr = pt.acc + (int64_t)(a - 18 - ny) * P;
          else if (a < 18 + ny + nacc + nw_) arr = W + (int64_t)(a - 18 - ny - nacc) * P;
          else {
            const int k = a - 18 - ny - nacc - nw_;
            arr = k == 0 ? pt.z : k == 1 ? pt.N : pt.Nbar;
          }
          return arr;
        });
      }
    }
    const int n = min(kLanes, nz - tile * kLanes);
    const bool active = lane < n;
    const int j = tile * kLanes + lane;   // this lane's cell at the stage's positions
    const int gd = g.doff + d;
    const double ox = __ldg(dirtab + gd), oy = __ldg(dirtab + MT + gd), oz = __ldg(dirtab + 2 * MT + gd);
    const double vz = __ldg(dirtab + 3 * MT + gd);
    const int sc = __ldg(sh_cur + gd);
    const int64_t p = g.poff + (int64_t)d * nz + wrapc(j - sc, nz);
    double bm[9];       // B = N rho - Nbar rhobar^* of the state deposited (Eq. 5)
    double zs = 0.0;    // and its position
    double n1 = 0.0, n2 = 0.0;
    if (active) {
      n1 = __ldg(pt.N + p);
      n2 = __ldg(pt.Nbar + p);
    }
    if constexpr (DEP_ONLY) {
      if (active) {
#pragma unroll
        for (int k = 0; k < 9; ++k) {
          const double x = __ldg(src_r + k * P + p), y = __ldg(src_b + k * P + p);
          bm[k] = (k == 4 || k == 6 || k == 8) ? fma(n2, y, n1 * x) : fma(-n2, y, n1 * x);
        }
        zs = __ldg(pt.z + p);
      }
    } else {
      // G = A0 - Omega . A of this lane's cell into shared memory
      if (frame_fast(g)) {
        // its tile's frame entry lane + 2, then (one value per lane) the
        // adjacent tiles' entries for the two cells at each end of the tile:
        // lanes 0-15 cells 0, 1 from the tile before, lanes 16-31 cells
        // n - 2, n - 1 from the tile after, added in that order
        const double* f0 = Fr + (int64_t)(g.toff32 + tile) * kSlotF + lane + 2;
#pragma unroll
        for (int c = 0; c < kNC; ++c)
          gsm[wib][c][lane] = fma(-oz, __ldg(f0 + (3 * kNC + c) * kFrame),
                                  fma(-oy, __ldg(f0 + (2 * kNC + c) * kFrame),
                                      fma(-ox, __ldg(f0 + (kNC + c) * kFrame), __ldg(f0 + c * kFrame))));
        const int nt = g.ntiles32, c = lane & (kNC - 1), right = lane >> 4;
        const int ce = right ? n - 2 + ((lane >> 3) & 1) : (lane >> 3) & 1;
        const int tn = right ? (tile == nt - 1 ? 0 : tile + 1) : (tile == 0 ? nt - 1 : tile - 1);
        const int k = right ? ce - n + 2 : min(kLanes, nz - tn * kLanes) + 2 + ce;
        const double* f1 = Fr + (int64_t)(g.toff32 + tn) * kSlotF + k;
        const double gc = fma(-oz, __ldg(f1 + (3 * kNC + c) * kFrame),
                              fma(-oy, __ldg(f1 + (2 * kNC + c) * kFrame),
                                  fma(-ox, __ldg(f1 + (kNC + c) * kFrame), __ldg(f1 + c * kFrame))));
        __syncwarp();
        if (!right) gsm[wib][c][ce] += gc;
        __syncwarp();
        if (right) gsm[wib][c][ce] += gc;
      } else {
        int off[5];
        frame_sources(g, active ? j : wrapc(j, nz), off);
#pragma unroll
        for (int c = 0; c < kNC; ++c)
          gsm[wib][c][lane] = fma(-oz, frame_value(Fr, off, 3 * kNC + c),
                                  fma(-oy, frame_value(Fr, off, 2 * kNC + c),
                                      fma(-ox, frame_value(Fr, off, kNC + c), frame_value(Fr, off, c))));
      }
      // lanes 0-15 (component lane mod 8): G of the cell left of lane 0
      // (lanes 0-7) and right of lane n - 1 (lanes 8-15)
      if (ORDER > 0 && lane < 2 * kNC) {
        const int c = lane & (kNC - 1);
        const int right = tile * kLanes + n;
        const int cell = lane < kNC ? (tile == 0 ? nz - 1 : tile * kLanes - 1) : (right == nz ? 0 : right);
        int off[5];
        frame_sources(g, cell, off);
        gedge[wib][lane] = fma(-oz, frame_value(Fr, off, 3 * kNC + c),
                               fma(-oy, frame_value(Fr, off, 2 * kNC + c),
                                   fma(-ox, frame_value(Fr, off, kNC + c), frame_value(Fr, off, c))));
      }
      __syncwarp();
      if (active) {
        double wt[NW];
        double r[9];
        load_weights<ORDER>(W, P, p, wt);
#pragma unroll
        for (int k = 0; k < 9; ++k) r[k] = src_r[k * P + p];
        double Hm[kNC];
#pragma unroll
        for (int c = 0; c < kNC; ++c) {
          if constexpr (ORDER == 0) {
            Hm[c] = gsm[wib][c][lane];
          } else {
            const double gl = lane == 0 ? gedge[wib][c] : gsm[wib][c][lane - 1];
            const double gr = lane == n - 1 ? gedge[wib][kNC + c] : gsm[wib][c][lane + 1];
            Hm[c] = fma(wt[0], gl, fma(wt[1], gsm[wib][c][lane], wt[2] * gr));
          }
        }
        double zn = 0.0;
        rk_particle<POT, s == 3 ? 2 : s, false, true>(g, pt, src_b, P, p, dry, bdt, cdt, dtb, dirtab + 3 * MT + gd, Hm, r,
                                      bm, &zn, n1, n2);
        zs = s < 4 ? fma(stage_frac(s) * dtb, vz, pt.z[p]) : zn;
      }
      __syncwarp();   // (gsm is rewritten by the next unit)
    }
    // the ring's move to the next stage's positions
    int delta = 0;
    if constexpr (!DEP_ONLY) {
      delta = wrapc(__ldg(sh_next + gd) - sc, nz);
      if (2 * delta > nz) delta -= nz;
      if (delta < -1 || delta > 1) {   // (excluded by the host; the unit's deposit is skipped)
        far = 1;
        continue;
      }
    }
    double wn[NW];
    zero_weights<ORDER>(wn);
    double bv[kNC];
#pragma unroll
    for (int c = 0; c < kNC; ++c) bv[c] = 0.0;
    if (active) {
      lat |= shape_weights<ORDER>(zs, (double)wrapc(j + delta, nz) + 0.5, g.inv_dz, g.nz_d, wn);
#pragma unroll
      for (int q = 0; q < NWS; ++q) W[q * P + p] = wn[q];
      bv[0] = bm[0] - bm[1];   // the traceless components
      bv[1] = bm[1] - bm[2];
#pragma unroll
      for (int k = 3; k < 9; ++k) bv[k - 1] = bm[k];
    }
    // this lane's cell tile * 32 + lane + delta receives from the particles on
    // lanes lane - 1, lane, lane + 1 of this unit
    const double wup = __shfl_up_sync(kFull, wn[2], 1), wdn = __shfl_down_sync(kFull, wn[0], 1);
    const double fl = lane == 0 ? 0.0 : wup;
    const double fr = lane == kLanes - 1 ? 0.0 : wdn;
    double* a = acc + lane + delta + 2;
#pragma unroll
    for (int c = 0; c < kNC; ++c) {
      const double v = bv[c];
      double cc;
      if constexpr (ORDER == 0) {
        cc = wn[1] * v;
      } else {
        const double vl = __shfl_up_sync(kFull, v, 1), vr = __shfl_down_sync(kFull, v, 1);
        cc = fma(fr, vr, fma(wn[1], v, fl * vl));
      }
      if (active) {
        a[c * kFrame] += cc;
        a[(kNC + c) * kFrame] = fma(ox, cc, a[(kNC + c) * kFrame]);
        a[(2 * kNC + c) * kFrame] = fma(oy, cc, a[(2 * kNC + c) * kFrame]);
        a[(3 * kNC + c) * kFrame] = fma(oz, cc, a[(3 * kNC + c) * kFrame]);
      }
    }
    if constexpr (ORDER > 0) {
      // the cells left of lane 0's and right of lane n - 1's: only those two
      // particles' outer weights; lane f * 8 + c adds component c of moment f
      // (1, Omega_x, Omega_y, Omega_z) of both
      __syncwarp();
      const int c = lane & (kNC - 1), f = lane >> 3;
      double bl = 0.0, br = 0.0;
#pragma unroll
      for (int k = 0; k < kNC; ++k) {
        const double x0 = __shfl_sync(kFull, bv[k], 0), x1 = __shfl_sync(kFull, bv[k], n - 1);
        if (k == c) {
          bl = x0;
          br = x1;
        }
      }
      const double wl = __shfl_sync(kFull, wn[0], 0), wr = __shfl_sync(kFull, wn[2], n - 1);
      const double of = f == 0 ? 1.0 : f == 1 ? ox : f == 2 ? oy : oz;
      double* row = acc + lane * kFrame;
      row[delta + 1] = fma(of, wl * bl, row[delta + 1]);
      row[n + delta + 2] = fma(of, wr * br, row[n + delta + 2]);
    }
    __syncwarp();
  }
  flush_frame(acc, partial + (w + stile) * kSlotF, lane);
  if (lat) atomicOr(err, lat);
  if (far) atomicOr(err, ERR_STEP);
}

__device__ __forceinline__ int box_of_tile32(const Batch& B, int64_t t) {
  int lo = 0, hi = B.nbox - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (B.box[mid].toff32 <= t) lo = mid; else hi = mid - 1;
  }
  return lo;
}

// Deposit combination of step form 2: the frame sums of every 32-cell tile,
// Fr[gtile * kSlotF + e] = kappa_b / dV_b x (sum over the warps that own
// units of the tile of their slot's entry e), in warp order.  A group of 32
// lanes takes 32 consecutive entries of one tile (kSlotF = 36 x 32), so every
// lane of a warp walks the same warps.  Split over warps and running sums as
// in combine_phase.  The potential at a cell is the sum of the frame entries
// that cover it (frame_sources).
static __global__ void k_frame_sum(Batch B, const double* __restrict__ partial, double* __restrict__ Fr, int64_t NT32,
                            int split, int* __restrict__ err) {
  __shared__ double sums[kWarps][kLanes];
  griddep_wait();
  const int64_t n = NT32 * kSlotF;
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
  const int grp = wib / split, wi = wib - grp * split;
  const int groups = kWarps / split;
  int bad = 0;
  for (int64_t base = (int64_t)blockIdx.x * groups * kLanes; base < n; base += (int64_t)gridDim.x * groups * kLanes) {
    const int64_t e0 = base + (int64_t)grp * kLanes;   // first entry of this group (one tile)
    double v = 0.0;
    const BoxGeo* g = nullptr;
    if (e0 < n) {
      const int64_t gtile = e0 / kSlotF;
      g = &B.box[box_of_tile32(B, gtile)];
      const int64_t tau = gtile - g->toff32;
      const int64_t wf = warp_of_unit32(g->uoff32 + tau * g->M, B);
      const int64_t wl = warp_of_unit32(g->uoff32 + (tau + 1) * g->M - 1, B);
      const double* src = partial + (e0 - gtile * kSlotF) + lane;
      double a[kCombineILP] = {};
      int64_t q = wf + wi;
      for (; q + (kCombineILP - 1) * split <= wl; q += kCombineILP * split) {
#pragma unroll
        for (int i = 0; i < kCombineILP; ++i) a[i] += __ldcg(src + (q + i * split + gtile) * kSlotF);
      }
      for (; q <= wl; q += split) a[0] += __ldcg(src + (q + gtile) * kSlotF);
#pragma unroll
      for (int h = kCombineILP / 2; h >= 1; h /= 2) {
#pragma unroll
        for (int i = 0; i < h; ++i) a[i] += a[i + h];
      }
      v = a[0];
    }
    if (split > 1) {
      sums[wib][lane] = v;
      __syncthreads();
      if (wi == 0)
        for (int i = 1; i < split; ++i) v += sums[wib + i][lane];
      __syncthreads();
    }
    if (e0 < n && wi == 0) {
      v *= g->kappa_dV;
      bad |= !isfinite(v);
      Fr[e0 + lane] = v;
    }
  }
  if (bad) atomicOr(err, ERR_NONFINITE);
}

// ------------------------------------------------------- fused step kernel
//
// All phases of nsteps RK4 steps in one cooperative launch (every block
// resident): per step the lattice shifts and ring weights, then per stage the
// deposit, its combination and the RK stage, separated by grid barriers.  The
// arithmetic and the order of every sum are those of the separate kernels with
// the same grid: results are bitwise the same.
//
// Grid barrier: each block's thread 0 adds to an arrival word (block 0 adds
// 2^31 - (blocks - 1), the others 1, so the top bit flips when the last block
// arrives and the word is ready for the next barrier) and waits for the flip.
// The wait is bounded: after limit_ns nanoseconds (device global timer), or as
// soon as another block has given up, the block sets the abort word and
// ERR_TIMEOUT and the kernel returns.  A launch that finds the abort word set
// returns at once; the host clears it (and the arrival word) when it reports
// the error.
enum : int { ERR_TIMEOUT = 16 };

struct StepArgs {
  const double* dirtab;
  int* shift;          // [4][MT] shift rows of the step
  double* wtab;        // [4 x kWSlots][MT] the rings' weights at those rows (nullptr: each particle's own)
  double* W;           // kept shape weights
  double* At;          // traceless grid potential
  double* partial;     // per-warp deposit partials
  int* err;
  unsigned* bar;       // [0] arrival word, [1] abort word
  unsigned long long limit_ns;
  int64_t nsteps;
  int split;           // combine split (as the separate deposit uses)
  int dry;
};

__device__ __forceinline__ unsigned ld_acquire_u32(const unsigned* p) {
  unsigned v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

__device__ __forceinline__ unsigned long long global_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

// Returns true if the launch must stop (a wait gave up here or elsewhere).
__device__ __forceinline__ bool grid_barrier(unsigned* bar, unsigned long long limit_ns, int* err) {
  __shared__ int stop;
  __syncthreads();
  if (threadIdx.x == 0) {
    int give_up = 0;
    const unsigned inc = blockIdx.x == 0 ? 0x80000000u - (gridDim.x - 1) : 1u;
    __threadfence();                         // this block's writes before its arrival
    const unsigned old = atomicAdd(bar, inc);
    const unsigned long long t0 = global_ns();
    while (((old ^ ld_acquire_u32(bar)) & 0x80000000u) == 0) {
      if (ld_acquire_u32(bar + 1) != 0u || global_ns() - t0 > limit_ns) {
        atomicExch(bar + 1, 1u);
        atomicOr(err, ERR_TIMEOUT);
        give_up = 1;
        break;
      }
    }
    __threadfence();                         // the other blocks' writes after the barrier
    stop = give_up;
  }
  __syncthreads();
  return stop != 0;
}

// The phases of the fused kernel, inlined (measured on GB300: calling them as
// separate functions, which keeps each phase's register allocation but saves
// and restores registers around every call, was 4-5% slower per step).
template <int ORDER>
__device__ __forceinline__ void fused_deposit(const Batch& B, int64_t w, int lane, const Parts& pt, const double* rnu,
                                           const double* rnb, const StepArgs& a, const int* srow,
                                           const double* wrow, double frac, double* buf) {
  double* W = wrow != nullptr ? nullptr : a.W;
  if (B.dpb > 0)
    deposit_phase<5, ORDER, true, true>(B, w, lane, pt.z, pt.N, pt.Nbar, rnu, rnb, a.dirtab, srow, wrow, frac,
                                        a.partial, W, a.err, buf);
  else
    deposit_phase<5, ORDER, true, false>(B, w, lane, pt.z, pt.N, pt.Nbar, rnu, rnb, a.dirtab, srow, wrow, frac,
                                         a.partial, W, a.err, buf);
}

__device__ __forceinline__ void fused_combine(const Batch& B, const StepArgs& a) {
  combine_phase(B, a.partial, a.At, kNT, 1, a.split, a.err);
}

template <bool POT, int ORDER>
__device__ __forceinline__ void fused_rk(const Batch& B, const Parts& pt, const StepArgs& a, const int* srow,
                                         const double* wrow, int s, SlabTable<kSlabTiles>& t) {
  if (s == 1) rk_phase<POT, ORDER, 1, true>(B, pt, a.W, wrow, a.dirtab, srow, a.At, pt.stage, s, a.dry, t);
  else if (s == 4) rk_phase<POT, ORDER, 4, true>(B, pt, a.W, wrow, a.dirtab, srow, a.At, pt.stage, s, a.dry, t);
  else rk_phase<POT, ORDER, 2, true>(B, pt, a.W, wrow, a.dirtab, srow, a.At, pt.stage, s, a.dry, t);
}

template <bool POT, int ORDER>
__global__ void __launch_bounds__(kThreads, 2) k_step(Batch B, Parts pt, StepArgs a) {
  extern __shared__ char smem[];   // the deposit's buffers, then the RK stage's table
  __shared__ int aborted;
  if (threadIdx.x == 0) aborted = ld_acquire_u32(a.bar + 1) != 0u;
  __syncthreads();
  if (aborted) return;
  const int lane = threadIdx.x & 31;
  const int64_t w = logical_warp();
  const int MT = B.MT;
  Fracs fr;
#pragma unroll
  for (int q = 0; q < 4; ++q) fr.v[q] = stage_frac(q);
  const int64_t P = B.Ptot;
  for (int64_t n = 0; n < a.nsteps; ++n) {
    for (int gd = blockIdx.x * blockDim.x + threadIdx.x; gd < MT; gd += gridDim.x * blockDim.x)
      shifts_phase<true, ORDER>(B, gd, pt.z, a.dirtab, fr, 4, a.shift, a.wtab);
    if (grid_barrier(a.bar, a.limit_ns, a.err)) return;
    for (int s = 1; s <= 4; ++s) {
      const int* srow = a.shift + (s - 1) * MT;
      const double* wrow = a.wtab != nullptr ? a.wtab + (s - 1) * kWSlots * MT : nullptr;
      const double* rnu = s == 1 ? pt.rho : pt.stage;
      const double* rnb = s == 1 ? pt.rhobar : pt.stage + 9 * P;
      fused_deposit<ORDER>(B, w, lane, pt, rnu, rnb, a, srow, wrow, stage_frac(s - 1),
                           (double*)smem + (threadIdx.x >> 5) * kDepBuf);
      if (grid_barrier(a.bar, a.limit_ns, a.err)) return;
      fused_combine(B, a);
      if (grid_barrier(a.bar, a.limit_ns, a.err)) return;
      fused_rk<POT, ORDER>(B, pt, a, srow, wrow, s, *(SlabTable<kSlabTiles>*)smem);
      if (grid_barrier(a.bar, a.limit_ns, a.err)) return;
    }
  }
}

// SplitMix64 (Steele, Lea & Flood, OOPSLA 2014): n-th output of the generator
// whose state starts at `seed`.
__device__ __forceinline__ uint64_t splitmix64(uint64_t seed, uint64_t n) {
  uint64_t x = seed + n * 0x9E3779B97F4A7C15ULL;
  x = (x ^ (x >> 30)) * 0xBF58476D1CE4E5B9ULL;
  x = (x ^ (x >> 27)) * 0x94D049BB133111EBULL;
  return x ^ (x >> 31);
}

__device__ __forceinline__ double uniform_pm1(uint64_t seed, int64_t p, int k) {
  const uint64_t h = splitmix64(seed, (uint64_t)p * 8u + (uint64_t)k + 1u);
  return 2.0 * ((double)(h >> 11) * 0x1.0p-53) - 1.0;
}

// Initial particles (Sec. 3.1): cell-centre lattice, weights of Eq. 8, flavour
// state of Eq. 9 (eps_x = |rho_ex|^2, rho_mutau = 0).  Plain roundings (no
// fused multiply-add) so the weights and states round like the formulas read.
// Box-local particle numbers key the random draws.  species: per box, at
// 8 * coff_b: n_nu[nz], n_nubar[nz], f_nu[3 nz], f_nubar[3 nz]; dirs[3 * MT].
static __global__ void k_init(Batch B, Parts pt, const double* __restrict__ species, const double* __restrict__ dirs,
                       int* __restrict__ err) {
  const int64_t gp = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (gp >= B.Ptot) return;
  const BoxGeo& g = B.box[box_of_particle(B, gp)];
  const int64_t p = gp - g.poff;
  const int d = (int)(p / g.nz), j0 = (int)(p % g.nz);
  double o[3];
  if (g.use_dirs) {
    const int gd = g.doff + d;
    o[0] = dirs[3 * gd]; o[1] = dirs[3 * gd + 1]; o[2] = dirs[3 * gd + 2];
  } else {
    const double mu = __dsub_rn(1.0, __ddiv_rn(__dadd_rn(__dmul_rn(2.0, (double)d), 1.0), (double)g.M));
    const double phi = __dmul_rn(__dmul_rn((double)d, 3.14159265358979323846), __dsub_rn(3.0, sqrt(5.0)));
    const double sn = sqrt(__dsub_rn(1.0, __dmul_rn(mu, mu)));
    o[0] = __dmul_rn(sn, cos(phi));
    o[1] = __dmul_rn(sn, sin(phi));
    o[2] = mu;
  }
  pt.z[gp] = __dmul_rn(__dadd_rn((double)j0, 0.5), g.dz);
  pt.ox[gp] = o[0]; pt.oy[gp] = o[1]; pt.oz[gp] = o[2];
  const int nz = g.nz;
  const double* sp_base = species + 8 * (int64_t)g.coff;
  double wgt[2];
  for (int sp = 0; sp < 2; ++sp) {
    const double n = sp_base[sp * nz + j0];
    const double* f = sp_base + 2 * nz + sp * 3 * nz + 3 * j0;
    const double fdo = __dadd_rn(__dadd_rn(__dmul_rn(f[0], o[0]), __dmul_rn(f[1], o[1])), __dmul_rn(f[2], o[2]));
    double wt = __ddiv_rn(__dmul_rn(__dadd_rn(n, __dmul_rn(3.0, fdo)), g.dV), (double)g.M);
    const double tol = 1e-12 * (fabs(n) + 3.0 * fabs(fdo)) * g.dV / g.M;
    if (wt < 0.0 && wt >= -tol) wt = 0.0;
    if (wt < 0.0) atomicOr(err, ERR_WEIGHT);
    wgt[sp] = wt;
  }
  pt.N[gp] = wgt[0];
  pt.Nbar[gp] = wgt[1];
  const int64_t P = B.Ptot;
  for (int sp = 0; sp < 2; ++sp) {
    double* r = sp ? pt.rhobar : pt.rho;
    const double emr = __dmul_rn(g.alpha, uniform_pm1(g.seed, p, 4 * sp + 0));
    const double emi = __dmul_rn(g.alpha, uniform_pm1(g.seed, p, 4 * sp + 1));
    const double etr = __dmul_rn(g.alpha, uniform_pm1(g.seed, p, 4 * sp + 2));
    const double eti = __dmul_rn(g.alpha, uniform_pm1(g.seed, p, 4 * sp + 3));
    const double eps_mu = __dadd_rn(__dmul_rn(emr, emr), __dmul_rn(emi, emi));
    const double eps_tau = __dadd_rn(__dmul_rn(etr, etr), __dmul_rn(eti, eti));
    r[0 * P + gp] = __dsub_rn(__dsub_rn(1.0, eps_mu), eps_tau);
    r[1 * P + gp] = eps_mu;
    r[2 * P + gp] = eps_tau;
    r[3 * P + gp] = emr;
    r[4 * P + gp] = emi;
    r[5 * P + gp] = etr;
    r[6 * P + gp] = eti;
    r[7 * P + gp] = 0.0;
    r[8 * P + gp] = 0.0;
  }
}

// Per box: maximum over cells of the diagonal components of n and nbar (Eq. 7).
// One block per box.
static __global__ void k_max_diag(Batch B, const double* __restrict__ mom, double* __restrict__ out) {
  __shared__ double sm[kThreads];
  const BoxGeo& g = B.box[blockIdx.x];
  double m = 0.0;
  for (int j = threadIdx.x; j < g.nz; j += kThreads)
    for (int a = 0; a < 3; ++a) {
      m = fmax(m, mom[(int64_t)a * B.NZ + g.coff + j]);
      m = fmax(m, mom[(int64_t)(36 + a) * B.NZ + g.coff + j]);
    }
  sm[threadIdx.x] = m;
  __syncthreads();
  for (int w = kThreads / 2; w > 0; w >>= 1) {
    if (threadIdx.x < w) sm[threadIdx.x] = fmax(sm[threadIdx.x], sm[threadIdx.x + w]);
    __syncthreads();
  }
  if (threadIdx.x == 0) out[blockIdx.x] = sm[0];
}

// Eq. 7 per box from the maxima: dt_b = min(C dz / c, C_F / (kappa n_max)).
static __global__ void k_dt_from_max(Batch B, const double* __restrict__ nmax, double* __restrict__ dt_out) {
  const int b = blockIdx.x * blockDim.x + threadIdx.x;
  if (b >= B.nbox) return;
  const BoxGeo& g = B.box[b];
  const double dt_adv = g.cfl_adv * g.dz / g.c_light;
  const double nm = nmax[b] > g.n_e ? nmax[b] : g.n_e;
  const double dt_flav = nm > 0.0 ? g.cfl_flavor / (g.kappa * nm) : dt_adv;
  dt_out[b] = dt_adv < dt_flav ? dt_adv : dt_flav;
}

// Writes one box descriptor and step size from kernel parameters (used where
// no host-to-device copy may be issued).
static __global__ void k_write_geo(BoxGeo g, double dt, BoxGeo* __restrict__ dst, double* __restrict__ dt_dst) {
  *dst = g;
  *dt_dst = dt;
}

// Domain diagnostics per box (Eq. 10, one snapshot of Eq. B1, Eq. 18), fixed-
// order block reduction over the box's cells.  One block per (box, quantity):
// blockIdx.x = box, blockIdx.y = q; out[63 * b + q].  mom: the [36][NZ] moments
// of the diagnostic deposit (rows 0-8 n, 9-17 f_x, 18-26 nbar, 27-35 fbar_x).
__device__ __forceinline__ double abs_entry(const double* __restrict__ m, int64_t NZ, int64_t j, int a, int b) {
  if (a == b) return fabs(m[(int64_t)a * NZ + j]);
  const int lo = a < b ? a : b, hi = a < b ? b : a;
  const int k = (lo == 0 && hi == 1) ? 3 : (lo == 0 ? 5 : 7);
  const double re = m[(int64_t)k * NZ + j], im = m[(int64_t)(k + 1) * NZ + j];
  return sqrt(re * re + im * im);
}

static __global__ void k_diagnostics(Batch B, const double* __restrict__ mom, double* __restrict__ out) {
  __shared__ double sm[kThreads];
  const BoxGeo& g = B.box[blockIdx.x];
  const int64_t NZ = B.NZ;
  const int q = blockIdx.y;
  double s = 0.0;
  for (int jj = threadIdx.x; jj < g.nz; jj += kThreads) {
    const int64_t j = g.coff + jj;
    double v;
    if (q < 36) {
      const int blk = q / 9, e = q % 9, a = e / 3, bb = e % 3;
      const int off = blk == 0 ? 0 : blk == 1 ? 18 : blk == 2 ? 9 : 27;
      v = abs_entry(mom + (int64_t)off * NZ, NZ, j, a, bb);
    } else if (q < 45) {
      v = mom[(int64_t)(q - 36) * NZ + j];
    } else if (q < 54) {
      v = mom[(int64_t)(18 + q - 45) * NZ + j];
    } else {
      const int k = q - 54;
      const double nbar = mom[(int64_t)(18 + k) * NZ + j];
      v = mom[(int64_t)k * NZ + j] + ((k == 4 || k == 6 || k == 8) ? nbar : -nbar);
    }
    s += v;
  }
  sm[threadIdx.x] = s;
  __syncthreads();
  for (int w = kThreads / 2; w > 0; w >>= 1) {
    if (threadIdx.x < w) sm[threadIdx.x] += sm[threadIdx.x + w];
    __syncthreads();
  }
  if (threadIdx.x == 0) out[63 * blockIdx.x + q] = sm[0] / g.nz;
}

// ------------------------------------------------------------------ adjoint
//
// Discrete adjoint of the RK4 step in the packed 9-real representation.  With
// the packing metric D = diag(1, 1, 1, 2, ..., 2) (<X, Y>_Frobenius = x^T D y),
// K(H, r) = -i[H, r] and the sign pattern S of Hbar = -H^* (packed: S H):
//   transpose of r -> K(H, r):  m -> -D K(H, D^-1 m)   (the generator is anti-self-adjoint)
//   transpose of H -> K(H, r):  m -> D K(r, D^-1 m)
//   transpose of H -> K(S H + V, rbar):  m -> S D K(rbar, D^-1 m)
// The self-interaction operator B -> H (deposit, Eq. 5, then interpolation,
// Eq. 6, with the shared weights) is symmetric, so its transpose is the same
// deposit-and-interpolate applied to the adjoint Gamma = dL/dH.

// First adjoint launch of stage s.  m = a lam + c lamn, the adjoint of this
// stage's derivative k_s, with the box's step dt: a = dt/6 (s = 1, 4) or dt/3,
// c = dt/2 (s = 1, 2) or dt (s = 3), lamn the adjoint of stage s + 1 (NULL
// for s = 4); writes x.out = J_rho^T m (direct terms) and x.gam = dL/dH_self.
// pt.rho / pt.rhobar point at the stage state.  The metric D folds into the
// commutator: D K(X, D^-1 m) is the commutator's raw output (halved diagonal,
// off-diagonals) for X and m2 = m with its diagonal doubled, so
//   out = -D K(H, D^-1 m) = raw(-H, m2),   gam += S D K(r, D^-1 m) = S raw(r, m2).
// H is formed as in the RK stage (rk_phase: the same work split, tables and
// integer arithmetic; 48 of ~200 FP64 instructions less, the pipe that bounds it):
// 1024 x 1000, 24 steps, backward from records 103.8 -> 94.2 ms.
template <bool POT, int ORDER, int TILES>
__global__ void __launch_bounds__(kThreads, 2)
k_adj_a(Batch B, Parts pt, const double* __restrict__ W, const double* __restrict__ dirtab,
        const int* __restrict__ shift, const double* __restrict__ A, AdjStage x, int s) {
  extern __shared__ char smem[];
  griddep_wait();
  rk_phase<POT, ORDER, 0, false>(B, pt, W, nullptr, dirtab, shift, A, nullptr, s, 0, *(SlabTable<TILES>*)smem, x);
}

// Second adjoint launch of one stage: GB = interpolation of the deposited
// Gamma grid E (= dL/dB), then lam_out += N GB (rho) and -Nbar conj(GB)
// (rhobar), gN += <GB, rho>, gNbar -= <conj(GB), rhobar>; finally
// lam_tot += lam_out.
template <int ORDER>
__global__ void __launch_bounds__(kThreads, 2)
k_adj_b(Batch B, Parts pt, const double* __restrict__ W, const double* __restrict__ dirtab,
        const int* __restrict__ shift, const double* __restrict__ E, double* __restrict__ lam_out,
        double* __restrict__ lam_tot, double* __restrict__ gN, double* __restrict__ gNbar) {
  griddep_wait();
  const int lane = threadIdx.x & 31;
  const int64_t w = logical_warp();
  const int64_t u0 = unit_begin(w, B), u1 = unit_begin(w + 1, B);
  if (u0 >= u1) return;
  const int64_t P = B.Ptot;
  const int MT = B.MT, NZ = B.NZ;
  constexpr int Hh = Sten<ORDER>::H, T = Sten<ORDER>::T, NWS = Sten<ORDER>::NWS;
  const double* __restrict__ rho = pt.rho;
  const double* __restrict__ rhobar = pt.rhobar;
  const double* __restrict__ Nw = pt.N;
  const double* __restrict__ Nbw = pt.Nbar;
  // arrays read per particle, for the L2 prefetch of the next unit: rho, rhobar (18),
  // lam_out, lam_tot (36), N, Nbar, gN, gNbar (4), weights (NWS)
  constexpr int narr = 18 + 36 + 4 + NWS;
  int b = box_of_unit(B, u0);
  for (int64_t u = u0; u < u1; ++u) {
    while (u >= B.box[b].uoff + (int64_t)B.box[b].ntiles * B.box[b].M) ++b;
    const BoxGeo& g = B.box[b];
    const int nz = g.nz, nt = g.ntiles;
    const int lu = (int)(u - g.uoff);
    const int d = lu / nt, tile = lu - d * nt;
    if (u + 1 < u1 && lu + 1 < nt * g.M) {   // prefetch the next unit of the same box (same ring or the next)
      const int dn = (lu + 1) / nt, tn = lu + 1 - dn * nt;
      const int i0 = tn * T - __ldg(shift + g.doff + dn);
      const int n = min(T, nz - tn * T);
      if (i0 >= 0 && i0 + n <= nz) {
        const int64_t base = g.poff + (int64_t)dn * nz + i0;
        prefetch_l2(lane, narr, base, n, [&](int a) {
          const double* arr;
          if (a < 9) arr = rho + (int64_t)a * P;
          else if (a < 18) arr = rhobar + (int64_t)(a - 9) * P;
          else if (a < 36) arr = lam_out + (int64_t)(a - 18) * P;
          else if (a < 54) arr = lam_tot + (int64_t)(a - 36) * P;
          else if (a == 54) arr = Nw;
          else if (a == 55) arr = Nbw;
          else if (a == 56) arr = gN;
          else if (a == 57) arr = gNbar;
          else arr = W + (int64_t)(a - 58) * P;
          return arr;
        });
      }
    }
    const int craw = tile * T - Hh + lane, j = wrapc(craw, nz);
    const bool active = lane >= Hh && lane < Hh + T && craw < nz;
    const int gd = g.doff + d;
    const double ox = __ldg(dirtab + gd), oy = __ldg(dirtab + MT + gd), oz = __ldg(dirtab + 2 * MT + gd);
    const int64_t p = g.poff + (int64_t)d * nz + wrapc(j - __ldg(shift + gd), nz);
    double wt[Sten<ORDER>::NW];
    zero_weights<ORDER>(wt);
    double n1 = 0.0, n2 = 0.0;
    if (active) {
      load_weights<ORDER>(W, P, p, wt);
      n1 = Nw[p];
      n2 = Nbw[p];
    }
    double GB[9];
    const double* Ej = E + g.coff + j;
#pragma unroll
    for (int k = 0; k < 9; ++k) {
      const double G = fma(-oz, __ldg(Ej + (int64_t)(27 + k) * NZ),
                           fma(-oy, __ldg(Ej + (int64_t)(18 + k) * NZ),
                               fma(-ox, __ldg(Ej + (int64_t)(9 + k) * NZ), __ldg(Ej + (int64_t)k * NZ))));
      GB[k] = gather<ORDER>(wt, G);
    }
    if (!active) continue;
    // neutrinos, then antineutrinos: every load of a half before its stores
#pragma unroll
    for (int which = 0; which < 2; ++which) {
      const double* __restrict__ r = which ? rhobar : rho;
      double rv[9], lo[9], lt[9];
#pragma unroll
      for (int k = 0; k < 9; ++k) {
        rv[k] = r[k * P + p];
        lo[k] = lam_out[(which * 9 + k) * P + p];
        lt[k] = lam_tot[(which * 9 + k) * P + p];
      }
      double sum = 0.0;
#pragma unroll
      for (int k = 0; k < 9; ++k) {
        // B = N rho - Nbar conj(rhobar): dB/drhobar = -Nbar conj(.), conjugation
        // flipping the imaginary components 4, 6, 8
        const double sg = which ? ((k == 4 || k == 6 || k == 8) ? 1.0 : -1.0) : 1.0;
        const double l = fma((which ? n2 : n1) * sg, GB[k], lo[k]);
        lam_out[(which * 9 + k) * P + p] = l;
        lam_tot[(which * 9 + k) * P + p] = lt[k] + l;
        sum = fma(sg * GB[k], rv[k], sum);
      }
      if (which) gNbar[p] += sum;
      else gN[p] += sum;
    }
  }
}

// Adjoint seed from a loss on the moments at the current positions: with
// dmom = dL/d(mom) on the [72][NZ] layout of the moments (Eq. 5 per species),
//   lam_rho,p    = N_p    (1/dV) sum_j w_pj (dmom_n,j    + Omega_p . dmom_f,j)
//   lam_rhobar,p = Nbar_p (1/dV) sum_j w_pj (dmom_nbar,j + Omega_p . dmom_fbar,j)
// and gN_p += lam_rho,p . rho_p / N_p (likewise gNbar); lam is overwritten.
template <int ORDER>
__global__ void __launch_bounds__(kThreads, 2)
k_adj_seed(Batch B, Parts pt, const double* __restrict__ dirtab, const int* __restrict__ shift,
           const double* __restrict__ dmom, double* __restrict__ lam, double* __restrict__ gN,
           double* __restrict__ gNbar, int* __restrict__ err) {
  const int lane = threadIdx.x & 31;
  const int64_t w = logical_warp();
  const int64_t u0 = unit_begin(w, B), u1 = unit_begin(w + 1, B);
  if (u0 >= u1) return;
  const int64_t P = B.Ptot;
  const int MT = B.MT, NZ = B.NZ;
  int bad = 0;
  int b = box_of_unit(B, u0);
  for (int64_t u = u0; u < u1; ++u) {
    while (u >= B.box[b].uoff + (int64_t)B.box[b].ntiles * B.box[b].M) ++b;
    const BoxGeo& g = B.box[b];
    const int nz = g.nz, nt = g.ntiles;
    const int lu = (int)(u - g.uoff);
    const int d = lu / nt, tile = lu - d * nt;
    constexpr int Hh = Sten<ORDER>::H, T = Sten<ORDER>::T;
    const int craw = tile * T - Hh + lane, j = wrapc(craw, nz);
    const bool active = lane >= Hh && lane < Hh + T && craw < nz;
    const int gd = g.doff + d;
    const double ox = __ldg(dirtab + gd), oy = __ldg(dirtab + MT + gd), oz = __ldg(dirtab + 2 * MT + gd);
    const int64_t p = g.poff + (int64_t)d * nz + wrapc(j - __ldg(shift + gd), nz);
    double wt[Sten<ORDER>::NW];
    zero_weights<ORDER>(wt);
    if (active) bad |= shape_weights<ORDER>(pt.z[p], (double)j + 0.5, g.inv_dz, g.nz_d, wt);
    const double* Ej = dmom + g.coff + j;
#pragma unroll
    for (int which = 0; which < 2; ++which) {
      const int64_t base = which * kNA;
      double GB[9];
#pragma unroll
      for (int k = 0; k < 9; ++k) {
        const double G = fma(oz, __ldg(Ej + (base + 27 + k) * NZ),
                             fma(oy, __ldg(Ej + (base + 18 + k) * NZ),
                                 fma(ox, __ldg(Ej + (base + 9 + k) * NZ), __ldg(Ej + (base + k) * NZ))));
        GB[k] = gather<ORDER>(wt, G) * g.inv_dV;
      }
      if (active) {
        const double Nw = which ? pt.Nbar[p] : pt.N[p];
        const double* r = which ? pt.rhobar : pt.rho;
        double sN = 0.0;
#pragma unroll
        for (int k = 0; k < 9; ++k) {
          lam[(which * 9 + k) * P + p] = Nw * GB[k];
          sN = fma(GB[k], r[k * P + p], sN);
        }
        if (which) gNbar[p] += sN;
        else gN[p] += sN;
      }
    }
  }
  if (bad) atomicOr(err, bad);
}

// Chain rule through Eq. 8, N_p = (n_c + 3 f_c . Omega_p) dV / M with c the
// particle's initial cell: per cell summed over directions,
// out[0] dL/dn_nu, out[1] dL/dn_nubar, out[2..4] dL/df_nu, out[5..7] dL/df_nubar ([8][NZ]).
// A block takes 32 cells, its warps every kWarps-th direction (one thread a
// cell walked them all before: 81 us for 256 x 96, one load in flight), added
// in warp order.
static __global__ void k_weight_grad(Batch B, const double* __restrict__ gN, const double* __restrict__ gNbar,
                              const double* __restrict__ dirtab, double* __restrict__ out) {
  static_assert(kWarps == 8, "warp k adds row k");
  __shared__ double sm[kWarps][8][kLanes];
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
  const int gc = blockIdx.x * kLanes + lane;
  double a[8] = {};
  double f = 0.0;
  if (gc < B.NZ) {
    const BoxGeo& g = B.box[box_of_cell(B, gc)];
    f = g.dV / g.M;
    const int64_t p0 = g.poff + gc - g.coff;
#pragma unroll 4
    for (int d = wib; d < g.M; d += kWarps) {
      const double x = __ldg(gN + p0 + (int64_t)d * g.nz), y = __ldg(gNbar + p0 + (int64_t)d * g.nz);
      a[0] += x;
      a[1] += y;
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        const double o = 3.0 * __ldg(dirtab + (int64_t)i * B.MT + g.doff + d);
        a[2 + i] = fma(o, x, a[2 + i]);
        a[5 + i] = fma(o, y, a[5 + i]);
      }
    }
  }
#pragma unroll
  for (int k = 0; k < 8; ++k) sm[wib][k][lane] = a[k];
  __syncthreads();
  double v = 0.0;
#pragma unroll
  for (int x = 0; x < kWarps; ++x) v += sm[x][wib][lane];
  if (gc < B.NZ) out[(int64_t)wib * B.NZ + gc] = v * f;
}

}  // namespace emu_dev
