// wide.cuh -- sums of products of doubles on the integer pipe.
//
// GB300 issues one FP64 instruction per SM every ~16 cycles (measured: DFMA
// 16.4, DADD and DMUL 19), and in that time ~33 half-rate integer instructions
// (IMAD.WIDE, SHF, LOP3) or ~65 full-rate ones (IADD, IMNMX); the two pipes
// run side by side.  The bilinear parts of the step (commutators, stencil
// sums) therefore run as fixed-point sums of 61-bit products with explicit
// exponents, at a third to a sixth of the FP64 pipe's time.
//
// Representation.  An operand is a signed integer V = h 2^32 + 2 l with
// |V| < 2^61 (h: the upper word; l: 31 bits with the sign of V) and an exponent
// e, the IEEE exponent field it is aligned to: the double x becomes
// V = x 2^(kBiasV - e), its 53 bits left-justified when e is x's own exponent
// field.  A complex operand has one exponent, the larger of its parts'.
// Products are (a b) / 2^64 = ah bh + 2 (ah bl + al bh) / 2^32 in an int64; the
// dropped al bl and the rounded middle term cost at most two units of 2^-56 of
// the product of the left-justified magnitudes.  A sum aligns its products to
// the largest exponent among them (arithmetic shifts, one unit each): the four
// groups of a commutator entry err by at most 12 units of 2^-56 of the largest
// product, a third to a half of a chain of FP64 multiply-adds in the mean
// (tests/test_wide_host.py measures both against exact sums: rms 3.7e-17 to
// 6e-17 of the entry against 5.5e-17 to 1.3e-16).
// Zero operands stay exactly zero, so zero products add exactly nothing.
// Subnormal inputs count as half their value (their field's exponent is that of
// the smallest normal numbers less one).  An infinite or
// NaN input is not represented: callers test exponents for kExpNonFinite (shape
// weights and directions, which have none, are tested where they are formed).
//
// The same code compiles for the host (g++), where the tests run it.
#pragma once

#include <cstdint>
#ifndef __CUDACC__
#define __host__
#define __device__
#define __forceinline__ inline
#endif
#define EMU_HD __host__ __device__ __forceinline__

namespace emu_wide {

struct Limbs { int h, l; };            // h 2^32 + 2 l
struct Real { Limbs v; int e; };       // v 2^(e - kBiasV)
struct Cplx { Limbs r, i; int e; };

constexpr int kBiasV = 1083;           // 1023 + 52 + 8: 53 bits shifted up by 8
constexpr int kBiasP = 2 * kBiasV - 64;   // a product of operands of exponents ea, eb: int64 2^(ea + eb - kBiasP)
constexpr int kExpNonFinite = 2047;

EMU_HD int hi_word(double x) {
#ifdef __CUDA_ARCH__
  return __double2hiint(x);
#else
  int64_t b;
  __builtin_memcpy(&b, &x, 8);
  return (int)(b >> 32);
#endif
}
EMU_HD int lo_word(double x) {
#ifdef __CUDA_ARCH__
  return __double2loint(x);
#else
  int64_t b;
  __builtin_memcpy(&b, &x, 8);
  return (int)b;
#endif
}
EMU_HD double from_words(int hi, int lo) {
#ifdef __CUDA_ARCH__
  return __hiloint2double(hi, lo);
#else
  const int64_t b = (int64_t)(((uint64_t)(uint32_t)hi << 32) | (uint32_t)lo);
  double x;
  __builtin_memcpy(&x, &b, 8);
  return x;
#endif
}
// Low word of (hi:lo) >> min(s, 32), s >= 0.
EMU_HD unsigned funnel_r(unsigned lo, unsigned hi, int s) {
#ifdef __CUDA_ARCH__
  return __funnelshift_rc(lo, hi, s);
#else
  return s >= 32 ? hi : (unsigned)((((uint64_t)hi << 32) | lo) >> s);
#endif
}
// x >> s for any s >= 0 (the PTX shifts clamp s).
EMU_HD int sar(int x, int s) {
#ifdef __CUDA_ARCH__
  int r;
  asm("shr.s32 %0, %1, %2;" : "=r"(r) : "r"(x), "r"(s));
  return r;
#else
  return x >> (s > 31 ? 31 : s);
#endif
}
EMU_HD unsigned shr(unsigned x, int s) {
#ifdef __CUDA_ARCH__
  unsigned r;
  asm("shr.u32 %0, %1, %2;" : "=r"(r) : "r"(x), "r"(s));
  return r;
#else
  return s > 31 ? 0u : x >> s;
#endif
}
EMU_HD int min_i(int a, int b) { return a < b ? a : b; }
EMU_HD int max_i(int a, int b) { return a > b ? a : b; }
// a b + c and a b: one IMAD.WIDE each.  (Written out in PTX: where the compiler
// moves an operand's sign extension away from the product it multiplies 64 by
// 64 bits, four instructions for one.)
EMU_HD int64_t mad(int a, int b, int64_t c) {
#ifdef __CUDA_ARCH__
  int64_t d;
  asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(d) : "r"(a), "r"(b), "l"(c));
  return d;
#else
  return (int64_t)a * b + c;
#endif
}
EMU_HD int64_t prod(int a, int b) {
#ifdef __CUDA_ARCH__
  int64_t d;
  asm("mul.wide.s32 %0, %1, %2;" : "=l"(d) : "r"(a), "r"(b));
  return d;
#else
  return (int64_t)a * b;
#endif
}

EMU_HD int exponent(double x) { return (hi_word(x) >> 20) & 0x7ff; }

EMU_HD Limbs negate(Limbs a) { return Limbs{-a.h, -a.l}; }

// x (exponent field e) left-justified / aligned to exponent E >= e.
EMU_HD Limbs limbs(double x, int e) {
  const int hi = hi_word(x), lo = lo_word(x), s = hi >> 31;
  const unsigned m = (unsigned)(hi & 0xfffff) + ((unsigned)min_i(e, 1) << 20);   // (no leading one at e = 0)
  return Limbs{((int)((m << 8) | ((unsigned)lo >> 24)) ^ s) - s, ((int)(((unsigned)lo << 7) & 0x7fffffffu) ^ s) - s};
}
EMU_HD Limbs limbs(double x, int e, int E) {
  const int hi = hi_word(x), lo = lo_word(x), s = hi >> 31, d = E - e;
  const unsigned m = (unsigned)(hi & 0xfffff) + ((unsigned)min_i(e, 1) << 20);
  const unsigned v1 = (m << 8) | ((unsigned)lo >> 24), v0 = (unsigned)lo << 8;
  const unsigned h = shr(v1, d), l = funnel_r(funnel_r(v0, v1, d), h, max_i(d - 32, 0));
  return Limbs{((int)h ^ s) - s, ((int)(l >> 1) ^ s) - s};
}

// x, |x| <= 1, as V = x 2^62 (direction components, shape weights), whatever
// its exponent field; with k > 0 V = x 2^(62 - k).
EMU_HD Limbs unit_limbs(double x, int k = 0) {
  const int hi = hi_word(x), lo = lo_word(x), s = hi >> 31, e = (hi >> 20) & 0x7ff, d = 1023 + k - e;
  const unsigned m = (unsigned)(hi & 0xfffff) + ((unsigned)min_i(e, 1) << 20);
  const unsigned v1 = (m << 10) | ((unsigned)lo >> 22), v0 = (unsigned)lo << 10;
  const unsigned h = shr(v1, d), l = funnel_r(funnel_r(v0, v1, d), h, max_i(d - 32, 0));
  return Limbs{((int)h ^ s) - s, ((int)(l >> 1) ^ s) - s};
}
// The k a component x of a direction needs: 0 up to 1 (and its rounding),
// otherwise such that three scaled components stay below 1/2 each.
EMU_HD int unit_excess(double x) {
  const int a = hi_word(x) & 0x7fffffff;
  return a > 0x3ff00001 ? (a >> 20) - 1021 : 0;
}
constexpr int kMaxExcess = 29;   // larger directions (above 2^27) count as infinite
// dot3 needs components whose magnitudes add up to at most 2.25 (unit vectors:
// 1.74): |x| in units of 2^-20, one that has an excess as more than that limit.
constexpr int kDotLimit = 9 << 18;
EMU_HD int unit_magnitude(double x) {
  const int a = hi_word(x) & 0x7fffffff;
  return a > 0x3ff00001 ? 1 << 24 : (int)shr((unsigned)(a & 0xfffff) | 0x100000u, 1023 - (a >> 20));
}
// The k of a direction (x, y, z) in dot3.
EMU_HD int direction_excess(double x, double y, double z) {
  const int k = max_i(max_i(unit_excess(x), unit_excess(y)), unit_excess(z));
  return k == 0 && unit_magnitude(x) + unit_magnitude(y) + unit_magnitude(z) > kDotLimit ? 1 : k;
}
// Limbs of an int64 below 2^61 in magnitude, and back.
EMU_HD Limbs split(int64_t v) { return Limbs{(int)(v >> 32), (int)((unsigned)v >> 1)}; }
EMU_HD int64_t join(Limbs a) { return (int64_t)(((uint64_t)(uint32_t)a.h << 32) + 2 * (int64_t)a.l); }

EMU_HD Real real(double x) {
  const int e = exponent(x);
  return Real{limbs(x, e), e};
}
EMU_HD Cplx cplx(double re, double im) {
  const int er = exponent(re), ei = exponent(im), e = max_i(er, ei);
  return Cplx{limbs(re, er, e), limbs(im, ei, e), e};
}

// Rounding addend of the middle term and the factor that folds it in.  From
// constant memory, so that they stay register operands of IMAD.WIDE: as
// literals the compiler turns them into 64-bit adds and shifts (mul 8 instead of
// 4 instructions, mul2 12 instead of 7).
#ifdef __CUDACC__
static __constant__ int64_t c_half = (int64_t)1 << 31;
static __constant__ int c_two = 2, c_one = 1;
#endif
EMU_HD int64_t half_unit() {
#ifdef __CUDA_ARCH__
  return c_half;
#else
  return (int64_t)1 << 31;
#endif
}
EMU_HD int two() {
#ifdef __CUDA_ARCH__
  return c_two;
#else
  return 2;
#endif
}
EMU_HD int one() {
#ifdef __CUDA_ARCH__
  return c_one;
#else
  return 1;
#endif
}
// a b / 2^64.  |V| < 2^61 keeps every partial sum in 63 bits.
EMU_HD int64_t mul(Limbs a, Limbs b) {
  const int64_t m = mad(a.h, b.l, mad(a.l, b.h, half_unit()));
  return mad((int)(m >> 32), two(), prod(a.h, b.h));
}
// The same with the middle term rounded down (two instructions less each: the
// rounding addend costs a 64-bit add).  For sums with as many subtracted as
// added products, in which the bias cancels.
EMU_HD int64_t mul_down(Limbs a, Limbs b) {
  const int64_t m = mad(a.h, b.l, prod(a.l, b.h));
  return mad((int)(m >> 32), two(), prod(a.h, b.h));
}
EMU_HD int64_t mul2_down(Limbs a, Limbs b, Limbs c, Limbs d) {
  const int64_t m = mad(a.h, b.l, mad(a.l, b.h, mad(c.h, d.l, prod(c.l, d.h))));
  return mad((int)(m >> 32), two(), mad(a.h, b.h, prod(c.h, d.h)));
}

// q + (a1 b1 + a2 b2 + a3 b3) / 2^64 for |a| < 2^61, |q| < 2^59 and |b1| + |b2| +
// |b3| <= 2.25 2^62 (direction_excess): the middle sum stays below 3 2^60 +
// 2.25 2^61 < 2^63, the result below 2^60.71.  (Components just below 1 each, a
// length of 1.73, wrapped it: 6e-9 of G.)
EMU_HD int64_t dot3(int64_t q, Limbs a1, Limbs b1, Limbs a2, Limbs b2, Limbs a3, Limbs b3) {
  const int64_t m =
      mad(a1.h, b1.l, mad(a1.l, b1.h, mad(a2.h, b2.l, mad(a2.l, b2.h, mad(a3.h, b3.l, mad(a3.l, b3.h, half_unit()))))));
  const int64_t p = mad(a1.h, b1.h, mad(a2.h, b2.h, mad(a3.h, b3.h, q)));
  return mad((int)(m >> 32), two(), p);
}

// v >> d, arithmetic, for any d >= 0; d2 = max(d - 32, 0) (shared by values of one shift).
EMU_HD int64_t align(int64_t v, int d, int d2) {
  const int hi = (int)(v >> 32), h = sar(hi, d);
  const unsigned l = funnel_r(funnel_r((unsigned)v, (unsigned)hi, d), (unsigned)h, d2);
  return (int64_t)(((uint64_t)(uint32_t)h << 32) | l);
}
EMU_HD int64_t align(int64_t v, int d) { return align(v, d, max_i(d - 32, 0)); }

// Sums of many terms with their moments (Eq. 5).  A contribution cv, |cv| <= 2^60
// at exponent es, is aligned to the sums' exponent ea >= es + sum_headroom(n) and
// added, a quarter of it to the zeroth moment's sum, a quarter times Omega to the
// others', so that n terms of one sign stay in 63 bits.  Alignment rounds down by
// half a unit in the mean.  The zeroth moment's quarter, rounded up from half,
// makes up for it, and so does half a unit times Omega in the rounding of the
// others': no bias is left.  (Floors alone left half a unit a term: 20 times the
// error of an FP64 sum for 225 terms of random sign, 90 times for 1000; now 0.1 to
// 0.8 of it for 1 to 4000 terms.)  A zero contribution adds exactly nothing.
EMU_HD int sum_headroom(int n) {
#ifdef __CUDA_ARCH__
  return max_i(32 - __clz(n), 5) - 5;
#else
  return max_i(32 - __builtin_clz((unsigned)n), 5) - 5;
#endif
}
// Factors of the moments: h 2^32 + l, l of full width and either sign, so that the
// dropped low products (at most a quarter of a unit) cancel in the mean.
struct Factor { int h, l; };
EMU_HD Factor factor(int64_t v) { return Factor{(int)(v >> 32) + (int)((unsigned)v >> 31), (int)v}; }
// v / 4 (directions scaled by 2^-ko: / 2^(2 + ko)); half = sum_half(ko).
EMU_HD int sum_half(int ko) { return 2 << min_i(ko, kMaxExcess); }
EMU_HD int64_t zeroth_moment(int64_t v, int ko, int half) { return align(v + half, 2 + ko, 0); }
// c + v om / 2^64 for om = 2^62 Omega; half = moment_half(om).
EMU_HD int64_t moment_half(Factor om) { return ((int64_t)1 << 31) + (om.h >> 1); }
EMU_HD int64_t moment_add(Factor v, Factor om, int64_t half, int64_t c) {
  const int64_t m = mad(v.h, om.l, mad(v.l, om.h, half));
  return mad((int)(m >> 32), one(), mad(v.h, om.h, c));
}

// v / 2^d rounded to nearest, d >= 1.
EMU_HD int64_t align_round(int64_t v, int d) { return (align(v, d - 1) + 1) >> 1; }

// c 2^k for a positive normal c, k not below its smallest normal result; NaN
// where the result is out of range (k at most 3000).
EMU_HD double scale_up(double c, int k) {
  const unsigned h = (unsigned)hi_word(c) + ((unsigned)k << 20);
  return from_words((int)(h < 0x7ff80000u ? h : 0x7ff80000u), lo_word(c));
}
// x 2^k for x = 0 or a normal x whose exponent stays normal.
EMU_HD double scale_nz(double x, int k) {
  const int hi = hi_word(x);
  return from_words(hi != 0 ? hi + (int)((unsigned)k << 20) : hi, lo_word(x));
}

// A sum v 2^k as a double, |k| < 2000: rounded where it is subnormal, infinite where
// it is too large.  Only the ends of the range of doubles take more than
// scaled_near, whose v 2^k has to be normal or zero; a caller with many sums tests
// them together, since a branch each keeps their conversions from overlapping (the
// interpolation call took 19 % longer).
EMU_HD int near(int k) { return min_i(max_i(k, -1022), 959); }   // (normal for any v)
EMU_HD double far_factor(int k) { return from_words((1023 + k - near(k)) << 20, 0); }
EMU_HD double scaled_near(int64_t v, int k) { return scale_nz((double)v, k); }
EMU_HD double scaled(int64_t v, int k) {
  return v != 0 && k != near(k) ? scaled_near(v, near(k)) * far_factor(k) : scaled_near(v, k);
}

// A traceless Hermitian matrix H as the commutator's left operand: diagonal
// differences H_11 - H_22, H_11 - H_33, H_22 - H_33 and off-diagonals.
struct Ham {
  Real d12, d13, d23;
  Cplx a, b, c;
};
// From the traceless components (H_11 - H_22, H_22 - H_33, off-diagonal reals).
EMU_HD Ham ham(const double (&H)[8]) {
  Ham h;
  h.d12 = real(H[0]);
  h.d13 = real(H[0] + H[1]);
  h.d23 = real(H[1]);
  h.a = cplx(H[2], H[3]);
  h.b = cplx(H[4], H[5]);
  h.c = cplx(H[6], H[7]);
  return h;
}

// A Hermitian matrix r (or its conjugate) as the right operand.
struct Mat {
  Real e12, e13, e23;    // r_11 - r_22, r_11 - r_33, r_22 - r_33
  Cplx x, y, z;
  Limbs nx, nz;          // minus the imaginary parts of x, z
};
EMU_HD Mat mat(const double* r, bool conj) {
  Mat m;
  m.e12 = real(r[0] - r[1]);
  m.e13 = real(r[0] - r[2]);
  m.e23 = real(r[1] - r[2]);
  m.x = cplx(r[3], r[4]);
  m.y = cplx(r[5], r[6]);
  m.z = cplx(r[7], r[8]);
  const int c = conj ? -1 : 0;
  m.x.i = Limbs{(m.x.i.h ^ c) - c, (m.x.i.l ^ c) - c};
  m.y.i = Limbs{(m.y.i.h ^ c) - c, (m.y.i.l ^ c) - c};
  m.z.i = Limbs{(m.z.i.h ^ c) - c, (m.z.i.l ^ c) - c};
  m.nx = negate(m.x.i);
  m.nz = negate(m.z.i);
  return m;
}
// Largest exponent field among the operands (kExpNonFinite: an input is infinite or NaN).
EMU_HD int top(const Ham& H) {
  return max_i(max_i(max_i(H.d12.e, H.d13.e), max_i(H.d23.e, H.a.e)), max_i(H.b.e, H.c.e));
}
EMU_HD int top(const Mat& m) {
  return max_i(max_i(max_i(m.e12.e, m.e13.e), max_i(m.e23.e, m.x.e)), max_i(m.y.e, m.z.e));
}

// Entries of C = [H, r], rounded to doubles up to a power of two each, so that a
// caller can finish one before it forms the next:
//   commutator_off<q>: C_12, C_13, C_23 (q = 0, 1, 2) = (cr + i ci) 2^(e - kBiasP),
//   commutator_diag:   K_11 / 2, K_22 / 2, K_33 / 2 of K = -i C = kd[q] 2^(ke[q] - kBiasP).
// D x - E a + (g1) - (g2) at the largest exponent (at least emin).  Two products
// are added and two subtracted: their rounding down cancels in the mean.
EMU_HD void off_diagonal(const Real& D, const Cplx& x, const Real& E, const Cplx& a, int64_t g1r, int64_t g1i, int e1,
                         int64_t g2r, int64_t g2i, int e2, int emin, double& cr, double& ci, int& oe) {
  const int ea = D.e + x.e, eb = E.e + a.e;
  const int e = max_i(max_i(max_i(ea, eb), max_i(e1, e2)), emin);
  const int da = e - ea, db = e - eb, d1 = e - e1, d2 = e - e2;
  const int fa = max_i(da - 32, 0), fb = max_i(db - 32, 0), f1 = max_i(d1 - 32, 0), f2 = max_i(d2 - 32, 0);
  cr = (double)(align(mul_down(D.v, x.r), da, fa) - align(mul_down(E.v, a.r), db, fb) + align(g1r, d1, f1) -
                align(g2r, d2, f2));
  ci = (double)(align(mul_down(D.v, x.i), da, fa) - align(mul_down(E.v, a.i), db, fb) + align(g1i, d1, f1) -
                align(g2i, d2, f2));
  oe = e;
}

template <int Q>
EMU_HD void commutator_off(const Ham& H, const Mat& m, int emin, double& cr, double& ci, int& e) {
  const Cplx &x = m.x, &y = m.y, &z = m.z, &a = H.a, &b = H.b, &c = H.c;
  if (Q == 0)   // C_12 = d12 x - e12 a + b z^* - y c^*
    off_diagonal(H.d12, x, m.e12, a, mul2_down(b.r, z.r, b.i, z.i), mul2_down(b.i, z.r, b.r, m.nz), b.e + z.e,
                 mul2_down(c.r, y.r, c.i, y.i), mul2_down(c.r, y.i, negate(c.i), y.r), c.e + y.e, emin, cr, ci, e);
  else if (Q == 1)   // C_13 = d13 y - e13 b + a z - x c
    off_diagonal(H.d13, y, m.e13, b, mul2_down(a.r, z.r, a.i, m.nz), mul2_down(a.r, z.i, a.i, z.r), a.e + z.e,
                 mul2_down(c.r, x.r, c.i, m.nx), mul2_down(c.r, x.i, c.i, x.r), c.e + x.e, emin, cr, ci, e);
  else   // C_23 = d23 z - e23 c + a^* y - x^* b
    off_diagonal(H.d23, z, m.e23, c, mul2_down(a.r, y.r, a.i, y.i), mul2_down(a.r, y.i, negate(a.i), y.r), a.e + y.e,
                 mul2_down(b.r, x.r, b.i, x.i), mul2_down(b.i, x.r, b.r, m.nx), b.e + x.e, emin, cr, ci, e);
}
EMU_HD void commutator_diag(const Ham& H, const Mat& m, int emin, double (&kd)[3], int (&ke)[3]) {
  const Cplx &x = m.x, &y = m.y, &z = m.z, &a = H.a, &b = H.b, &c = H.c;
  // p = Im(a x^*), q = -Im(b y^*), t = Im(c z^*): K_11 / 2 = p - q, K_22 / 2 = t - p, K_33 / 2 = q - t
  const int64_t p = mul2_down(a.i, x.r, a.r, m.nx), q = mul2_down(b.r, y.i, negate(b.i), y.r),
                t = mul2_down(c.i, z.r, c.r, m.nz);
  const int ep = a.e + x.e, eq = b.e + y.e, et = c.e + z.e;
  ke[0] = max_i(max_i(ep, eq), emin);
  ke[1] = max_i(max_i(ep, et), emin);
  ke[2] = max_i(max_i(eq, et), emin);
  kd[0] = (double)(align(p, ke[0] - ep) - align(q, ke[0] - eq));
  kd[1] = (double)(align(t, ke[1] - et) - align(p, ke[1] - ep));
  kd[2] = (double)(align(q, ke[2] - eq) - align(t, ke[2] - et));
}

}  // namespace emu_wide
