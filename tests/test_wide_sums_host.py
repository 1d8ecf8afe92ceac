"""The sums of csrc/wide.cuh that carry deposits and interpolations, compiled for
the host, against exact rational arithmetic."""
import ctypes
import subprocess
from fractions import Fraction as F
from pathlib import Path

import numpy as np
import pytest

CSRC = Path(__file__).resolve().parent.parent / "paper_2101_02745_gb300" / "csrc"
HARNESS = r'''
#include "wide.cuh"
using namespace emu_wide;
extern "C" {
// G = A0 - Omega . A from operands at one exponent, as the kernels form it: value 2^(*e - kBiasV)
int64_t dot(const double* A, const double* o, int* e) {
  int ea[4], top = 0;
  for (int k = 0; k < 4; ++k) { ea[k] = exponent(A[k]); top = max_i(top, ea[k]); }
  const int ko = direction_excess(o[0], o[1], o[2]);
  Limbs a[4], b[3];
  for (int k = 0; k < 4; ++k) a[k] = limbs(A[k], ea[k], top);
  for (int k = 0; k < 3; ++k) b[k] = unit_limbs(-o[k], ko);
  *e = top + 2 + ko - kBiasV;
  return join(split(dot3(align(join(a[0]) >> 2, ko, 0), a[1], b[0], a[2], b[1], a[3], b[2])));
}
double scaled_of(int64_t v, int k) { return scaled(v, k); }
// Zeroth and first moment of n terms, each the sum of three taps w v, as a deposit adds
// them; om: the terms' direction component (scaled by 2^-ko): value 2^(*ea + 4 - kBiasV).
// alternate: half a unit for the first moment as one every second term
void sums(const double* v, const double* wt, const double* om, int n, int ko, int alternate, int64_t* acc, int* ea) {
  const int head = sum_headroom(n), half = sum_half(ko);
  acc[0] = acc[1] = 0;
  *ea = 0;
  for (int d = 0; d < n; ++d) {
    int e[3], et = 0;
    for (int k = 0; k < 3; ++k) et = max_i(et, e[k] = exponent(v[3 * d + k]));
    int64_t cv = 0;
    for (int k = 0; k < 3; ++k) cv += align(mul(limbs(v[3 * d + k], e[k]), unit_limbs(wt[3 * d + k])), et - e[k]);
    const int es = et + ko;
    if (es + head > *ea) {
      const int sh = es + head - *ea;
      *ea += sh;
      acc[0] = align(acc[0], sh);
      acc[1] = align(acc[1], sh);
    }
    const int dd = *ea - es;
    const int64_t x = align(cv, dd);
    const Factor f = factor(join(unit_limbs(om[d], ko)));
    acc[0] += zeroth_moment(x, ko, half);
    acc[1] = alternate ? moment_add(factor(x + (d & 1)), f, half_unit(), acc[1])
                       : moment_add(factor(x), f, moment_half(f), acc[1]);
  }
}
}
'''


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("sums")
    (d / "h.cpp").write_text(HARNESS)
    # (sums that leave 64 bits wrap, as on the device)
    subprocess.check_call(["g++", "-O2", "-fwrapv", "-std=c++17", "-shared", "-fPIC", f"-I{CSRC}", "-o",
                           str(d / "h.so"), str(d / "h.cpp")])
    lib = ctypes.CDLL(str(d / "h.so"))
    lib.dot.restype = ctypes.c_int64
    lib.scaled_of.restype = ctypes.c_double
    lib.scaled_of.argtypes = [ctypes.c_int64, ctypes.c_int]
    return lib


def _ptr(a):
    return a.ctypes.data_as(ctypes.c_void_p)


def _directions(kind, n, rng):
    if kind == "corner":     # every component just below 1 (a length of 1.73), any signs
        return (1 - 2.0 ** -rng.integers(20, 53, (n, 3))) * rng.choice([-1.0, 1.0], (n, 3))
    if kind == "beyond":     # lengths from 1.7 to 2.3, one component up to 1.3
        return rng.uniform(0.9, 1.3, (n, 3)) * rng.choice([-1.0, 1.0], (n, 3))
    d = rng.normal(size=(n, 3))
    d /= np.linalg.norm(d, axis=1, keepdims=True)
    return d if kind == "unit" else d * np.exp(rng.uniform(np.log(0.01), np.log(1e6), (n, 1)))


@pytest.mark.parametrize("kind", ["unit", "corner", "beyond", "any length"])
@pytest.mark.parametrize("operands", ["largest", "random"])
def test_dot_product_of_any_direction(lib, kind, operands):
    """G against exact sums.  In units of 4 x 2^(exponent - kBiasV) = 2^-58 of the largest operand times
    2^k (the direction's excess): A0 rounded down 1, per product 1/2 + 1/4 from the truncated operands and 1
    from the dropped low product, 1 from the rounded middle sum, 1 from the split result: below 9; 2^k is at
    most 4 times the largest component, or 2."""
    rng = np.random.default_rng(3)
    n = 2000
    o = _directions(kind, n, rng)
    A = rng.uniform(-1, 1, (n, 4)) * np.exp(rng.uniform(-3, 0, (n, 4)))
    if operands == "largest":   # significands just below 2, each product of the sum of one sign
        A = (2 - 2.0 ** -50 * rng.integers(1, 2 ** 20, (n, 4))) * np.c_[np.ones(n), -np.sign(o)]
    e = ctypes.c_int()
    for a, d in zip(A, o):
        got = F(lib.dot(_ptr(a), _ptr(d), ctypes.byref(e))) * F(2) ** e.value
        ref = F(a[0]) - sum(F(x) * F(y) for x, y in zip(a[1:], d))
        scale = F(np.abs(a).max()) * F(max(2.0, 4 * np.abs(d).max()))
        assert abs(got - ref) <= 9 * F(2) ** -58 * scale, (a, d, float(got - ref))


def _sums(lib, v, w, om, ko=0, alternate=0):
    """(got, exact, FP64 chain) of both moments, and the largest term."""
    acc, ea = np.zeros(2, np.int64), ctypes.c_int()
    v, w, om = (np.ascontiguousarray(a, float) for a in (v, w, om))
    lib.sums(_ptr(v), _ptr(w), _ptr(om), len(om), ko, alternate, _ptr(acc), ctypes.byref(ea))
    got = [F(float(a)) * F(2) ** (ea.value + 4 - 1083) for a in acc.astype(float)]
    exact, f0, f1, big = [F(0), F(0)], 0.0, 0.0, 0.0
    for vv, ww, o in zip(v, w, om):
        c = 0.0
        for x, y in zip(vv, ww):
            c = float(F(c) + F(x) * F(y))       # (a multiply-add rounds once)
        f0, f1 = f0 + c, float(F(f1) + F(o) * F(c))
        t = sum(F(x) * F(y) for x, y in zip(vv, ww))
        exact[0] += t
        exact[1] += t * F(o)
        big = max(big, abs(float(t)))
    return got, exact, (f0, f1), big


@pytest.mark.parametrize("n", [1, 8, 31, 32, 225, 1000])
@pytest.mark.parametrize("kind", ["random signs", "one sign", "forward"])
@pytest.mark.parametrize("alternate", [0, 1])
def test_sums_err_no_more_than_double_precision(lib, alternate, kind, n):
    """The rms error of both moments of n terms is at most that of FP64 multiply-adds, and its mean is
    that of unbiased rounding (within five standard errors)."""
    rng = np.random.default_rng(n)
    trials = 40 if n > 100 else 100
    ours, chain = np.zeros((trials, 2)), np.zeros((trials, 2))
    for t in range(trials):
        d = rng.uniform(-0.5, 0.5, n)
        w = np.stack([0.5 * (0.5 - d) ** 2, 0.75 - d * d, 0.5 * (0.5 + d) ** 2], axis=1)
        v = rng.uniform(0.2, 1.2, (n, 3)) * (1.0 if kind == "one sign" else rng.choice([-1.0, 1.0], (n, 3)))
        om = rng.uniform(0.9, 1.0, n) if kind == "forward" else rng.uniform(-1.0, 1.0, n)
        got, exact, fp64, big = _sums(lib, v, w, om, 0, alternate)
        ours[t] = [float(g - x) / big for g, x in zip(got, exact)]
        chain[t] = [float(F(g) - x) / big for g, x in zip(fp64, exact)]
    rms, ref = (np.sqrt((a ** 2).mean(axis=0)) for a in (ours, chain))
    assert np.all(rms <= ref), (rms, ref)
    assert np.all(np.abs(ours.mean(axis=0)) <= 5 * rms / np.sqrt(trials)), (ours.mean(axis=0), rms)


@pytest.mark.parametrize("alternate", [0, 1])
@pytest.mark.parametrize("ko", [0, 1, 7])
@pytest.mark.parametrize("n", [1, 31, 32, 63, 64, 1023, 1024])
def test_sums_of_the_largest_terms_fit(lib, n, ko, alternate):
    """n terms of one sign at the largest significand, taps that add up to 2: within 2^-50 of the sum."""
    v = np.full((n, 3), -(2 - 2.0 ** -52))
    w = np.tile([0.5, 1.0, 0.5], (n, 1))
    got, exact, _, _ = _sums(lib, v, w, np.full(n, 2.0 ** ko), ko, alternate)
    for g, x in zip(got, exact):
        assert abs(g - x) <= F(2) ** -50 * abs(x) * (2 ** ko if x is exact[0] else 1)


@pytest.mark.parametrize("alternate", [0, 1])
def test_zero_terms_add_nothing(lib, alternate):
    n = 64
    v = np.zeros((n, 3))
    v[5] = [0.25, -1.5, 0.75]
    w = np.tile([0.125, 0.75, 0.125], (n, 1))
    om = np.linspace(-1, 1, n)
    got, exact, _, _ = _sums(lib, v, w, om, 0, alternate)
    assert got[0] == exact[0]                     # (few bits: exact)
    one, _, _, _ = _sums(lib, v[5:6], w[5:6], om[5:6], 0, alternate)
    assert abs(got[1] - exact[1]) <= F(2) ** -52 and abs(one[1] - exact[1]) <= F(2) ** -55


def test_scaled_results(lib):
    """v 2^k over every exponent a sum can have: exact, rounded once where subnormal, infinite where too large."""
    for v in (0, 1, -3, 2 ** 53 - 1, -(2 ** 62 + 2 ** 20), 2 ** 63 - 1, -2 ** 63):
        for k in (-1079, -1078, -1075, -1060, -1023, -1022, -1021, 0, 900, 958, 959, 960, 961, 967, 970, 1000):
            with np.errstate(over="ignore"):
                want = np.ldexp(np.float64(v), k)
            assert lib.scaled_of(v, k) == want, (v, k)
