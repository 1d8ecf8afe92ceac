"""The integer-pipe sums of csrc/wide.cuh, compiled for the host, against exact
rational arithmetic: commutators and stencil sums over operand scales from order
one to deep in the linear phase, with zero, subnormal and extreme operands."""
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
void comm(const double* H, const double* r, int conj, int emin, double* v, int* e) {
  double h[8];
  for (int k = 0; k < 8; ++k) h[k] = H[k];
  const Ham hm = ham(h);
  const Mat m = mat(r, conj != 0);
  int o, ke[3];
  double kd[3];
  commutator_off<0>(hm, m, emin, v[0], v[1], o); e[0] = e[1] = o - kBiasP;
  commutator_off<1>(hm, m, emin, v[2], v[3], o); e[2] = e[3] = o - kBiasP;
  commutator_off<2>(hm, m, emin, v[4], v[5], o); e[4] = e[5] = o - kBiasP;
  commutator_diag(hm, m, emin, kd, ke);
  for (int q = 0; q < 3; ++q) { v[6 + q] = kd[q]; e[6 + q] = ke[q] - kBiasP; }
}
int top_of(const double* H, const double* r) {
  double h[8];
  for (int k = 0; k < 8; ++k) h[k] = H[k];
  return max_i(top(ham(h)), top(mat(r, false)));
}
}
'''


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("wide")
    (d / "h.cpp").write_text(HARNESS)
    subprocess.check_call(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", f"-I{CSRC}", "-o", str(d / "h.so"),
                           str(d / "h.cpp")])
    return ctypes.CDLL(str(d / "h.so"))


def _ptr(a):
    return a.ctypes.data_as(ctypes.c_void_p)


def _operands(rng, eps, n):
    """H (traceless components) and r with off-diagonals of relative size eps (eps^2 for the last pair)."""
    s = np.array([1, 1, eps, eps, eps, eps, eps * eps, eps * eps])
    H = 1e11 * s * rng.uniform(-1, 1, (n, 8))
    r = np.concatenate([rng.uniform(0, 1, (n, 3)), s[2:] * rng.uniform(-1, 1, (n, 6))], axis=1)
    return H, r


def _groups(H, r):
    """Per entry the products of C = [H, r] (exact), then K_aa / 2, grouped as complex products."""
    d12, d23, ar, ai, br, bi, cr, ci = [F(float(v)) for v in H]
    d13 = d12 + d23
    r11, r22, r33, xr, xi, yr, yi, zr, zi = [F(float(v)) for v in r]
    e21, e31, e32 = r22 - r11, r33 - r11, r33 - r22
    return [
        [[d12 * xr], [e21 * ar], [br * zr, bi * zi], [-cr * yr, -ci * yi]],
        [[d12 * xi], [e21 * ai], [bi * zr, -br * zi], [-cr * yi, ci * yr]],
        [[d13 * yr], [e31 * br], [ar * zr, -ai * zi], [-cr * xr, ci * xi]],
        [[d13 * yi], [e31 * bi], [ar * zi, ai * zr], [-cr * xi, -ci * xr]],
        [[d23 * zr], [e32 * cr], [ar * yr, ai * yi], [-br * xr, -bi * xi]],
        [[d23 * zi], [e32 * ci], [ar * yi, -ai * yr], [-bi * xr, br * xi]],
        [[ai * xr, -ar * xi], [bi * yr, -br * yi]],
        [[ci * zr, -cr * zi], [-ai * xr, ar * xi]],
        [[-bi * yr, br * yi], [-ci * zr, cr * zi]],
    ]


def _run(lib, H, r, conj=False, emin=0):
    v, e = np.zeros(9), np.zeros(9, np.int32)
    H, r = np.ascontiguousarray(H, float), np.ascontiguousarray(r, float)
    lib.comm(_ptr(H), _ptr(r), int(conj), emin, _ptr(v), _ptr(e))
    return [F(float(a)) * F(2) ** int(b) for a, b in zip(v, e)]


def _scale(H, r):
    """Largest product of complex magnitudes (larger parts) of each entry, as the alignment sees it."""
    H, r = [abs(float(v)) for v in H], [float(v) for v in r]
    d12, d13, d23 = H[0], H[0] + H[1], H[1]
    a, b, c = max(H[2:4]), max(H[4:6]), max(H[6:8])
    x, y, z = (max(abs(r[k]), abs(r[k + 1])) for k in (3, 5, 7))
    e21, e31, e32 = abs(r[1] - r[0]), abs(r[2] - r[0]), abs(r[2] - r[1])
    o12, o13, o23 = max(d12 * x, e21 * a, b * z, c * y), max(d13 * y, e31 * b, a * z, c * x), \
        max(d23 * z, e32 * c, a * y, b * x)
    return [o12, o12, o13, o13, o23, o23, max(a * x, b * y), max(c * z, a * x), max(b * y, c * z)]


@pytest.mark.parametrize("eps", [1.0, 1e-3, 1e-6, 1e-20, 1e-100])
def test_commutator_error(lib, eps):
    """At most 12 units of 2^-56 per entry from the sum, 2^-53 each from the rounded operand differences
    and the result: below 2^-51 of the largest product; and a smaller rms error than the FP64 chain's."""
    rng = np.random.default_rng(1)
    H, r = _operands(rng, eps, 300)
    ours, chain = [], []
    for h, m in zip(H, r):
        got, sc = _run(lib, h, m), _scale(h, m)
        for k, groups in enumerate(_groups(h, m)):
            ref = sum(p for g in groups for p in g)
            assert abs(got[k] - ref) <= F(2) ** -51 * F(sc[k]) * 2, (k, float(got[k] - ref), sc[k])
            acc = np.float64(0)
            for p in reversed([p for g in groups for p in g]):   # a chain of multiply-adds: one rounding per product
                acc = np.float64(float(p + F(float(acc))))
            ours.append(float(abs(got[k] - ref)) / sc[k])
            chain.append(float(abs(F(float(acc)) - ref)) / sc[k])
    assert np.sqrt(np.mean(np.square(ours))) < 1.05 * np.sqrt(np.mean(np.square(chain)))


def test_zero_and_conjugate(lib):
    rng = np.random.default_rng(2)
    H, r = _operands(rng, 1e-3, 20)
    for h, m in zip(H, r):
        d = m.copy()
        d[3:] = 0.0                       # diagonal r with diagonal H: exactly nothing
        hd = h.copy()
        hd[2:] = 0.0
        assert all(v == 0 for v in _run(lib, hd, d))
        mc = m.copy()
        mc[[4, 6, 8]] *= -1               # the conjugate matrix, formed by the caller or by the flag
        assert _run(lib, h, mc) == _run(lib, h, m, conj=True)


def test_extreme_operands(lib):
    H = np.array([1e-300, 3e-310, 1e150, -1e-200, 0.0, 5e-324, -1e-50, 1e50])
    r = np.array([1e-308, 1.0, -1e-16, 1e-300, 0.0, 1e120, -1e-150, 5e-324, 1e-12])
    got, sc = _run(lib, H, r), _scale(H, r)
    for k, groups in enumerate(_groups(H, r)):
        ref = sum(p for g in groups for p in g)
        # subnormal operands keep their own bits: the bound holds absolutely at the entry's largest product
        assert abs(got[k] - ref) <= F(2) ** -50 * F(sc[k]) + F(2) ** -1100
    big = H.copy()
    big[3] = np.inf
    assert lib.top_of(_ptr(big), _ptr(r)) >= 2047
    rn = r.copy()
    rn[2] = np.nan
    assert lib.top_of(_ptr(H), _ptr(rn)) >= 2047
    assert lib.top_of(_ptr(H), _ptr(r)) < 2047
