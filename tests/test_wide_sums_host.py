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
