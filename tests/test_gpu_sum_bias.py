"""Direction sums of many terms of random sign carry no bias: the off-diagonals of
the potential and its fluxes against extended-precision sums, 1000 directions a
warp.

Each term's B is formed in FP64 (two roundings, below 2^-52 of the largest), the
sum of M terms then errs by less than M 2^-52 of the largest term: FP64 sums stay
far below, sums that round every term down exceed it."""
import numpy as np
import pytest

from paper_2101_02745_gb300 import workloads as W
from tests.test_gpu_work_splits import _box, torch  # noqa: F401

pytestmark = pytest.mark.gpu
M, NZ = 8000, 20


def _check(A, kappa_dV, B, om):
    """A[36][NZ] of terms B[k][M][NZ] (particles at cell centres: weights 1/8, 3/4, 1/8)."""
    for k in (3, 4, 5, 6):
        b = B[k].astype(np.longdouble)
        c = 0.75 * b + 0.125 * (np.roll(b, 1, axis=1) + np.roll(b, -1, axis=1))
        for m in range(4):
            ref = kappa_dV * (c if m == 0 else c * om[m - 1].astype(np.longdouble)).sum(axis=0)
            err = np.abs(A[9 * m + k] - ref).max() / (kappa_dV * np.abs(B[k]).max())
            assert err < M * 2.0 ** -52, (k, m, float(err))


def _terms(wl, box):
    h = box.get_host()
    box.sync()
    shape = (M, -1)
    N, Nb = h["N"].reshape(shape), h["Nbar"].reshape(shape)
    sign = [1, 1, 1, 1, -1, 1, -1, 1, -1]
    B = [N * h["rho"][k].reshape(shape) - sign[k] * Nb * h["rhobar"][k].reshape(shape) for k in range(9)]
    return B, [h[k].reshape(shape) for k in ("ox", "oy", "oz")]


def test_direction_sums(torch):  # noqa: F811
    wl = W.random_box(NZ, M, seed=3)   # (cells of 1/16: the positions and their weights are exact)
    box = _box(wl, 1)
    B, om = _terms(wl, box)
    _check(box.deposit(0, 0.0).cpu().numpy(), np.longdouble(wl.kappa) / (wl.area * wl.dz), B, om)
