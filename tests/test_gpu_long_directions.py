"""Directions whose components are each just below 1 (a length of 1.73): scaled by
1/2 before G = A0 - Omega . A is formed, in every kernel that forms it.

Tolerances as elsewhere: one interpolation 1e-12 against the density scale of its
summands, the first steps against the oracle 1e-10 (family-wise)."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2101_02745_gb300 import workloads as W
from tests.compare import density_scales, family_err, oracle_potential, pack
from tests.test_gpu_work_splits import _box, _check_steps, _oracle, torch  # noqa: F401

pytestmark = pytest.mark.gpu


def _corners(M):
    s = 1 - 2.0 ** -40
    return s * np.array([[1 - 2 * (d & 1), 1 - (d & 2), 1 - (d & 4) / 2] for d in range(M)])


def _workload(nz, order):
    wl = W.with_shape(W.random_box(nz, 8, seed=nz + order), order)
    wl.dirs = _corners(8)
    wl.f_nu, wl.f_nubar = wl.f_nu / 2, wl.f_nubar / 2   # (weights stay positive)
    return wl


@pytest.mark.parametrize("order", [0, 1, 2, 3])
@pytest.mark.parametrize("rk_form", [0, 1])
def test_lattice(torch, order, rk_form):  # noqa: F811
    wl = _workload(67, order)
    cfg, parts = _oracle(wl)
    box = _box(wl, 304, rk_form)
    grid = O.deposit(cfg, parts)
    s = wl.kappa * 3 * density_scales(grid)[2]
    A, Aref = box.deposit(0, 0.0).cpu().numpy(), oracle_potential(grid, wl.kappa)
    assert max(family_err(A[9 * f:9 * (f + 1)], Aref[9 * f:9 * (f + 1)], s) for f in range(4)) < 1e-12
    H = box.interpolate_H(0.0).cpu().numpy()
    assert family_err(H, pack(O.hamiltonian(cfg, grid, parts)), s) < 1e-12
    _check_steps(wl, _box(wl, 304, rk_form), factor=0.17)


def test_anywhere(torch):  # noqa: F811
    wl = _workload(67, 2)
    cfg, parts = _oracle(wl)
    rng = np.random.default_rng(2)
    z = parts["z"] + rng.uniform(-0.45, 0.45, len(parts)) * wl.dz
    parts["z"] = z - wl.Lz * np.floor(z / wl.Lz)
    parts["omega"] = _corners(8)[rng.integers(0, 8, len(parts))]   # (a direction each: off the lattice)
    box = _box(wl)
    box.set_host(z=parts["z"].copy(), **{k: parts["omega"][:, i].copy() for i, k in enumerate(("ox", "oy", "oz"))})
    assert box.general()
    dt = 0.17 * O.timestep(cfg, O.deposit(cfg, parts))
    box.step(4, dt)
    O.run(cfg, parts, dt, 4)
    h = box.get_host()
    box.sync()
    assert family_err(h["rho"], pack(parts["rho"])) < 1e-10
    assert family_err(h["rhobar"], pack(parts["rhobar"])) < 1e-10


def test_3d(torch):  # noqa: F811
    from tests.test_gpu_3d import _box as box3, _oracle as oracle3
    wl = W.random_box3(4, 3, 33, 8, seed=4)
    wl.dirs = _corners(8)
    wl.f_nu, wl.f_nubar = wl.f_nu / 2, wl.f_nubar / 2
    cfg, parts = oracle3(wl)
    dt = 0.17 * O.timestep3(cfg, O.deposit3(cfg, parts))
    box = box3(wl)
    box.step(4, dt)
    O.run3(cfg, parts, dt, 4)
    h = box.get_host()
    box.sync()
    assert family_err(h["rho"], pack(parts["rho"])) < 1e-10
    assert family_err(h["rhobar"], pack(parts["rhobar"])) < 1e-10
