"""Deposits and interpolations of fields at either end of the range of doubles: the
results' exponents, which the fixed-point sums carry beside them, are neither
limited nor cut off.  Against the oracle to 1e-12 of the largest value, as for
ordinary densities."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2101_02745_gb300 import workloads as W
from tests.compare import oracle_moments, oracle_potential, pack
from tests.test_gpu_work_splits import _box, _oracle, torch  # noqa: F401

pytestmark = pytest.mark.gpu

# (densities, kappa): terms from 1e-293 down to 1e-305 (normal numbers), the potential at 1e-50 and at
# 1e-291; terms near 1e306
SCALES = [(1e-291, 1e243), (1e-291, 1.0), (4e307, 1e-300)]


def _near(got, ref):
    top = np.abs(ref).max()
    assert np.all(np.isfinite(got)) and np.abs(got / top - ref / top).max() <= 1e-12


def _scaled(wl, n, kappa):
    for k in ("n_nu", "n_nubar", "f_nu", "f_nubar"):
        setattr(wl, k, getattr(wl, k) / 1e33 * n)
    wl.kappa = kappa
    return wl


@pytest.mark.parametrize("order", [0, 2, 3])
@pytest.mark.parametrize("n,kappa", SCALES)
def test_fields(torch, order, n, kappa):  # noqa: F811
    wl = _scaled(W.with_shape(W.random_box(67, 4, seed=order), order), n, kappa)
    cfg, parts = _oracle(wl)
    box = _box(wl)
    grid = O.deposit(cfg, parts)
    with np.errstate(under="ignore"):
        _near(box.deposit(0, 0.0).cpu().numpy(), oracle_potential(grid, wl.kappa))
        _near(box.interpolate_H(0.0).cpu().numpy(), pack(O.hamiltonian(cfg, grid, parts)))
        _near(box.moments().cpu().numpy(), oracle_moments(grid))
    box.sync()


def _slow(wl):
    """Terms near 1e-294 whose phases H dt are of order one: kappa 1e293, particles slow enough for such a step."""
    wl = _scaled(wl, 1e-291, 1e293)
    wl.c_light = 1.0
    return wl, 3e-3


def _check_step(box, run, cfg, parts, dt):
    box.step(2, dt)
    run(cfg, parts, dt, 2)
    h = box.get_host()
    box.sync()
    for k in ("rho", "rhobar"):
        ref = pack(parts[k])
        assert np.abs(ref[3:] - h[k][3:]).max() <= 1e-10 * np.abs(ref).max()
        _near(h[k], ref)


@pytest.mark.parametrize("blocks", [304, 1])
@pytest.mark.parametrize("dep_form", [0, 1])
def test_step(torch, blocks, dep_form):  # noqa: F811
    wl, dt = _slow(W.random_box(67, 30, seed=2))
    cfg, parts = _oracle(wl)
    box = _box(wl, blocks)
    box.set_deposit_form(dep_form)
    start = pack(parts["rho"]).copy()
    _check_step(box, O.run, cfg, parts, dt)
    assert np.abs(pack(parts["rho"]) - start).max() > 1e-9     # (the field acts)


def test_step_anywhere(torch):  # noqa: F811
    wl, dt = _slow(W.random_box(67, 30, seed=2))
    cfg, parts = _oracle(wl)
    box = _box(wl)
    box.set_layout(1)
    _check_step(box, O.run, cfg, parts, dt)


def test_step_3d(torch):  # noqa: F811
    from tests.test_gpu_3d import _box as box3, _oracle as oracle3
    wl, dt = _slow(W.random_box3(4, 3, 9, 6, seed=2))
    cfg, parts = oracle3(wl)
    _check_step(box3(wl), O.run3, cfg, parts, dt)
