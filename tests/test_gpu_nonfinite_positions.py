"""A particle without a finite position is reported (EMU_ENUMERIC; a ring's first
particle may also put the ring's shift, and with it the ring, off its sites:
EMU_ELATTICE, which is reported first) and shows in the results, in every kernel that forms shape weights: the first particle of a ring
(whose weights its ring may share) or a later one, with and without the ring
table (taken when every warp walks several directions), off the lattice, and on
each axis of a 3D box.  The positions are written in the bound arrays, where no
layout check sees them."""
import numpy as np
import pytest

from paper_2101_02745_gb300 import workloads as W
from tests.test_gpu_work_splits import _box, torch  # noqa: F401

pytestmark = pytest.mark.gpu
BAD = [np.nan, np.inf, -np.inf]


def _raises(box, first=False):
    from paper_2101_02745_gb300.emu import EMU_ELATTICE, EMU_ENUMERIC, EmuError
    with pytest.raises(EmuError) as ei:
        box.sync()
    assert ei.value.code == EMU_ENUMERIC or (first and ei.value.code == EMU_ELATTICE)


@pytest.mark.parametrize("bad", BAD)
@pytest.mark.parametrize("order", [0, 1, 2, 3])
@pytest.mark.parametrize("rk_form,blocks", [(0, 304), (1, 304), (0, 1), (1, 1)])
@pytest.mark.parametrize("ring,site", [(5, 0), (5, 40)])
def test_step(torch, order, rk_form, blocks, ring, site, bad):  # noqa: F811
    wl = W.with_shape(W.random_box(61, 13, seed=7), order)
    box = _box(wl, blocks, rk_form)
    box.set_layout(0)
    box.t["z"][ring * 61 + site] = bad
    box.step(1, 1e-13)
    rho = box.t["rho"].cpu().numpy()
    assert np.isnan(rho[:, ring * 61 + site]).any()
    _raises(box, site == 0)


@pytest.mark.parametrize("step_form", [1, 2])
@pytest.mark.parametrize("ring,site", [(5, 0), (5, 40)])
def test_step_forms(torch, step_form, ring, site):  # noqa: F811
    box = _box(W.random_box(61, 13, seed=7), 152)
    box.set_layout(0)
    box.set_step_form(step_form)
    box.t["z"][ring * 61 + site] = np.nan
    box.step(1, 1e-13)
    _raises(box, site == 0)


@pytest.mark.parametrize("order", [1, 2, 3])
@pytest.mark.parametrize("site", [0, 40])
def test_fields(torch, order, site):  # noqa: F811
    box = _box(W.with_shape(W.random_box(61, 13, seed=7), order))
    box.set_layout(0)
    A = box.deposit(0, 0.0).clone()
    p = 5 * 61 + site
    box.t["z"][p] = np.nan
    H = box.interpolate_H(0.0).cpu().numpy()      # from the sound potential: that particle's alone
    assert np.isnan(H[:, p]).all() and np.isfinite(np.delete(H, p, axis=1)).all()
    _raises(box, site == 0)
    assert torch.isfinite(A).all() and not torch.isfinite(box.deposit(0, 0.0)).all()
    _raises(box, site == 0)
    assert not torch.isfinite(box.moments()).all()
    _raises(box, site == 0)


def test_anywhere(torch):  # noqa: F811
    box = _box(W.random_box(61, 13, seed=7))
    box.set_layout(1)
    box.t["z"][5 * 61 + 40] = np.nan
    box.step(1, 1e-13)
    assert np.isnan(box.t["rho"].cpu().numpy()[:, 5 * 61 + 40]).any()
    _raises(box)


@pytest.mark.parametrize("axis", ["x", "y", "z"])
@pytest.mark.parametrize("order", [0, 2, 3])
@pytest.mark.parametrize("site", [0, 77])
def test_3d(torch, axis, order, site):  # noqa: F811
    from paper_2101_02745_gb300.emu import Box3D
    box = Box3D.from_workload(W.random_box3(4, 5, 9, 6, seed=1, shape_order=order))
    p = 3 * 180 + site
    box.t[axis][p] = np.inf
    box.step(1, 1e-13)
    assert np.isnan(box.t["rho"].cpu().numpy()[:, p]).any()
    _raises(box, site == 0)
