"""Parts of a tile whose warps take several directions each: the block's sums and
their exponents go to the buffers the particle data came through.  Every lane
keeps to its own column of them (checked where the kernel is compiled); here the
step, in each shape order, matches the oracle and repeats bitwise.

Tolerance as elsewhere: the first steps against the oracle 1e-10 (family-wise)."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2101_02745_gb300 import workloads as W
from tests.compare import family_err, pack

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2101_02745_gb300 import build
    build.build()
    return torch


# (cells, directions, blocks): one tile whose parts hold 67 (8 or 9 directions a
# warp), 17 (2 or 3) and 9 (1 or 2) directions
@pytest.mark.parametrize("order", [0, 1, 2, 3])
@pytest.mark.parametrize("nz,M,blocks", [(28, 200, 3), (27, 66, 4), (20, 9, 1)])
def test_several_directions_a_warp(torch, order, nz, M, blocks):
    from paper_2101_02745_gb300.emu import Box
    wl = W.with_shape(W.random_box(nz, M, seed=nz * M + order), order)
    cfg = O.config(wl.nz, wl.ndir, wl.Lz, wl.kappa, wl.c_light, wl.cfl_adv, wl.cfl_flavor, wl.area,
                   shape_order=wl.shape_order)
    parts = O.init(cfg, wl.n_nu, wl.n_nubar, wl.f_nu, wl.f_nubar, wl.alpha, wl.seed, wl.dirs)
    dt = 0.917 * O.timestep(cfg, O.deposit(cfg, parts))   # (below the limit: order 0 meets its discontinuities there)
    out = []
    for _ in range(3):
        box = Box.from_workload(wl)
        box.set_grid(blocks)
        box.step(4, dt)
        out.append(box.get_host())
        box.sync()
    for h in out[1:]:
        assert all(np.array_equal(h[k], out[0][k]) for k in h)
    O.run(cfg, parts, dt, 4)
    assert family_err(out[0]["rho"], pack(parts["rho"])) < 1e-10
    assert family_err(out[0]["rhobar"], pack(parts["rhobar"])) < 1e-10
