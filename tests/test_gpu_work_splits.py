"""The work splits of the lattice step and its operands at the sizes where they
change: the RK stage's slabs of 1, 2, 4 and 8 tiles and its parts of a tile, the
deposit's parts of a tile and ranges of units, directions that are not unit
vectors (their operands are scaled), one species absent, non-finite input on
every split, and the adjoint's weight sums.

Tolerances as elsewhere: the first steps against the oracle 1e-10 (family-wise),
one deposit or interpolation 1e-12 against the density scale of its summands.
The RK stage does the same arithmetic per particle in either form: bitwise."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2101_02745_gb300 import workloads as W
from tests.compare import density_scales, family_err, oracle_potential, pack

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2101_02745_gb300 import build
    build.build()
    return torch


def _oracle(wl):
    cfg = O.config(wl.nz, wl.ndir, wl.Lz, wl.kappa, wl.c_light, wl.cfl_adv, wl.cfl_flavor, wl.area,
                   shape_order=wl.shape_order)
    return cfg, O.init(cfg, wl.n_nu, wl.n_nubar, wl.f_nu, wl.f_nubar, wl.alpha, wl.seed, wl.dirs)


def _box(wl, blocks=304, rk_form=-1):
    from paper_2101_02745_gb300.emu import Box
    box = Box.from_workload(wl)
    box.set_grid(blocks)
    box.set_rk_form(rk_form)
    return box


def _check_steps(wl, box, steps=4, factor=0.917):
    cfg, parts = _oracle(wl)
    # (below Eq. 7's limit: there the order-0 shape meets its discontinuities)
    dt = factor * O.timestep(cfg, O.deposit(cfg, parts))
    box.step(steps, dt)
    O.run(cfg, parts, dt, steps)
    h = box.get_host()
    box.sync()
    assert family_err(h["rho"], pack(parts["rho"])) < 1e-10
    assert family_err(h["rhobar"], pack(parts["rhobar"])) < 1e-10
    assert np.abs(h["z"] - parts["z"]).max() <= 1e-13 * wl.Lz
    return h


# (cells, directions, blocks): the deposit's tiles have 32, 30 (orders 1, 2) or 28
# (order 3) cells.  One tile and one cell more of each; fewer directions than a
# part's least (5), exactly it (6), one more (7), several parts of unequal
# length (13, 50); 304 blocks: parts; 3 blocks with 1 to 3 tiles: longer parts
# (more directions than warps); 2 or 1 blocks with more tiles than blocks: ranges
SPLITS = [(1, 5, 304), (28, 6, 304), (29, 7, 304), (30, 13, 304), (31, 50, 304), (33, 5, 304), (61, 50, 3),
          (30, 50, 1), (61, 13, 1), (97, 50, 2), (1000, 9, 304)]


@pytest.mark.parametrize("order", [0, 1, 2, 3])
@pytest.mark.parametrize("nz,M,blocks", SPLITS)
def test_parts_and_ranges(torch, order, nz, M, blocks):
    wl = W.with_shape(W.random_box(nz, M, seed=nz + 3 * M + order), order)
    a, b = _box(wl, blocks, 0), _box(wl, blocks, 1)
    ha, hb = _check_steps(wl, a), _check_steps(wl, b)
    for k in ha:
        assert np.array_equal(ha[k], hb[k]), k


# slabs of 1, 2, 4 and 8 tiles, each full, with a short last tile and with a short last slab
@pytest.mark.parametrize("nz", [32, 33, 64, 65, 127, 129, 256, 257, 511, 520])
@pytest.mark.parametrize("order", [2, 3])
def test_slabs(torch, order, nz):
    wl = W.with_shape(W.random_box(nz, 9, seed=nz + order), order)
    for blocks in (1, 5, 304):
        _check_steps(wl, _box(wl, blocks, 1))


def test_batch_of_unequal_boxes(torch):
    """Parts across boxes of different tile and direction counts equal each box alone to rounding."""
    from paper_2101_02745_gb300.emu import Box
    wls = [W.random_box(31, 7, seed=1), W.random_box(95, 20, seed=2), W.random_box(1, 5, seed=3)]
    box = Box.from_workloads(wls)
    dts = []
    for wl in wls:
        cfg, parts = _oracle(wl)
        dts.append(0.917 * O.timestep(cfg, O.deposit(cfg, parts)))
    box.batch_set_dt(np.array(dts))
    box.batch_step(4)
    h = box.get_host()
    box.sync()
    p0 = 0
    for wl, dt in zip(wls, dts):
        cfg, parts = _oracle(wl)
        O.run(cfg, parts, dt, 4)
        P = wl.nz * wl.ndir
        assert family_err(h["rho"][:, p0:p0 + P], pack(parts["rho"])) < 1e-10, wl.name
        p0 += P


def _directions(M, seed, longest):
    rng = np.random.default_rng(seed)
    d = rng.normal(size=(M, 3))
    d /= np.linalg.norm(d, axis=1, keepdims=True)
    return d * rng.uniform(0.3, longest, M)[:, None]


@pytest.mark.parametrize("longest", [1.5, 7.0])
@pytest.mark.parametrize("order", [0, 2, 3])
@pytest.mark.parametrize("rk_form", [0, 1])
def test_directions_of_other_lengths(torch, order, rk_form, longest):
    wl = W.with_shape(W.random_box(67, 12, seed=5), order)
    wl.dirs = _directions(12, 1, longest)
    wl.f_nu, wl.f_nubar = wl.f_nu / longest, wl.f_nubar / longest   # (weights stay positive)
    cfg, parts = _oracle(wl)
    box = _box(wl, 304, rk_form)
    grid = O.deposit(cfg, parts)
    s = wl.kappa * longest ** 2 * density_scales(grid)[2]
    A, Aref = box.deposit(0, 0.0).cpu().numpy(), oracle_potential(grid, wl.kappa)
    assert max(family_err(A[9 * f:9 * (f + 1)], Aref[9 * f:9 * (f + 1)], s) for f in range(4)) < 1e-12
    H = box.interpolate_H(0.0).cpu().numpy()
    assert family_err(H, pack(O.hamiltonian(cfg, grid, parts)), s) < 1e-12
    _check_steps(wl, _box(wl, 304, rk_form), factor=0.3 / longest)


@pytest.mark.parametrize("longest", [1.5, 7.0])
def test_directions_of_other_lengths_anywhere(torch, longest):
    wl = W.random_box(67, 9, seed=6)
    cfg, parts = _oracle(wl)
    rng = np.random.default_rng(2)
    z = parts["z"] + rng.uniform(-0.45, 0.45, len(parts)) * wl.dz
    parts["z"] = z - wl.Lz * np.floor(z / wl.Lz)
    parts["omega"] = _directions(len(parts), 3, longest)
    box = _box(wl)
    box.set_host(z=parts["z"].copy(), **{k: parts["omega"][:, i].copy() for i, k in enumerate(("ox", "oy", "oz"))})
    assert box.general()
    dt = 0.3 / longest * O.timestep(cfg, O.deposit(cfg, parts))
    box.step(4, dt)
    O.run(cfg, parts, dt, 4)
    h = box.get_host()
    box.sync()
    assert family_err(h["rho"], pack(parts["rho"])) < 1e-10
    assert family_err(h["rhobar"], pack(parts["rhobar"])) < 1e-10


@pytest.mark.parametrize("blocks", [304, 1])
def test_one_species_absent(torch, blocks):
    wl = W.random_box(61, 13, seed=8)
    wl.n_nubar = np.zeros_like(wl.n_nubar)
    wl.f_nubar = np.zeros_like(wl.f_nubar)
    _check_steps(wl, _box(wl, blocks))


@pytest.mark.parametrize("bad", [np.nan, np.inf])
@pytest.mark.parametrize("rk_form,blocks", [(0, 304), (1, 304), (0, 1), (1, 1)])
def test_nonfinite_is_reported_on_every_split(torch, rk_form, blocks, bad):
    from paper_2101_02745_gb300.emu import EmuError, EMU_ENUMERIC
    wl = W.random_box(61, 13, seed=7)
    box = _box(wl, blocks, rk_form)
    r = box.get_host()["rhobar"].copy()
    r[6, 61 * 5 + 40] = bad
    box.set_host(rhobar=r)
    box.step(1, 1e-13)
    with pytest.raises(EmuError) as ei:
        box.sync()
    assert ei.value.code == EMU_ENUMERIC


@pytest.mark.parametrize("nz,M", [(1, 1), (31, 7), (32, 8), (33, 9), (65, 40)])
def test_weight_gradient_sums(torch, nz, M):
    """Sums of M terms in any order: |error| <= (M + 8) 2^-53 sum |terms|."""
    wl = W.random_box(nz, M, seed=nz + M)
    box = _box(wl)
    rng = np.random.default_rng(nz)
    g = rng.normal(size=(2, M, nz))
    h = box.get_host()
    om = [h[k].reshape(M, nz) for k in ("ox", "oy", "oz")]
    out = box.weight_gradient(*(torch.tensor(v.ravel(), device="cuda") for v in g)).cpu().numpy()
    box.sync()
    f = wl.area * (wl.Lz / nz) / M
    for sp in range(2):
        rows = [(sp, g[sp])] + [(2 + 3 * sp + i, 3.0 * om[i] * g[sp]) for i in range(3)]
        for k, terms in rows:
            bound = (M + 8) * 2.0 ** -53 * np.abs(terms).sum(axis=0)
            assert np.all(np.abs(out[k] / f - terms.sum(axis=0)) <= bound + 1e-300), k
