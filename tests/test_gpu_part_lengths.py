"""Parts of a tile at the lines of their least length (boxes of one tile, by the
grid's blocks): 4 directions below 1.5 units a block, 4 in the deposit and 6 in the
RK stage below 2, 6 from there on; fewer directions than a part's least, exactly
it and one more.

The first steps against the oracle 1e-10 (family-wise); the RK stage's two work
splits bitwise."""
import numpy as np
import pytest

from paper_2101_02745_gb300 import workloads as W
from tests.test_gpu_work_splits import _box, _check_steps, torch  # noqa: F401

pytestmark = pytest.mark.gpu


# (directions, blocks)
@pytest.mark.parametrize("M,blocks", [(3, 304), (4, 304), (5, 304), (11, 8), (12, 8), (13, 8), (15, 8), (16, 8),
                                      (17, 8), (6, 3), (7, 3), (4, 1), (5, 1)])
@pytest.mark.parametrize("order", [0, 2, 3])
def test_part_lengths(torch, order, M, blocks):  # noqa: F811
    wl = W.with_shape(W.random_box(27, M, seed=M + order), order)
    ha, hb = (_check_steps(wl, _box(wl, blocks, rk)) for rk in (0, 1))
    for k in ha:
        assert np.array_equal(ha[k], hb[k]), k
