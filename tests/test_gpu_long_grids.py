"""Grids of few columns and very many rows: the tiles' row index is a grid dimension of the
launch, which holds 65535 tiles, so the tallest grid a launch takes is set by the
tile's height (16 rows: 1,048,560).  Every row must see what a short periodic grid sees."""
import numpy as np
import pytest

from paper_1607_06834_gb300 import workloads as W
from tests.gpu_common import dev, host

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize('curv', [False, True])
@pytest.mark.parametrize('ny', [458752, 983040, 1048544])
def test_residual_of_a_tall_grid_repeats_that_of_a_short_one(curv, ny):
    from paper_1607_06834_gb300 import rok
    nx, period = 2, 32
    out = []
    rng = np.random.default_rng(1)
    q = np.array([1.0, 0.3, -0.2, 2.7])[:, None, None] * (1.0 + 0.05 * rng.uniform(-1, 1, (4, period, nx)))
    for rows in (period, ny):
        prob = W.FlowProblem(kind=W.EULER, nx=nx, ny=rows, lx=float(nx), ly=float(rows))
        if curv:
            prob.xv, prob.yv = np.meshgrid(np.arange(nx + 1.0), np.arange(rows + 1.0))
        y = np.ascontiguousarray(np.tile(q, (1, rows // period, 1)))
        out.append(host(rok.rok_residual(rok.rok_init(prob, krylov_max=0), dev(y))))
    assert np.array_equal(out[1].reshape(4, -1, period, nx), np.broadcast_to(out[0][:, None], (4, ny // period, period, nx)))
