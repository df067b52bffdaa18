"""The multipliers of the stage systems' LU round as divisions do (FMA build as strict build).
L = I - h gamma H is upper Hessenberg: while no rows are exchanged, step k divides one
entry, the untouched -h gamma H[k+1, k], by the pivot.  The factors are read from
the step's tape, found by the Hessenberg matrix that lies before them."""
import numpy as np
import pytest

from paper_1607_06834_gb300 import workloads as W
from tests.gpu_common import dev, host

pytestmark = pytest.mark.gpu

STRIDE = 64
GAMMA = 0.5728160624821349


@pytest.mark.parametrize('rounding', ['fast', 'strict'])
@pytest.mark.parametrize('M', [2, 12, 30])
def test_multipliers_are_rounded_quotients(M, rounding):
    from paper_1607_06834_gb300 import rok
    prob, y0 = W.taylor_green(32, reynolds=300.0)
    y = np.ascontiguousarray(y0 + 0.01 * W.random_smooth_state(prob, seed=2))
    ctx = rok.rok_init(prob, krylov_max=M, rounding=rok.ROK_ROUND_FAST if rounding == 'fast' else rok.ROK_ROUND_STRICT)
    _, H, me = rok.rok_arnoldi(ctx, dev(y), M)
    assert me == M
    h = 0.02 / np.abs(host(H)).max()   # diagonally dominant: no exchanges
    d = host(rok.rok_step_record(ctx, dev(y), h, M)).view(np.float64)
    start = [k for k in np.flatnonzero(d[:4096] == host(H)[0, 0]) if d[k + STRIDE] == host(H)[1, 0]]
    assert len(start) == 1
    H = d[start[0]:start[0] + (STRIDE + 1) * STRIDE].reshape(-1, STRIDE)
    LU = d[start[0] + H.size:start[0] + H.size + STRIDE * STRIDE].reshape(-1, STRIDE)
    hg = h * GAMMA
    for k in range(M - 1):
        assert abs(LU[k, k]) > abs(hg * H[k + 1, k])
        assert LU[k + 1, k] == -(hg * H[k + 1, k]) / LU[k, k], (k, LU[k + 1, k])
