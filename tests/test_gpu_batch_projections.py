"""Projections of a batch's Gram-Schmidt passes on the integer pipe, and the
binary64 sums that take their place for operands of zeros: a gas at rest but for
a bump in one corner (f, and the Krylov vectors, vanish exactly in most lanes),
beside a smooth flow.  The FMA build's step agrees with the strict one to 1e-6
of its change (the FD quotients amplify last-bit differences by 1/eps, 1e-8 of
J v)."""
import numpy as np
import pytest

from paper_1607_06834_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _bump(n):
    """Density and pressure bump of 1e-2 over n / 8 cells of a gas at rest; h at CFL 0.2."""
    prob, _ = W.isentropic_vortex(8)
    prob.nx = prob.ny = n
    rho, p = np.ones((n, n)), np.full((n, n), 1.0 / prob.gamma)
    k = n // 8
    s = 1e-2 * np.outer(np.hanning(k + 2)[1:-1], np.hanning(k + 2)[1:-1])
    rho[3:3 + k, 5:5 + k] += s
    p[3:3 + k, 5:5 + k] *= 1.0 + s
    return prob, np.stack([rho, 0.0 * rho, 0.0 * rho, p / (prob.gamma - 1.0)]), 0.2 * prob.lx / n


@pytest.mark.parametrize('m', [1, 4, 5, 9])     # a part of a block, a block, one more, several
def test_batched_projections_with_lanes_of_zeros(m):
    from paper_1607_06834_gb300 import rok
    prob, y = W.taylor_green(40, reynolds=300.0)
    parts = [_bump(32), _bump(57), _bump(96), (prob, y, 0.002)]
    out = []
    for rounding in (rok.ROK_ROUND_FAST, rok.ROK_ROUND_STRICT):
        b = rok.rok_batch_init([q[0] for q in parts], krylov_max=m, rounding=rounding)
        z = b.pack([q[1] for q in parts])
        rok.rok_batch_step(b, z, [q[2] for q in parts], m)
        out.append(b.unpack(z))
    for (prob, y, _), a, s in zip(parts, *out):
        change = np.abs(s - y).max()
        assert change > 0.0 and np.abs(a - s).max() <= 1e-6 * change, prob.nx
