"""Gram-Schmidt by block passes (FMA build, one launch per block of four basis
vectors: the path of grids beyond the column kernel's reach), forced on small
problems with rok_set_persistent(False).

On the GPU's own basis: orthonormality, and the Arnoldi relation J v_j =
V H[:, j] + h_{j+1,j} v_{j+1} with the same FD product (its rounding is the same
in both uses).  Each of the j + 1 <= 18 projections of a column rounds a few
times (u = 2^-53) at the size of w, so 1e-13 of ||J v_j|| leaves a margin of
about 20; modified Gram-Schmidt loses orthogonality in proportion to the
conditioning of the Krylov vectors (1e-9 bounds it on these cases)."""
import numpy as np
import pytest

from oracle import integrators as I
from paper_1607_06834_gb300 import workloads as W
from tests.gpu_common import dev, host

pytestmark = pytest.mark.gpu


@pytest.fixture(scope='module')
def rok():
    from paper_1607_06834_gb300 import rok as r
    return r


def _cases():
    out = {}
    for n in (41, 2047, 2048, 4099):            # odd lengths, one and several chunks
        out['lorenz%d' % n] = W.lorenz96(n)
    p, y = W.taylor_green(48, reynolds=300.0)
    out['tgv48'] = (p, np.ascontiguousarray(y + 0.01 * W.random_smooth_state(p, seed=1)))
    p, y = W.isentropic_vortex(512)             # more chunks than thread blocks
    out['vortex512'] = (p, y)
    return out


CASES = _cases()


@pytest.mark.parametrize('M', [1, 4, 5, 18])    # a part of a block, a block, one more, several
@pytest.mark.parametrize('name', CASES)
def test_block_passes_give_an_arnoldi_basis(rok, name, M):
    prob, y = CASES[name]
    ctx = rok.rok_init(prob, krylov_max=M)
    rok.rok_set_persistent(ctx, False)
    yd = dev(y)
    V, H, me = rok.rok_arnoldi(ctx, yd, M)
    assert me == M
    G = host(V @ V.T)
    assert np.abs(G - np.eye(M)).max() <= 1e-9
    f = rok.rok_residual(ctx, yd)
    eps = I.fd_eps(I.norm(y))
    worst = 0.0
    for j in range(M - 1):
        jv = rok.rok_jvp(ctx, yd, V[j].reshape(yd.shape).contiguous(), fy=f, eps=eps).ravel()
        r = jv - H[:j + 2, j] @ V[:j + 2]
        worst = max(worst, float(r.norm() / jv.norm()))
    print('\n[gs] %s M %d: orthogonality %.1e, Arnoldi relation %.1e' % (name, M, np.abs(G - np.eye(M)).max(), worst))
    assert worst <= 1e-13
    Hh = host(H)
    assert np.all(np.tril(Hh, -2) == 0.0) and np.all(np.diag(Hh, -1) > 0.0)


@pytest.mark.parametrize('period', [4, 5, 10])
def test_block_passes_stop_at_a_breakdown(rok, period):
    # a p-periodic Lorenz-96 state: the Krylov space has dimension p (the last
    # block full, with one vector, with two)
    prob, y = W.lorenz96(20, seed=3)
    y = np.ascontiguousarray(np.tile(y[:period], 20 // period))
    ctx = rok.rok_init(prob, krylov_max=12)
    rok.rok_set_persistent(ctx, False)
    V, H, me = rok.rok_arnoldi(ctx, dev(y), 12)
    assert me == period
    assert np.abs(host(V @ V.T) - np.eye(me)).max() <= 1e-9
