"""The even split of the FMA build's Gram-Schmidt columns and projections over
CTAs, at sizes where it can go wrong: one CTA, ranges of one entry a thread and
one more, last CTAs nearly empty, and every number of entries a thread.

On the GPU's own basis: orthonormality and the Arnoldi relation with the same FD
product, with the bounds of the block-pass tests (1e-9: conditioning of the
Krylov vectors; 1e-13 of ||J v_j||: each of at most 9 projections rounds a few
times at the size of w).  The projections of the stage systems enter the
step: FMA against strict build to 1e-6 of the step's change (the FD quotients
amplify last-bit differences by 1/eps, 1e-8 of J v)."""
import numpy as np
import pytest

from oracle import integrators as I
from paper_1607_06834_gb300 import workloads as W
from tests.gpu_common import dev, host

pytestmark = pytest.mark.gpu

# 77220 = 152 * 508 + 4: rounding the range up to a multiple of 4 would leave the last of 152 CTAs empty
SIZES = [40, 510, 512, 514, 1026, 16384, 20004, 77220, 77824, 79000, 233472, 311300, 400000, 544768, 622592, 700000,
         900000, 1000000, 1245184, 1245188, 1300004, 2500000]   # the last three: tiles of a longer range


@pytest.mark.parametrize('n', SIZES)
def test_columns_and_projections_over_the_even_split(n):
    from paper_1607_06834_gb300 import rok
    M = 6
    prob, y = W.lorenz96(n, seed=n)
    ctx = rok.rok_init(prob, krylov_max=M)
    yd = dev(y)
    V, H, me = rok.rok_arnoldi(ctx, yd, M)
    assert me == M
    assert np.abs(host(V @ V.T) - np.eye(M)).max() <= 1e-9
    f = rok.rok_residual(ctx, yd)
    eps = I.fd_eps(I.norm(y))
    for j in range(M - 1):
        jv = rok.rok_jvp(ctx, yd, V[j].reshape(yd.shape).contiguous(), fy=f, eps=eps).ravel()
        assert float((jv - H[:j + 2, j] @ V[:j + 2]).norm() / jv.norm()) <= 1e-13
    out = []
    for rounding in (rok.ROK_ROUND_FAST, rok.ROK_ROUND_STRICT):
        c = rok.rok_init(prob, krylov_max=M, rounding=rounding)
        z = dev(y)
        rok.rok_step(c, z, 0.01, M)
        out.append(host(z))
    assert np.abs(out[0] - out[1]).max() <= 1e-6 * np.abs(out[1] - y).max()
