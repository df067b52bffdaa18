"""Binary32 basis entries widened on the integer pipe (projections and stage
vectors of the FMA build): zeros, subnormals and normal entries side by side.

Lorenz-96 without forcing from a state of isolated entries of 1 over a floor of
1e-42: f, and with it the binary32 basis, holds exact zeros, subnormals (1e-42
to 1e-39) and normal entries.  Both builds take binary32 Gram-Schmidt (CGS2
against MGS), so a step of the FMA build agrees with the strict one, which
converts by instruction, to some tens of u32 = 6e-8 of the change: 1e-5."""
import numpy as np
import pytest

from paper_1607_06834_gb300 import workloads as W
from tests.gpu_common import dev, host

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize('n', [64, 4096])       # one CTA, several
@pytest.mark.parametrize('floor', [0.0, 1e-42, 1e-39])
def test_mixed_step_with_zero_and_subnormal_basis_entries(n, floor):
    from paper_1607_06834_gb300 import rok
    prob, y = W.lorenz96(n, forcing=0.0)
    y = np.full_like(y, floor)
    flat = y.ravel()
    flat[5::32] = 1.0
    flat[6::32] = -0.5
    flat[7::32] = 0.75
    out = []
    for rounding in (rok.ROK_ROUND_FAST, rok.ROK_ROUND_STRICT):
        ctx = rok.rok_init(prob, krylov_max=4, rounding=rounding, basis=rok.ROK_BASIS_FP32)
        yd = dev(y)
        rok.rok_step(ctx, yd, 0.05, 4)
        out.append(host(yd))
    change = np.abs(out[1] - y).max()
    assert change > 0.0 and np.isfinite(out[0]).all()
    assert np.abs(out[0] - out[1]).max() <= 1e-5 * change
