"""Residual VJP and exact JVP over the branches of the face flux: subsonic waves
(the reduced acoustic sums), waves inside Harten's fix (|u -+ c| < delta),
supersonic ones and a normal velocity of exactly zero, in either direction,
against the oracle's complex-step Jacobian.  Both are derivatives of the same
discrete residual, of at most a few hundred roundings an entry: 1e-12 of the
result's size, as for the other derivative tests."""
import numpy as np
import pytest

from oracle import adjoint as A
from oracle import core
from paper_1607_06834_gb300 import workloads as W
from tests.gpu_common import dev, host

pytestmark = pytest.mark.gpu

GRIDS = {
    'uniform': dict(nx=18, ny=17, lx=2.0, ly=1.7, mu=0.01),
    'uniform-sutherland': dict(nx=17, ny=18, lx=2.0, ly=1.7, mu=0.01, sutherland_s=0.4, t_ref=0.5),
    'curvilinear': dict(nx=18, ny=17, mu=0.01, sutherland_s=0.4, t_ref=0.5),
}
STREAMS = {'rest': (0.0, 0.0), 'sub': (0.4, -0.3), 'fix': (1.0, -0.95), 'sonic-left': (-1.0, 0.2), 'super': (-2.5, 1.8)}


@pytest.mark.parametrize('grid', GRIDS)
@pytest.mark.parametrize('stream', STREAMS)
def test_derivative_products_over_the_wave_branches(grid, stream):
    from paper_1607_06834_gb300 import rok
    kw = dict(GRIDS[grid])
    if grid == 'curvilinear':
        kw['xv'], kw['yv'] = W.perturbed_box_grid(kw['nx'], kw['ny'], 2.0, 1.7, amp=0.3, seed=6)
    prob = W.FlowProblem(kind=W.NAVIER_STOKES, **kw)
    rng = np.random.default_rng(3)
    shape = (prob.ny, prob.nx)
    rho = 1.0 + 0.1 * rng.uniform(-1.0, 1.0, shape)
    p = (1.0 + 0.1 * rng.uniform(-1.0, 1.0, shape)) / prob.gamma      # c about 1
    u, v = (s + (0.05 * rng.uniform(-1.0, 1.0, shape) if s else 0.0) + 0.0 * rho for s in STREAMS[stream])
    y = np.stack([rho, rho * u, rho * v, p / (prob.gamma - 1.0) + 0.5 * rho * (u * u + v * v)])
    if stream == 'rest':
        p0 = np.full(shape, 1.0 / prob.gamma)     # no jumps of pressure: the normal velocity stays exactly zero
        y[3] = p0 / (prob.gamma - 1.0)
    d = rng.standard_normal(y.shape)
    ctx = rok.rok_init(prob, krylov_max=4)
    got = rok.rok_vjp(ctx, dev(y), dev(d))
    ref = A.residual_vjp(prob, y, d)
    if stream == 'rest':   # |u| is not differentiable at 0: the one-sided derivative, by the dual numbers alone
        jv = host(rok.rok_jvp(ctx, dev(y), dev(d), mode=rok.ROK_JVP_EXACT))
        strict = rok.rok_init(prob, krylov_max=4, rounding=rok.ROK_ROUND_STRICT)
        js = host(rok.rok_jvp(strict, dev(y), dev(d), mode=rok.ROK_JVP_EXACT))
        assert np.linalg.norm(jv - js) <= 1e-12 * np.linalg.norm(js)
        assert abs(np.sum(d * js) - np.sum(host(got) * d)) <= 1e-12 * np.sum(np.abs(d * js))
        return
    assert np.abs(host(got) - ref).max() <= 1e-12 * np.abs(ref).max()
    jv = host(rok.rok_jvp(ctx, dev(y), dev(d), mode=rok.ROK_JVP_EXACT))
    jo = core.jvp_exact(prob, y, d)
    assert np.linalg.norm(jv - jo) <= 1e-12 * np.linalg.norm(jo)
    plain, _ = rok.rok_vjp(ctx, dev(y), dev(d), mubar=True)      # the viscosity adjoint changes nothing else
    assert bool((plain == got).all())
