"""Rounding errors of the FMA build's residual against an evaluation in long double,
beside those of the strict build (plain binary64), zone by zone and component by
component: the fixed-point faces may not be less accurate than binary64 where the
flow is far from the state in cell 0, where velocities are small, or where only
viscous terms are left.

Bar: the rms error over the zone at most 1.5 times the strict build's (two
binary64 evaluations in different orders differ by up to about that factor), plus
u / 20 of the component's own rms (u = 2^-53) where the strict build's error vanishes."""
import numpy as np
import pytest

from paper_1607_06834_gb300 import workloads as W
from tests.gpu_common import U, dev, host
from tests.long_residual import residual

pytestmark = pytest.mark.gpu

NX, NY = 64, 48


@pytest.fixture(scope='module')
def rok():
    from paper_1607_06834_gb300 import rok as r
    return r


def _modes(seed, n=4):
    rng = np.random.default_rng(seed)
    s, t = 2 * np.pi * np.arange(NX) / NX, 2 * np.pi * np.arange(NY) / NY
    f = np.zeros((NY, NX))
    for _ in range(n):
        a, b = rng.integers(1, 4, 2)
        ph = rng.uniform(0, 2 * np.pi, 2)
        f += rng.normal() * np.outer(np.cos(b * t + ph[1]), np.sin(a * s + ph[0]))
    return f / np.abs(f).max()


def _prob(gas, mu=1e-3):
    kw = dict(kind=W.EULER) if gas == 'euler' else dict(kind=W.NAVIER_STOKES, mu=mu)
    if gas == 'sutherland':
        kw.update(sutherland_s=0.4, t_ref=1.0)
    if gas == 'aligned':   # the same box as a curvilinear grid: its metrics are exact
        kw['xv'], kw['yv'] = np.meshgrid(np.arange(NX + 1.0), np.arange(NY + 1.0))
        kw['name'] = gas
    return W.FlowProblem(nx=NX, ny=NY, lx=float(NX), ly=float(NY), **kw)


def _state(prob, rho, u, v, p):
    rho, u, v, p = np.broadcast_arrays(*(np.asarray(a, dtype=np.float64) for a in (rho, u, v, p, np.zeros((NY, NX)))))[:4]
    return np.ascontiguousarray(np.stack([rho, rho * u, rho * v, p / (prob.gamma - 1.0) + 0.5 * rho * (u * u + v * v)]))


def _zone(rho, p, mach=0.3):
    """A smooth flow of density rho and pressure p, with a patch of (1, 1) around cell 0;
    the zone leaves the patch out."""
    i, j = np.meshgrid(np.arange(NX), np.arange(NY))
    d = np.hypot(np.minimum(i, NX - i), np.minimum(j, NY - j))
    w = 0.5 * (1.0 - np.tanh((d - 10.0) / 3.0))
    r, q = rho ** (1.0 - w), p ** (1.0 - w)
    c = np.sqrt(1.4 * q / r)
    return (r * (1.0 + 0.02 * _modes(1)), c * mach * (0.8 + 0.3 * _modes(2)), c * mach * (0.6 + 0.3 * _modes(3)),
            q * (1.0 + 0.02 * _modes(4)), d > 22.0)


def _states():
    t = 2 * np.pi * np.arange(NX) / NX
    s = (2 * np.pi * np.arange(NY) / NY)[:, None]
    everywhere = np.ones((NY, NX), dtype=bool)
    out = {'like-cell-0': _zone(1.0, 1.0), 'light': _zone(0.3, 0.3), 'low-pressure': _zone(1.0, 0.08),
           'light-low-pressure': _zone(0.3, 0.08), 'dense': _zone(20.0, 30.0), 'far': _zone(1e-4, 1e-5)}
    for m in (1e-1, 1e-2, 1e-3, 1e-5, 1e-8):
        out['mach-%g' % m] = (1.0 + 0.05 * _modes(5), m * (0.7 + 0.4 * _modes(6)), m * (0.5 + 0.4 * _modes(7)),
                              1.0 + m * m * _modes(8), everywhere)
    for a in (1e-3, 1e-6, 1e-9):   # a small transverse velocity carried along by the flow
        out['passive-%g' % a] = (1.0 + 0.1 * np.sin(t), 0.35, a * np.cos(2 * t), 1.0, everywhere)
    for a in (1e-1, 1e-5, 1e-12):   # a shear layer at rest but for its own velocity
        out['shear-%g' % a] = (1.0, a * np.sin(s), 0.0, 1.0, everywhere)
    out['conduction'] = (1.0 + 0.1 * np.sin(s) * np.cos(t), 0.0, 0.0, 1.0, everywhere)
    out['supersonic'] = (1.0 + 0.05 * _modes(5), 3.0 + 0.1 * _modes(6), 1.0 + 0.1 * _modes(7), 1.0 + 0.05 * _modes(8),
                         everywhere)
    return out


STATES = _states()


def _rms(x):
    return np.sqrt((x.astype(np.float64) ** 2).mean())


@pytest.mark.parametrize('gas', ['euler', 'navier-stokes', 'sutherland', 'aligned'])
@pytest.mark.parametrize('name', STATES)
def test_errors_are_those_of_binary64(rok, gas, name):
    *q, zone = STATES[name]
    prob = _prob(gas)
    y = _state(prob, *q)
    exact = residual(prob, y)
    f, fs = (host(rok.rok_residual(rok.rok_init(prob, krylov_max=1, rounding=r), dev(y)))
             for r in (rok.ROK_ROUND_FAST, rok.ROK_ROUND_STRICT))
    ratios, bad = [], []
    for k in range(4):
        e, es = _rms((f - exact)[k][zone]), _rms((fs - exact)[k][zone])
        bar = 1.5 * es + U / 20 * _rms(exact[k][zone])
        ratios.append(e / es if es > 0.0 else float(e > 0.0))
        if e > bar:
            bad.append(k)
    print('\n[fixed precision] %s %s: rms error / binary64 %s' % (gas, name, ' '.join('%.2f' % r for r in ratios)))
    assert not bad, (gas, name, ratios)
