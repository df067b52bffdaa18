"""The fixed-point stencil of the FMA build at values that lie exactly on the ends of its
ranges: powers of two in density and pressure ratios, velocities and sound speeds,
and one unit in the last place beside them, against the CPU oracle.

A power of two below the largest density of a face is an ordinary contact (ratio
4, say), and its reciprocal is a power of two as well: the one place where a number
fills its format to the last bit.

Bar: that of the FMA build's residual elsewhere, 64 u (max|F| + max|viscous
flux|) / h per entry, u = 2^-53 (a few rounding units for each of the four faces a
cell sums).  A velocity of the wrong sign is an error of order max|F| / h."""
import numpy as np
import pytest

from oracle import core
from paper_1607_06834_gb300 import workloads as W
from tests.gpu_common import U, dev, flux_scale, host

pytestmark = pytest.mark.gpu


@pytest.fixture(scope='module')
def rok():
    from paper_1607_06834_gb300 import rok as r
    return r


GAS = {
    'euler': dict(kind=W.EULER),
    'navier-stokes': dict(kind=W.NAVIER_STOKES, mu=1e-3),
    'sutherland': dict(kind=W.NAVIER_STOKES, mu=1e-3, sutherland_s=0.4, t_ref=1.0),
    'curvilinear': dict(kind=W.NAVIER_STOKES, mu=1e-3),
}
NX, NY = 42, 24


def _problem(gas):
    prob = W.FlowProblem(nx=NX, ny=NY, lx=float(NX), ly=float(NY), **GAS[gas])
    if gas == 'curvilinear':
        prob.xv, prob.yv = W.perturbed_box_grid(NX, NY, float(NX), float(NY), amp=0.2, seed=3)
    return prob


def _side(prob, rho, u, v, p):
    return np.array([rho, rho * u, rho * v, p / (prob.gamma - 1.0) + 0.5 * rho * (u * u + v * v)])


def _steps(prob, levels, along=0):
    """Primitive states in bands along i, along j and along the diagonal (jumps of every
    orientation): two levels as blocks of cells, more as a staircase down and up again, one
    cell a level, along i, j or the diagonal."""
    n = len(levels)
    q = np.stack([_side(prob, *s) for s in levels])          # (level, variable)
    i, j = np.meshgrid(np.arange(NX), np.arange(NY))
    if n == 2:
        k = ((i >= 9) & (i < 21)) | ((j >= 14) & (j < 20)) | ((i + j) % 64 > 52)
    else:
        t = {0: i, 1: j, 2: i + j}[along]
        k = np.abs((t + n - 1) % (2 * n - 2) - (n - 1))   # 0 .. n - 1 .. 0
    return np.ascontiguousarray(np.moveaxis(q[k.astype(int)], -1, 0))


def _near(x):
    return {'': x, '+ulp': np.nextafter(x, np.inf), '-ulp': np.nextafter(x, 0.0)}


def _states():
    out = {}
    for k in (1, 2):           # contacts (unlimited MUSCL keeps them positive up to ratios of about 6)
        for tag, r in _near(2.0 ** -k).items():
            out['contact-2^-%d%s' % (k, tag)] = ((1.0, 0.5, 0.2, 1.0), (r, 0.5, 0.2, 1.0))
        out['contact-2^%d' % k] = ((1.0, 0.5, 0.2, 1.0), (2.0 ** k, 0.5, 0.2, 1.0))
    for k in (1, 2):           # pressure steps
        for tag, r in _near(2.0 ** -k).items():
            out['pressure-2^-%d%s' % (k, tag)] = ((1.0, 0.25, -0.125, 1.0), (0.75, 0.25, -0.125, r))
    for k in (1, 2):           # staircases: reconstructed states are powers of two as well
        for tag, r in _near(2.0 ** -k).items():
            out['density-stairs-2^-%d%s' % (k, tag)] = tuple((r ** e, 0.5, 0.2, 1.0) for e in range(4))
            out['pressure-stairs-2^-%d%s' % (k, tag)] = tuple((1.0, 0.5, 0.2, r ** e) for e in range(4))
            out['both-stairs-2^-%d%s' % (k, tag)] = tuple((r ** e, 0.5, 0.2, r ** e) for e in range(4))
    for v in (0.5, 1.0, 2.0, 4.0):   # velocities of exactly a power of two beside p = rho = 1
        for tag, s in _near(v).items():
            out['velocity-%g%s' % (v, tag)] = ((1.0, s, 0.25 * s, 1.0), (0.875, s, 0.25 * s, 0.875))
    for m in (1.0, 4.0, 5.0, 6.0, 7.0):   # c^2 exactly one, at supersonic Mach numbers
        out['mach-%g' % m] = ((1.0, m, 0.0, 1.0 / 1.4), (1.0 + 2.0 ** -20, m, 0.0, 1.0 / 1.4))
    return out


STATES = _states()


def _bar(prob, y):
    h = 1.0
    if prob.xv is not None:
        h = min(np.hypot(np.diff(prob.xv, axis=a), np.diff(prob.yv, axis=a)).min() for a in (0, 1))
    b = flux_scale(prob, y)
    if prob.mu > 0.0:
        vel = np.abs(y[1:3] / y[0]).max()
        T = ((prob.gamma - 1.0) * y[3] / y[0]).max()
        g = max((T / prob.t_ref) ** 1.5, 1.0) if prob.sutherland_s > 0.0 else 1.0
        b += prob.mu * g / (h * h) * (vel * vel + vel + prob.gamma / ((prob.gamma - 1.0) * prob.prandtl) * T)
    return 64 * U * b


def _check(prob, y, f, what):
    fo = core.residual(prob, y)
    assert np.isfinite(fo).all(), what
    err, bar = np.abs(f - fo).max(), _bar(prob, y)
    assert err <= bar, (what, err / bar)


@pytest.mark.parametrize('gas', GAS)
def test_steps_on_the_ends_of_the_ranges(rok, gas):
    prob = _problem(gas)
    ctx = rok.rok_init(prob, krylov_max=1)
    for name, levels in STATES.items():
        for lv in (levels, levels[::-1]):   # which of them fills cell 0
            for along in range(3 if len(lv) > 2 else 1):
                y = _steps(prob, lv, along)
                _check(prob, y, host(rok.rok_residual(ctx, dev(y))), (gas, name, along))


@pytest.mark.parametrize('gas', ['euler', 'navier-stokes', 'sutherland'])
def test_steps_on_the_ends_of_the_ranges_in_a_batch(rok, gas):
    probs = [_problem(gas) for _ in STATES]
    states = [_steps(p, lv) for p, lv in zip(probs, STATES.values())]
    b = rok.rok_batch_init(probs, krylov_max=1)
    f = b.unpack(rok.rok_batch_residual(b, b.pack(states)))
    for name, p, y, fk in zip(STATES, probs, states, f):
        _check(p, y, fk, (gas, name))
