"""The fixed-point stencil of the FMA build (uniform and curvilinear grids) against the CPU
oracle at the edges of its ranges: faces inside the windows run on the integer
pipe, all others in binary64, face by face.

Bar (as for the FMA build's residual elsewhere): 64 u max|F|/h per entry, u =
2^-53, F the physical flux, h the smallest cell width.  The fixed-point faces
carry a few 2^-60 of the scale units, the binary64 primitives and faces a few
u, and a cell sums four faces; the bar was set before the first run."""
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


def _flow(nx, ny, mach, rho=1.0, p=1.0, amp=0.05, seed=0, kind=W.NAVIER_STOKES, **kw):
    """A perturbed uniform stream of the given density, pressure and Mach number."""
    prob = W.FlowProblem(kind=kind, nx=nx, ny=ny, lx=1.0, ly=1.0 * ny / nx, **kw)
    rng = np.random.default_rng(seed)
    c = np.sqrt(prob.gamma * p / rho)
    r = rho * (1.0 + amp * rng.uniform(-1, 1, (ny, nx)))
    q = p * (1.0 + amp * rng.uniform(-1, 1, (ny, nx)))
    u = c * (mach * 0.8 + amp * rng.uniform(-1, 1, (ny, nx)))
    v = c * (mach * 0.6 + amp * rng.uniform(-1, 1, (ny, nx)))
    y = np.stack([r, r * u, r * v, q / (prob.gamma - 1.0) + 0.5 * r * (u * u + v * v)])
    return prob, np.ascontiguousarray(y)


def _cases():
    visc = dict(mu=1e-3)
    out = {
        'ragged-33x17': _flow(33, 17, 0.3, **visc),
        'tiles-16x16-213x199': _flow(213, 199, 0.3, **visc),
        'tiles-32x15-1001x690': _flow(1001, 690, 0.3, kind=W.EULER),
        'tiles-16x16-412x397': _flow(412, 397, 0.3, **visc),
        'smallest-2x2': _flow(2, 2, 0.3, **visc),
        'si-units': _flow(40, 24, 0.2, rho=1.2, p=101325.0, mu=1.8e-5),
        'tiny-units': _flow(24, 24, 0.2, rho=3e-9, p=2e-13, mu=1e-14),
        'low-mach': _flow(24, 20, 1e-3, amp=1e-4, **visc),
        'transonic': _flow(48, 20, 1.0, amp=0.2, **visc),       # Harten's fix acts on many faces
        'supersonic-2': _flow(32, 32, 2.0, **visc),             # the supersonic form
        'supersonic-6': _flow(32, 16, 6.0, **visc),             # velocities outside the window
        'strong-jumps': _flow(40, 40, 0.5, amp=0.6, kind=W.EULER),
        'viscous-cells': _flow(24, 24, 0.1, mu=50.0),           # viscous coefficients above the units
        'sutherland': _flow(36, 20, 0.3, mu=1e-3, sutherland_s=0.4, t_ref=0.9),
        'sutherland-cold-ref': _flow(20, 36, 0.3, mu=1e-3, sutherland_s=0.4, t_ref=9.0),   # T / t_ref outside
        'monatomic': _flow(24, 24, 0.4, gamma=5.0 / 3.0, **visc),
        'gamma-1.15': _flow(24, 24, 0.4, gamma=1.15, **visc),   # outside the constants' range: binary64 kernel
        'kappa-1-no-fix': _flow(24, 24, 0.4, muscl_kappa=-1.0, entropy_fix=0.0, **visc),
    }
    prob, y = _flow(40, 32, 0.2, **visc)
    y = y.copy()
    y[:, 0, 0] *= 2.0 ** 20       # cell 0, which sets the units, far from the rest
    out['odd-cell-0'] = (prob, y)
    prob, y = _flow(40, 32, 0.2, kind=W.EULER)
    y = y.copy()
    y[:, 10:14, 20:25] *= 1e-4    # a light pocket: its faces in binary64, the rest in fixed point
    out['light-pocket'] = (prob, y)
    return out


def _curv(nx, ny, seed, state_amp=0.05, scale=1.0, amp=0.25, bc=None, **kw):
    """A perturbed box (cells of several shapes) with a smooth random state in scaled units."""
    xv, yv = W.perturbed_box_grid(nx, ny, 2.0, 1.7, amp=amp, seed=seed)
    prob = W.FlowProblem(kind=kw.pop('kind', W.NAVIER_STOKES), nx=nx, ny=ny, xv=xv, yv=yv,
                         bc=bc or (W.PERIODIC,) * 4, **kw)
    y = W.random_smooth_state(prob, seed=seed, amp=state_amp)
    u = np.sqrt(scale)
    y = y * np.array([1.0, u, u, scale])[:, None, None]   # pressures and T in units of `scale`
    q = np.array([1.0, 0.3 * u, -0.2 * u, scale * (1.0 / prob.gamma / (prob.gamma - 1.0) + 0.065)])
    prob.q_inf = tuple(float(x) for x in q)
    return prob, np.ascontiguousarray(y)


def _curv_cases():
    walls = (W.WALL, W.WALL, W.WALL, W.FARFIELD)
    out = {
        'curv-periodic-37x29': _curv(37, 29, 1, mu=0.01),
        'curv-walls-farfield': _curv(33, 34, 2, mu=0.01, bc=walls),
        'curv-euler-farfield': _curv(35, 18, 3, kind=W.EULER, bc=(W.FARFIELD,) * 4),
        'curv-sutherland-walls': _curv(20, 47, 4, mu=0.01, bc=walls, sutherland_s=0.4, t_ref=0.7),
        'curv-large-units': _curv(24, 24, 5, mu=0.01, scale=3e5, bc=walls),
        'curv-aligned-box': _curv(24, 24, 6, mu=0.01, amp=0.0),   # normals of one exactly
        'curv-2x2': _curv(2, 2, 7, mu=0.01, amp=0.0, bc=walls),
        'curv-strong-jumps': _curv(32, 32, 8, mu=0.01, state_amp=0.35, bc=walls),
        'curv-viscous-cells': _curv(24, 24, 9, mu=3e3, bc=walls),
    }
    prob, y = _curv(30, 26, 10, mu=0.01, bc=walls)
    prob.q_inf = tuple(1e4 * q for q in prob.q_inf)   # the free stream outside the window
    out['curv-odd-free-stream'] = (prob, y)
    for name, kw in (('ogrid-impulsive', {}), ('ogrid-constant-mu', {'sutherland': False})):
        prob, y, _ = W.cylinder_ogrid(40, 72, **kw)
        out[name] = (prob, y)
        out[name + '-perturbed'] = (prob, np.ascontiguousarray(y + 0.02 * W.random_smooth_state(prob, seed=5)))
    return out


CASES = {**_cases(), **_curv_cases()}


def _width(prob):
    e = [np.hypot(np.diff(prob.xv, axis=a), np.diff(prob.yv, axis=a)).min() for a in (0, 1)]
    return float(min(e))


def _strict(rok, prob, y):
    return host(rok.rok_residual(rok.rok_init(prob, krylov_max=1, rounding=rok.ROK_ROUND_STRICT), dev(y)))


@pytest.mark.parametrize('name', CASES)
def test_residual_in_and_out_of_the_windows(rok, name):
    prob, y = CASES[name]
    ctx = rok.rok_init(prob, krylov_max=1)
    f = host(rok.rok_residual(ctx, dev(y)))
    fo = core.residual(prob, y)
    # the unlimited MUSCL states of two cases have negative densities: not a
    # number there, in the strict build and in this one alike
    nan = np.isnan(_strict(rok, prob, y))
    assert np.array_equal(np.isnan(f), nan)
    f, fo = f[~nan], fo[~nan]
    # (unphysical cells, where a state has any, give no flux scale)
    phys = (y[0] > 0.0) & (y[3] > 0.5 * (y[1] ** 2 + y[2] ** 2) / y[0])
    y = np.where(phys, y, y[:, phys].mean(axis=1)[:, None, None])
    tol = 64 * U * flux_scale(prob, y)
    if prob.mu > 0.0:   # the viscous flux's own scale: gradients across one cell
        h = min(prob.lx / prob.nx, prob.ly / prob.ny) if prob.xv is None else _width(prob)
        vel = np.abs(y[1:3] / y[0]).max()
        T = ((prob.gamma - 1.0) * y[3] / y[0]).max()
        k = prob.gamma / ((prob.gamma - 1.0) * prob.prandtl)
        g = (T / prob.t_ref) ** 1.5 if prob.sutherland_s > 0.0 else 1.0
        tol += 64 * U * prob.mu * max(g, 1.0) / (h * h) * (vel * vel + vel + k * T)
    err = np.abs(f - fo).max()
    print('\n[fixed] %s: max error %.3e of the bar' % (name, err / tol))
    assert err <= tol, (name, err, tol)


def test_nonfinite_cell_is_reported_and_stays_local(rok):
    prob, y = _flow(48, 40, 0.2, mu=1e-3)
    y = y.copy()
    y[3, 20, 30] = np.nan
    ctx = rok.rok_init(prob, krylov_max=1)
    f = host(rok.rok_residual(ctx, dev(y)))
    fo = _strict(rok, prob, y)   # bit-exact against the oracle on finite states
    assert np.array_equal(np.isnan(f), np.isnan(fo))
    ok = np.isfinite(fo)
    assert np.abs(f[ok] - fo[ok]).max() <= 64 * U * flux_scale(prob, np.nan_to_num(y, nan=2.5))
    with pytest.raises(rok.RokError) as e:
        rok.rok_sync(ctx)
    assert e.value.status == rok.ROK_ERR_NONFINITE


def test_uniform_state_has_zero_residual(rok):
    prob, y = _flow(40, 24, 0.3, amp=0.0, mu=1e-3)
    ctx = rok.rok_init(prob, krylov_max=1)
    assert np.array_equal(host(rok.rok_residual(ctx, dev(y))), np.zeros_like(y))
