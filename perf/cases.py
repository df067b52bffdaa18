"""Measured workloads of the framework: single entry points and whole ROK4 steps.

Each case is one call a user's program makes: the residual f(y) and its
derivative products (the building blocks of any integrator a user writes
around them), one ROK4 step of a single grid, and one ROK4 step of a batch of
grids.  The flows are those of the repository's benchmark configurations (an
Euler vortex, a low-Mach Taylor-Green vortex, a viscous cylinder on a
stretched O-grid with Sutherland's law), each start state perturbed by a few
seeded smooth modes.  Steps restart from the case's initial state in every
pass, at CFL 1: the arithmetic of a step does not depend on h, and at a small
CFL the finite-difference noise of the Krylov space stays far below the
result's own digits, so two evaluations of the same step can be compared.

``exact`` evaluates the same formulas in plain torch (binary64): ghost cells,
MUSCL, Roe's flux with Harten's fix, the diamond-gradient viscous flux, and
the ROK4 step with modified Gram-Schmidt; derivative products by torch's
automatic differentiation.
"""
import math

import numpy as np
import torch

from paper_1607_06834_gb300 import rok
from paper_1607_06834_gb300 import workloads as W

CFL = 1.0


def listed():
    return [
        # the smallest call a user makes: f(y) on the 64 x 64 Euler vortex
        {'name': 'residual-vortex-64', 'op': 'residual', 'flow': 'vortex', 'nx': 64, 'ny': 64},
        # f(y) at the benchmark's size: explicit integrators, monitoring
        {'name': 'residual-tgv-512', 'op': 'residual', 'flow': 'tgv', 'nx': 512, 'ny': 512},
        # f(y) on the curvilinear O-grid (wall, far field, Sutherland's law)
        {'name': 'residual-cylinder-256x512', 'op': 'residual', 'flow': 'cylinder', 'nx': 512, 'ny': 256},
        # exact JVP on a ragged grid with Sutherland's law: one matvec of a user's own Newton-Krylov solver
        {'name': 'jvp-sutherland-301x203', 'op': 'jvp', 'flow': 'tgv-sutherland', 'nx': 301, 'ny': 203},
        # transposed product J^T u at the gradient workload's size: adjoint and sensitivity analysis
        {'name': 'vjp-tgv-256', 'op': 'vjp', 'flow': 'tgv', 'nx': 256, 'ny': 256},
        # the same on the cylinder O-grid
        {'name': 'vjp-cylinder-256x512', 'op': 'vjp', 'flow': 'cylinder', 'nx': 512, 'ny': 256},
        # one ROK4 step of a small grid, where launches and latencies count
        {'name': 'rok-vortex-64', 'op': 'rok', 'flow': 'vortex', 'nx': 64, 'ny': 64, 'm': 12},
        # the benchmark's ROK4 step
        {'name': 'rok-tgv-512', 'op': 'rok', 'flow': 'tgv', 'nx': 512, 'ny': 512, 'm': 20},
        # the same step with the binary32 Krylov basis
        {'name': 'rok32-tgv-512', 'op': 'rok32', 'flow': 'tgv', 'nx': 512, 'ny': 512, 'm': 20},
        # one ROK4 step of the stiff cylinder, large Krylov dimension
        {'name': 'rok-cylinder-256x512', 'op': 'rok', 'flow': 'cylinder', 'nx': 512, 'ny': 256, 'm': 30},
        # one ROK4 step of a grid four times the benchmark's
        {'name': 'rok-tgv-1024', 'op': 'rok', 'flow': 'tgv', 'nx': 1024, 'ny': 1024, 'm': 20},
        # one ROK4 step of 64 independent grids (sides 32..384, Euler and Navier-Stokes) stepped together
        {'name': 'batch-64', 'op': 'batch', 'flow': 'mixed', 'count': 64, 'n_min': 32, 'n_max': 384, 'm': 16},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(['residual', 'residual', 'jvp', 'vjp', 'rok', 'rok', 'rok32', 'batch'])
    if op == 'batch':
        n_min = _log_int(rng, 24, 128)
        return {'op': op, 'flow': 'mixed', 'count': rng.randint(4, 64), 'n_min': n_min,
                'n_max': min(384, n_min + _log_int(rng, 16, 256)), 'm': rng.randint(6, 16)}
    flow = rng.choice(['vortex', 'tgv', 'tgv', 'tgv-sutherland', 'cylinder'])
    if flow == 'cylinder':
        nx, ny = _log_int(rng, 64, 512), _log_int(rng, 32, 256)
    else:
        # the binary32 basis takes grids up to 2 x 2048 entries per co-resident thread block
        most = 512 if op == 'rok32' else 1024
        nx = _log_int(rng, 48, most)
        ny = min(most, max(48, int(nx * rng.uniform(0.6, 1.6))))
    c = {'op': op, 'flow': flow, 'nx': nx, 'ny': ny}
    if op in ('rok', 'rok32'):
        c['m'] = rng.randint(8, 20)
    return c


# ---- problems and start states -------------------------------------------------------

def _problem(case):
    nx, ny, flow = case['nx'], case['ny'], case['flow']
    if flow == 'cylinder':
        prob, y, _ = W.cylinder_ogrid(ny, nx)
        return prob, y
    if flow == 'vortex':
        prob, _ = W.isentropic_vortex(8)
        prob.nx, prob.ny, prob.ly = nx, ny, prob.lx * ny / nx
        X, Y = W.cell_centres_uniform(nx, ny, prob.lx, prob.ly)
        return prob, W.vortex_state(X, Y, 0.5 * prob.lx, 0.5 * prob.ly, lx=prob.lx, ly=prob.ly)
    prob, _ = W.taylor_green(8)
    prob.nx, prob.ny = nx, ny   # the square box, cells of any aspect ratio
    X, Y = W.cell_centres_uniform(nx, ny, prob.lx, prob.ly)
    p0 = 1.0 / (prob.gamma * 0.01)
    p = p0 + 0.25 * (np.cos(2.0 * X) + np.cos(2.0 * Y))
    u, v = np.sin(X) * np.cos(Y), -np.cos(X) * np.sin(Y)
    y = np.stack([np.ones_like(X), u, v, p / (prob.gamma - 1.0) + 0.5 * (u * u + v * v)])
    if flow == 'tgv-sutherland':
        prob.sutherland_s, prob.t_ref = 110.4 / 278.0, p0
    return prob, y


def _modes(prob, rng):
    """Three smooth seeded modes, periodic over the index box, of size about one."""
    s = 2.0 * np.pi * np.arange(prob.nx) / prob.nx
    t = 2.0 * np.pi * np.arange(prob.ny) / prob.ny
    f = np.zeros((prob.ny, prob.nx))
    for _ in range(3):
        a, b = rng.integers(1, 5, 2)
        ph = rng.uniform(0.0, 2.0 * np.pi, 2)
        f += 0.5 * rng.normal() * np.outer(np.cos(b * t + ph[1]), np.sin(a * s + ph[0]))
    return f


def _perturbed(prob, y, seed):
    rng = np.random.default_rng(seed)
    amp = 1e-2 if prob.curvilinear else 1e-3
    return np.stack([y[k] * (1.0 + amp * _modes(prob, rng)) for k in range(4)])


def _start(case, seed):
    prob, y = _problem(case)
    y = _perturbed(prob, y, seed)
    d = None
    if case['op'] in ('jvp', 'vjp'):
        rng = np.random.default_rng(seed + 1)
        d = torch.from_numpy(rng.standard_normal(y.shape))
    return prob, torch.from_numpy(np.ascontiguousarray(y)), d


def _instances(case, seed):
    inst = W.batched_instances(case['count'], case['n_min'], case['n_max'])
    return [i.problem for i in inst], [_perturbed(i.problem, i.y0, seed + 1000 * k) for k, i in enumerate(inst)]


# ---- what a user's program holds, and one pass ---------------------------------------

def prepare(case, seed):
    op = case['op']
    if op == 'batch':
        probs, states = _instances(case, seed)
        b = rok.rok_batch_init(probs, krylov_max=case['m'])
        y0 = b.pack(states)
        rok.rok_batch_tune(b, y0)
        rok.rok_batch_set_graph(b, True)
        return {'op': op, 'b': b, 'y0': y0, 'y': y0.clone(), 'm': case['m'],
                'h': [_Plain(p, 'cpu').dt(torch.from_numpy(s)) for p, s in zip(probs, states)]}
    prob, y, d = _start(case, seed)
    m = case.get('m', 4)
    ctx = rok.rok_init(prob, krylov_max=m, basis=rok.ROK_BASIS_FP32 if op == 'rok32' else rok.ROK_BASIS_FP64)
    y0 = y.cuda()
    s = {'op': op, 'ctx': ctx, 'y0': y0, 'm': m}
    if d is not None:
        s['d'] = d.cuda()
    if op in ('rok', 'rok32'):
        s['h'] = rok.rok_dt_from_cfl(ctx, y0, CFL)
        s['y'] = y0.clone()
        rok.rok_set_graph(ctx, True)
    else:
        s['out'] = torch.empty_like(y0)
    return s


def run(s):
    op = s['op']
    if op == 'residual':
        return rok.rok_residual(s['ctx'], s['y0'], s['out'])
    if op == 'jvp':
        return rok.rok_jvp(s['ctx'], s['y0'], s['d'], mode=rok.ROK_JVP_EXACT, out=s['out'])
    if op == 'vjp':
        return rok.rok_vjp(s['ctx'], s['y0'], s['d'], out=s['out'])
    s['y'].copy_(s['y0'])
    if op == 'batch':
        rok.rok_batch_step(s['b'], s['y'], s['h'], s['m'])
    else:
        rok.rok_step(s['ctx'], s['y'], s['h'], s['m'])
    return s['y']


def _cells(case):
    if case['op'] == 'batch':
        inst = W.batched_instances(case['count'], case['n_min'], case['n_max'])
        return sum(i.problem.ncells for i in inst)
    return case['nx'] * case['ny']


def work(case):
    """Bytes: inputs and outputs once (the Krylov basis is not counted).  Flops
    per cell and residual: 352 (Euler), 420 (Navier-Stokes, uniform), 480
    (curvilinear with Sutherland's law), counting + - x / sqrt one each and
    every face once; a derivative product about three residuals; a ROK4 step
    m + 4 residuals, the Gram-Schmidt of m columns, and four projections and
    stage vectors."""
    cells = _cells(case)
    n = 4 * cells
    f = {'vortex': 352, 'tgv': 420, 'tgv-sutherland': 450, 'cylinder': 480, 'mixed': 386}[case['flow']] * cells
    op = case['op']
    if op == 'residual':
        return {'bytes': 16 * n, 'flops': f}
    if op in ('jvp', 'vjp'):
        return {'bytes': 24 * n, 'flops': 3 * f}
    m = case['m']
    return {'bytes': 16 * n, 'flops': (m + 4) * f + n * (2 * m * (m + 1) + 3 * m + 16 * m + 8)}


# ---- the same in plain torch ----------------------------------------------------------

def _ghosts(prob, w, inf):
    """Two ghost layers around the primitives w (k, ny, nx): j sides first, then
    i sides; walls mirror (rho, -u, -v, p, T), far fields are the free stream."""
    sign = torch.ones(w.shape[0], 1, 1, dtype=w.dtype, device=w.device)
    sign[1:3] = -1.0

    def side(bc, edge, wrap, dim):
        if bc == W.PERIODIC:
            return wrap
        if bc == W.WALL:
            return sign * edge.flip(dim)
        return inf.expand_as(edge)

    w = torch.cat([side(prob.bc[2], w[:, :2], w[:, -2:], 1), w, side(prob.bc[3], w[:, -2:], w[:, :2], 1)], 1)
    return torch.cat([side(prob.bc[0], w[:, :, :2], w[:, :, -2:], 2), w,
                      side(prob.bc[1], w[:, :, -2:], w[:, :, :2], 2)], 2)


def _metrics(prob, device):
    """Unit normals, face lengths, diamond coefficients of the i- and j-faces, 1 / volume."""
    if not prob.curvilinear:
        dx, dy = prob.lx / prob.nx, prob.ly / prob.ny
        return ((1.0, 0.0, dy, (1.0 / dx, 0.0, 0.0, 1.0 / dy)),
                (0.0, 1.0, dx, (0.0, -1.0 / dx, 1.0 / dy, 0.0)), 1.0 / (dx * dy))
    z = torch.from_numpy(prob.xv + 1j * prob.yv).to(device)   # vertices as x + i y
    per = z[:, -1:] - z[:, :1]
    z = torch.cat([z[:, -2:-1] - per, z, z[:, 1:2] + per], 1)   # i periodic
    ze = torch.cat([2.0 * z[:1] - z[1:2], z, 2.0 * z[-1:] - z[-2:-1]], 0)   # j extrapolated
    c = 0.25 * (ze[:-1, :-1] + ze[:-1, 1:] + ze[1:, 1:] + ze[1:, :-1])   # cell centres, one ghost layer
    z = z[:, 1:-1]

    def cross(a, b):
        return a.real * b.imag - a.imag * b.real

    def face(e, normal, p0, p1, p2, p3):
        n = normal * e / e.abs()
        d1, d2 = p2 - p0, p3 - p1
        r = 1.0 / cross(d1, d2)
        return n.real, n.imag, e.abs(), (d2.imag * r, -d1.imag * r, -d2.real * r, d1.real * r)

    fi = face(z[1:] - z[:-1], -1j, c[1:-1, :-1], z[:-1], c[1:-1, 1:], z[1:])
    fj = face(z[:, 1:] - z[:, :-1], 1j, c[:-1, 1:-1], z[:, 1:], c[1:, 1:-1], z[:, :-1])
    area = 0.5 * cross(z[1:, 1:] - z[:-1, :-1], z[1:, :-1] - z[:-1, 1:])
    return fi, fj, 1.0 / area


def _abs(x):
    return torch.where(x < 0.0, -x, x)   # with the derivative +1 at 0


def _face_flux(prob, m2, m1, p1, p2, dV, geo):
    """Flux times face length between cells m1 and p1 (their outer neighbours m2,
    p2; dV the vertex differences of u, v, T along the face)."""
    nx, ny, length, (c0, c1, c2, c3) = geo
    g, gm1 = prob.gamma, prob.gamma - 1.0
    lo, hi = 0.25 * (1.0 - prob.muscl_kappa), 0.25 * (1.0 + prob.muscl_kappa)
    dc = p1 - m1
    rL, uL, vL, pL = (m1 + lo * (m1 - m2) + hi * dc)[:4]
    rR, uR, vR, pR = (p1 - lo * (p2 - p1) - hi * dc)[:4]
    qL, qR = uL * nx + vL * ny, uR * nx + vR * ny
    HL = g / gm1 * pL / rL + 0.5 * (uL * uL + vL * vL)
    HR = g / gm1 * pR / rR + 0.5 * (uR * uR + vR * vR)
    sL, sR = rL.sqrt(), rR.sqrt()
    wl = sL / (sL + sR)
    wr = 1.0 - wl
    rt, u, v, H = sL * sR, wl * uL + wr * uR, wl * vL + wr * vR, wl * HL + wr * HR
    k = 0.5 * (u * u + v * v)
    c_sq = gm1 * (H - k)
    c, q = c_sq.sqrt(), u * nx + v * ny
    dr, du, dv, dp, dq = rR - rL, uR - uL, vR - vL, pR - pL, qR - qL
    delta = prob.entropy_fix * (_abs(q) + c)

    def harten(x):
        a = _abs(x)
        return torch.where(a < delta, (a * a + delta * delta) / (2.0 * delta), a)

    w1 = harten(q - c) * (dp - rt * c * dq) / (2.0 * c_sq)
    w2 = _abs(q) * (dr - dp / c_sq)
    w3 = harten(q + c) * (dp + rt * c * dq) / (2.0 * c_sq)
    ws = _abs(q) * rt
    D = (w1 + w2 + w3,
         w1 * (u - c * nx) + w2 * u + w3 * (u + c * nx) + ws * (du - dq * nx),
         w1 * (v - c * ny) + w2 * v + w3 * (v + c * ny) + ws * (dv - dq * ny),
         w1 * (H - c * q) + w2 * k + w3 * (H + c * q) + ws * (u * du + v * dv - q * dq))
    A = (rL * qL + rR * qR, rL * qL * uL + rR * qR * uR + (pL + pR) * nx,
         rL * qL * vL + rR * qR * vR + (pL + pR) * ny, rL * qL * HL + rR * qR * HR)
    F = torch.stack([0.5 * (a - d) for a, d in zip(A, D)])
    if prob.kind == W.NAVIER_STOKES:
        mean = 0.5 * (m1 + p1)
        (ux, uy), (vx, vy), (Tx, Ty) = [(dc[i] * c0 + dV[n] * c1, dc[i] * c2 + dV[n] * c3)
                                        for n, i in enumerate((1, 2, 4))]
        mu, div = mean[5], ux + vy
        txx, tyy, txy = mu * (2.0 * ux - 2.0 / 3.0 * div), mu * (2.0 * vy - 2.0 / 3.0 * div), mu * (uy + vx)
        tx, ty = txx * nx + txy * ny, txy * nx + tyy * ny
        heat = mu * g / (gm1 * prob.prandtl) * (Tx * nx + Ty * ny)
        F = F - torch.stack([torch.zeros_like(tx), tx, ty, mean[1] * tx + mean[2] * ty + heat])
    return F * length


def _prims(prob, q):
    rho, u, v = q[0], q[1] / q[0], q[2] / q[0]
    p = (prob.gamma - 1.0) * (q[3] - 0.5 * (q[1] * u + q[2] * v))
    T = p / rho
    t, s = T / prob.t_ref, prob.sutherland_s
    mu = prob.mu * t * t.sqrt() * (1.0 + s) / (t + s) if s > 0.0 else torch.full_like(T, prob.mu)
    return torch.stack([rho, u, v, p, T, mu])


class _Plain:
    """f(y) of one problem in plain torch (differentiable)."""

    def __init__(self, prob, device):
        self.prob = prob
        self.fi, self.fj, self.inv_vol = _metrics(prob, device)
        self.inf = _prims(prob, torch.tensor(prob.q_inf, dtype=torch.float64, device=device)[:, None, None])

    def f(self, y):
        w = _ghosts(self.prob, _prims(self.prob, y), self.inf)
        t = w[[1, 2, 4], 1:-1, 1:-1]   # u, v, T with one ghost layer
        vert = 0.25 * (t[:, :-1, :-1] + t[:, :-1, 1:] + t[:, 1:, :-1] + t[:, 1:, 1:])
        r, c = w[:, 2:-2], w[:, :, 2:-2]
        Fi = _face_flux(self.prob, r[:, :, :-3], r[:, :, 1:-2], r[:, :, 2:-1], r[:, :, 3:], vert[:, 1:] - vert[:, :-1],
                        self.fi)
        Fj = _face_flux(self.prob, c[:, :-3], c[:, 1:-2], c[:, 2:-1], c[:, 3:], vert[:, :, :-1] - vert[:, :, 1:],
                        self.fj)
        return -((Fi[:, :, 1:] - Fi[:, :, :-1]) + (Fj[:, 1:] - Fj[:, :-1])) * self.inv_vol

    def dt(self, y):
        """CFL time step: acoustic rates and viscous bound of every cell."""
        prob = self.prob
        rho, u, v, p, _, mu = _prims(prob, y)
        c = (prob.gamma * p / rho).sqrt()
        rate, s2 = 0.0, 0.0
        for face, dim in ((self.fi, 1), (self.fj, 0)):
            sx, sy = face[0] * face[2], face[1] * face[2]
            if prob.curvilinear:   # mean of the cell's two faces
                n = sx.shape[dim] - 1
                sx, sy = (0.5 * (s.narrow(dim, 0, n) + s.narrow(dim, 1, n)) for s in (sx, sy))
            sq = sx * sx + sy * sy
            rate = rate + ((u * sx + v * sy).abs() + c * sq ** 0.5) * self.inv_vol
            s2 = s2 + sq
        if prob.kind == W.NAVIER_STOKES:
            nu = max(4.0 / 3.0, prob.gamma / prob.prandtl) * mu / rho
            rate = rate + 2.0 * nu * s2 * self.inv_vol ** 2
        return CFL / float(rate.max())


def _plain_rok(f, y, h, M):
    """One ROK4 step (four stages, classical RK4 alpha and b) with one-sided
    difference quotients and modified Gram-Schmidt."""
    gamma = 0.5728160624821349
    goff = [[0.0] * 4, [0.025068629909359066, 0.0, 0.0, 0.0], [0.2477474325727758, -1.405913872491725, 0.0, 0.0],
            [0.6, -0.020369905583413464, -1.7503308492902152, 0.0]]
    eps = math.sqrt(2.0 ** -52 * (1.0 + float(y.norm())))
    eps = 2.0 ** math.floor(math.log2(eps) + 0.5)
    F = f(y)
    V = torch.zeros(M, y.numel(), dtype=y.dtype, device=y.device)
    H = torch.zeros(M, M, dtype=y.dtype, device=y.device)
    V[0] = (F / F.norm()).ravel()
    for j in range(M):
        w = ((f(y + eps * V[j].view_as(y)) - F) / eps).ravel()
        for i in range(j + 1):
            H[i, j] = V[i] @ w
            w = w - H[i, j] * V[i]
        if j + 1 < M:
            H[j + 1, j] = w.norm()
            V[j + 1] = w / H[j + 1, j]
    A = torch.eye(M, dtype=y.dtype, device=y.device) - h * gamma * H
    ks, lam = [], []
    for i in range(4):
        if i:
            F = f(y + (0.5 if i < 3 else 1.0) * ks[-1])
        phi = V @ F.ravel()
        acc = sum((goff[i][j] * lam[j] for j in range(i)), torch.zeros_like(phi))
        lam.append(torch.linalg.solve(A, h * phi + h * (H @ acc)))
        ks.append(((lam[i] - h * phi) @ V).view_as(y) + h * F)
    return y + (ks[0] + 2.0 * ks[1] + 2.0 * ks[2] + ks[3]) / 6.0


def exact(case, seed):
    device = 'cuda' if torch.cuda.is_available() else 'cpu'
    op = case['op']
    if op == 'batch':
        probs, states = _instances(case, seed)
        parts = []
        for prob, y in zip(probs, states):
            P, y = _Plain(prob, device), torch.from_numpy(y)
            h = P.dt(y)
            parts.append(_plain_rok(P.f, y.to(device), h, case['m']).ravel())
            parts.append(torch.zeros(-parts[-1].numel() % 2048, dtype=y.dtype, device=device))   # padding
        return torch.cat(parts)
    prob, y, d = _start(case, seed)
    P, y = _Plain(prob, device), y.to(device)
    if op == 'residual':
        return P.f(y)
    if op == 'jvp':
        return torch.func.jvp(P.f, (y,), (d.to(device),))[1]
    if op == 'vjp':
        y.requires_grad_(True)
        return torch.autograd.grad(P.f(y), y, d.to(device))[0]
    return _plain_rok(P.f, y, P.dt(y), case['m'])
