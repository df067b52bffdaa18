"""f(y) on a uniform periodic grid in the widest floating-point type NumPy has
(64 significand bits or more): what rounding errors of the binary64 builds are
measured against.  Plain formulas, cell by cell as arrays (Sec. 3.2: MUSCL, Roe's
flux with Harten's fix, central viscous terms)."""
import numpy as np

from paper_1607_06834_gb300 import workloads as W

L = np.longdouble


def _flux(prob, m2, m1, p1, p2, along, n, h, ht):
    """Flux between cells m1 and p1 (outer neighbours m2, p2) with the normal along
    velocity component n; along: four-cell differences of (u, v) along the face."""
    g = L(prob.gamma)
    gm1 = L(np.float64(prob.gamma) - 1.0)
    lo, hi = L(0.25 * (1.0 - prob.muscl_kappa)), L(0.25 * (1.0 + prob.muscl_kappa))
    t = 3 - n
    dc = p1 - m1
    wl, wr = m1 + lo * (m1 - m2) + hi * dc, p1 - lo * (p2 - p1) - hi * dc
    rL, nL, tL, pL = wl[0], wl[n], wl[t], wl[3]
    rR, nR, tR, pR = wr[0], wr[n], wr[t], wr[3]
    inv = 1 / gm1
    HL, HR = (inv + 1) * pL / rL + (nL * nL + tL * tL) / 2, (inv + 1) * pR / rR + (nR * nR + tR * tR) / 2
    sL, sR = np.sqrt(rL), np.sqrt(rR)
    a = sL / (sL + sR)
    b = sR / (sL + sR)
    rt, un, ut, H = sL * sR, a * nL + b * nR, a * tL + b * tR, a * HL + b * HR
    k = (un * un + ut * ut) / 2
    c2 = gm1 * (H - k)
    c = np.sqrt(c2)
    dr, dn, dt, dp = rR - rL, nR - nL, tR - tL, pR - pL
    delta = L(prob.entropy_fix) * (abs(un) + c)

    def harten(x):
        with np.errstate(divide='ignore', invalid='ignore'):
            return np.where(abs(x) < delta, (x * x + delta * delta) / (2 * delta), abs(x))

    w1 = harten(un - c) * (dp - rt * c * dn) / (2 * c2)
    w2 = abs(un) * (dr - dp / c2)
    w3 = harten(un + c) * (dp + rt * c * dn) / (2 * c2)
    ws = abs(un) * rt * dt
    F = np.zeros_like(m1[:4])
    F[0] = (rL * nL + rR * nR - (w1 + w2 + w3)) / 2
    F[n] = (rL * nL * nL + pL + rR * nR * nR + pR - (w1 * (un - c) + w2 * un + w3 * (un + c))) / 2
    F[t] = (rL * nL * tL + rR * nR * tR - ((w1 + w2 + w3) * ut + ws)) / 2
    F[3] = (rL * nL * HL + rR * nR * HR - (w1 * (H - c * un) + w2 * k + w3 * (H + c * un) + ws * ut)) / 2
    if prob.kind == W.NAVIER_STOKES:
        mean = (m1 + p1) / 2
        gn, gt, gT = dc[n] / h, dc[t] / h, dc[4] / h          # along the normal
        an, at = along[n - 1] / (4 * ht), along[t - 1] / (4 * ht)
        mu = mean[5]
        tnn = mu * (2 * gn - 2 * (gn + at) / 3)
        tnt = mu * (an + gt)
        F[n] -= tnn
        F[t] -= tnt
        F[3] -= mean[n] * tnn + mean[t] * tnt + mu * g / (gm1 * L(prob.prandtl)) * gT
    return F


def residual(prob, y):
    """f(y) in long double; y as binary64 (4, ny, nx)."""
    assert prob.xv is None or prob.name == 'aligned'
    q = np.asarray(y).astype(L)
    gm1 = L(np.float64(prob.gamma) - 1.0)
    rho, u, v = q[0], q[1] / q[0], q[2] / q[0]
    p = gm1 * (q[3] - (q[1] * u + q[2] * v) / 2)
    T = p / rho
    if prob.sutherland_s > 0.0:
        t, s = T / L(prob.t_ref), L(prob.sutherland_s)
        mu = L(prob.mu) * t * np.sqrt(t) * (1 + s) / (t + s)
    else:
        mu = np.full_like(T, L(prob.mu))
    w = np.stack([rho, u, v, p, T, mu])
    dx, dy = L(prob.lx) / prob.nx, L(prob.ly) / prob.ny

    def sh(a, k, axis):   # a[i + k]
        return np.roll(a, -k, axis=axis)

    uv = w[1:3]
    f = 0
    for n, axis, other, h, ht in ((1, 2, 1, dx, dy), (2, 1, 2, dy, dx)):
        m2, m1, p2 = sh(w, -2, axis), sh(w, -1, axis), sh(w, 1, axis)
        pair = uv + sh(uv, -1, axis)
        F = _flux(prob, m2, m1, w, p2, sh(pair, 1, other) - sh(pair, -1, other), n, h, ht)   # lower faces
        f = f - (sh(F, 1, axis) - F) / h
    return f
