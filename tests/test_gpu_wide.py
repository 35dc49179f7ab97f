"""Residual beside a jump of many decimal orders, on its low side, against the
scheme in numpy's long double: each component within 1e-12 of the fluxes of the
low side alone (tests/parity.py takes a whole grid's). The MP limiter bounds a
face value by the cells beside the face and the detector takes the faces around
the jump off the flux reconstruction, so FP64 arithmetic is accurate there to its
own scale, whatever lies six cells away. (The oracle adds the limiter's step to
the unlimited value, which the jump dominates, and is not.) One-dimensional
states along x and y, every instance of the FP64 form, sizes of different tile
shapes."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SIZES = [(37, 32), (70, 64), (123, 101), (271, 239)]
FORMS = {"plain": {}, "order4": {"order": 4}, "cons": {"cons": True}, "viscous": {}, "viscous_cons": {"cons": True}}
GAMMA = 1.4


@pytest.fixture(scope="module")
def env():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2305_00762_gb300 import build, gbr
    build.build()
    gbr.load()
    return torch, gbr


def minmod(a, b):
    return np.where((a < 0) != (b < 0), 0, np.where(np.abs(a) < np.abs(b), a, b))


def left_value(w, e, scale, order):
    """Eqs. grb, mp5Condition, mp-procedure of a field carried at `scale` times
    its value, from five values and gradients."""
    d = [w[k] - w[2] for k in range(5)]
    if order == 4:
        delta = e[2] / 2 + (e[1] - e[3]) / 24 + (d[1] + d[3]) / 6
    else:
        delta = (420 * e[2] + 60 * (e[1] - e[3]) + 178 * (d[1] + d[3]) + 3 * (d[0] + d[4])) / 840
    pl = w[2] + delta
    ok = delta * (delta - minmod(d[3], -7 * d[1])) <= (np.longdouble(1e-20) * scale) ** 2
    c = [2 * (w[k + 1] - 2 * w[k] + w[k - 1]) - (e[k + 1] - e[k - 1]) / 2 for k in (1, 2, 3)]
    md = (w[2] + w[3]) / 2 - minmod(c[1], c[2]) / 2
    ul, lc = w[2] - 7 * d[1], (3 * w[2] - w[1]) / 2 + minmod(c[1], c[0]) * 4 / 3
    lo = np.maximum(np.minimum(np.minimum(w[2], w[3]), md), np.minimum(np.minimum(w[2], ul), lc))
    hi = np.minimum(np.maximum(np.maximum(w[2], w[3]), md), np.maximum(np.maximum(w[2], ul), lc))
    return np.where(ok, pl, np.minimum(np.maximum(pl, lo), hi))


def reference(Q, dx, order, cons):
    """Residual of a one-dimensional state [4][n] (un is Q[1] / Q[0]) at cells
    6 .. n - 7."""
    q = np.asarray(Q, dtype=np.longdouble)
    n = q.shape[1]
    g = np.longdouble(1.4)
    r, u, v = q[0], q[1] / q[0], q[2] / q[0]
    p = (g - 1) * (q[3] - (q[1] * u + q[2] * v) / 2)
    j = np.arange(5, n - 6)  # faces j + 1/2

    def mean(a):
        return (a[j] + a[j + 1]) / 2

    c = np.sqrt(g * mean(p) / mean(r))
    rc, ic2, ub, vb = mean(r) * c, 1 / (c * c), mean(u), mean(v)
    var = [a[j + k] for a in (q if cons else (r, u, v, p)) for k in range(-5, 7)]
    var = [var[12 * m:12 * m + 12] for m in range(4)]
    if cons:
        b1 = (g - 1) * ic2
        b2 = b1 * (ub * ub + vb * vb) / 2

        def fields(x):
            A, t = b2 * x[0] - b1 * (ub * x[1] + vb * x[2] - x[3]), (ub * x[0] - x[1]) / c
            return [(A + t) / 2, (A - t) / 2, x[0] - A, x[2] - vb * x[0]]
        scale = [1, 1, 1, 1]
    else:
        def fields(x):
            return [x[3] - rc * x[1], x[3] + rc * x[1], x[0] - ic2 * x[3], x[2]]
        scale = [2 * c * c, 2 * c * c, 1, 1]
    W = [fields([var[m][k] for m in range(4)]) for k in range(12)]
    states = []
    for side in range(2):
        s = []
        for f in range(4):
            w = [W[k][f] for k in range(12)]
            if side:
                w = w[::-1]
            e = [None] * 3 + [(45 * (w[k + 1] - w[k - 1]) - 9 * (w[k + 2] - w[k - 2]) + (w[k + 3] - w[k - 3])) / 60
                              for k in range(3, 9)]
            s.append(left_value(w[3:8], e[3:8], scale[f], order))
        if cons:
            rho = s[0] + s[1] + s[2]
            un, ut = ub + c * (s[1] - s[0]) / rho, vb + s[3] / rho
            pr = c * c * (s[0] + s[1]) - (g - 1) / 2 * ((c * (s[1] - s[0])) ** 2 + s[3] ** 2) / rho
        else:
            pr, un, ut = (s[0] + s[1]) / 2, (s[1] - s[0]) / (2 * rc), s[3]
            rho = s[2] + pr * ic2
        cell = j + side
        bad = (rho <= 0) | (pr <= 0)
        states.append([np.where(bad, a[cell], b) for a, b in zip((r, u, v, p), (rho, un, ut, pr))])

    def flux(s):
        E = s[3] / (g - 1) + s[0] * (s[1] ** 2 + s[2] ** 2) / 2
        return np.array([s[0] * s[1], s[0] * s[1] ** 2 + s[3], s[0] * s[1] * s[2], s[1] * (E + s[3])]), E

    (FL, EL), (FR, ER) = flux(states[0]), flux(states[1])
    (rL, uL, vL, pL), (rR, uR, vR, pR) = states
    a, b = np.sqrt(rL), np.sqrt(rR)

    def roe(x, y):
        return (a * x + b * y) / (a + b)

    ut_, vt_, H = roe(uL, uR), roe(vL, vR), roe((EL + pL) / rL, (ER + pR) / rR)
    ct = np.sqrt((g - 1) * (H - (ut_ ** 2 + vt_ ** 2) / 2))
    SL, SR = np.minimum(uL - np.sqrt(g * pL / rL), ut_ - ct), np.maximum(uR + np.sqrt(g * pR / rR), ut_ + ct)
    mL, mR = rL * (SL - uL), rR * (SR - uR)
    S = (pR - pL + uL * mL - uR * mR) / (mL - mR)

    def star(s, E, Sk, m):
        k = m / (Sk - S)
        return np.array([k, k * S, k * s[2], k * (E / s[0] + (S - s[1]) * (S + s[3] / m))])

    QL, QR = [np.array([s[0], s[0] * s[1], s[0] * s[2], E]) for s, E in ((states[0], EL), (states[1], ER))]
    sL, sR = star(states[0], EL, SL, mL), star(states[1], ER, SR, mR)
    # central part: the states' fluxes where a cell of j-2 .. j+3 is troubled
    eps = np.longdouble(0.45 / 0.55 * 1e-6)
    k = np.arange(2, n - 2)
    ra = np.abs(r[k] - r[k - 1]) + np.abs(r[k] - 2 * r[k - 1] + r[k - 2])
    rb = np.abs(r[k] - r[k + 1]) + np.abs(r[k] - 2 * r[k + 1] + r[k + 2])
    troubled = np.zeros(n, bool)
    troubled[k] = (2 * ra * rb + eps) / (ra * ra + rb * rb + eps) < 0.5
    trouble = np.any([troubled[j + i] for i in range(-2, 4)], axis=0)
    f, _ = flux((r, u, v, p))
    cw, den = ((1821, -461, 85, -4, -1), 2880) if order == 4 else ((1052, -250, 38, 1, -1), 1680)
    Fs = sum(w * (f[:, j - i] + f[:, j + 1 + i]) for i, w in enumerate(cw)) / np.longdouble(den)
    F = np.where(trouble, (FL + FR) / 2, Fs) - (np.abs(SL) * (sL - QL) + np.abs(S) * (sR - sL) + np.abs(SR) * (QR - sR)) / 2
    return -(F[:, 1:] - F[:, :-1]) / dx, np.abs(f)


@pytest.mark.parametrize("axis", ["x", "y"])
@pytest.mark.parametrize("form", FORMS)
@pytest.mark.parametrize("size", SIZES, ids=lambda s: f"{s[0]}x{s[1]}")
@pytest.mark.parametrize("low", [1e-4, 1e-7, 1e-10])
def test_low_side_of_a_jump(env, low, size, form, axis):
    torch, gbr = env
    kw = FORMS[form]
    nx, ny = size
    n = nx if axis == "x" else ny
    at = n // 2
    k = np.arange(n)
    wave = 1e-3 * np.sin(9.0 * (k + 0.5) / n + 1.0)
    f = np.where(k >= at, low, 1.0)
    r, p, u, v = f * (1.0 + wave), f * (0.8 + wave), 0.3 + wave, np.where(k >= at, 0.2 * low, 0.2) * (1.0 + 5.0 * wave)
    Q = np.stack([r, r * u, r * v, p / 0.4 + 0.5 * r * (u * u + v * v)])
    grid = Q[:, None, :].repeat(ny, 1) if axis == "x" else Q[[0, 2, 1, 3]][:, :, None].repeat(nx, 2)
    # A viscosity too small to tell takes the viscous instances (MEG7-cons: its
    # chain rule multiplies the jump's gradient by 1 / rho, to 1e10, and the
    # transverse flux is 1e-22).
    mu = 1e-60 if form.startswith("viscous") else 0.0
    h = 1.0 / n
    s = gbr.Solver(nx, ny, h, h, GAMMA, mu, 0.72, (gbr.GBR_BC_TRANSMISSIVE,) * 4, **kw)
    s.set_state(np.ascontiguousarray(grid))
    R = s.residual()
    s.close()
    R = R[:, ny // 2] if axis == "x" else R[[0, 2, 1, 3]][:, :, nx // 2]
    ref, flux = reference(Q, h, kw.get("order", 7), kw.get("cons", False))
    cells = np.arange(at + 1, at + 9)  # the first one's fluxes are of the low side
    err = np.abs(R[:, cells] - ref[:, cells - 6]).max(1) * h / flux[:, cells].max(1)
    assert (err <= 1e-12).all(), err
