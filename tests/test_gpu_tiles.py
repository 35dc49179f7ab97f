"""The FP64 form's tile shapes (8 x 4, 16 x 8, 16 x 15, chosen by the grid):
residual and flags against the oracle at sizes that take each of them with
ragged last tiles, for every instance (plain, fourth order, viscous,
MEG7-cons) -- the parity tolerance of tests/parity.py, 1e-12 -- and a grid cut
out of a larger one, whose interior cells must not depend on the shape."""
import numpy as np
import pytest

from paper_2305_00762_gb300 import cases as C

from .parity import assert_residual_close, tie_faces_ok

pytestmark = pytest.mark.gpu

SIZES = {"8x4": (37, 21), "16x8": (190, 117), "16x15": (271, 239)}
FORMS = {"plain": {}, "order4": {"order": 4}, "cons": {"cons": True}, "viscous": {}, "viscous_cons": {"cons": True}}


@pytest.fixture(scope="module")
def env():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import oracle as O
    from paper_2305_00762_gb300 import build, gbr
    build.build()
    O.build()
    gbr.load()
    return torch, O, gbr


def make(form, nx, ny):
    if form.startswith("viscous"):
        return C.viscous_shock_tube(nx, ny)
    return C.riemann_2d(nx, ny, split=(0.55, 0.4))


@pytest.mark.parametrize("form", FORMS)
@pytest.mark.parametrize("size", SIZES)
def test_residual_of_every_shape(env, size, form):
    torch, O, gbr = env
    nx, ny = SIZES[size]
    c, kw = make(form, nx, ny), FORMS[form]
    cfg = O.Config(nx, ny, c.dx, c.dy, c.gamma, c.mu, c.Pr, c.bc, order=kw.get("order", 7), cons=int(kw.get("cons", False)))
    Q = c.Q
    for _ in range(2):  # off the piecewise-constant data
        Q, rc = O.rk3_step(cfg, Q, 0.2 / O.max_wavespeed(cfg, Q))
        assert rc == 0
    s = gbr.Solver.for_case(c, **kw)
    s.record_flags(True)
    s.set_state(Q)
    R = s.residual()
    sx, sy = s.flags()
    Ro, sxo, syo = O.residual(cfg, Q, want_flags=True)
    excl = tie_faces_ok(O, cfg, Q, sx, sxo, sy, syo)
    assert_residual_close(R, Ro, Q, c, exclude=excl, what=f"{size} {form}")
    s.close()


@pytest.mark.parametrize("form", ["plain", "cons"])
def test_residual_does_not_depend_on_the_shape(env, form):
    torch, O, gbr = env
    c = make(form, 271, 239)
    out = {}
    for nx, ny in SIZES.values():
        s = gbr.Solver(nx, ny, c.dx, c.dy, c.gamma, c.mu, c.Pr, c.bc, **FORMS[form])
        s.set_state(np.ascontiguousarray(c.Q[:, :ny, :nx]))
        out[nx] = s.residual()[:, :21 - 6, :37 - 6]  # cells whose stencils end inside the smallest grid
        s.close()
    ref = out[271]
    for R in out.values():
        assert np.array_equal(R, ref)


@pytest.mark.parametrize("form", FORMS)
@pytest.mark.parametrize("size", ["8x4", "16x8"])
def test_no_flux_from_a_state_without_sound(env, size, form):
    """A fast cell of negative pressure: the mean pressure with a neighbour is
    negative too, so each of its faces falls back to the cells' own states; the
    Roe average has a speed of sound (the velocities differ), the cell has none.
    Such a face has no flux: NaN in every component, not the finite remainder of
    a minimum that drops a NaN. The step reports the state."""
    torch, O, gbr = env
    nx, ny = SIZES[size]
    c = make(form, nx, ny)
    Q = c.Q.copy()
    r, p = Q[0], 0.4 * (Q[3] - 0.5 * (Q[1] ** 2 + Q[2] ** 2) / Q[0])
    u, v = Q[1, 10, 18] / r[10, 18] + 50.0, Q[2, 10, 18] / r[10, 18] + 50.0
    Q[1:, 10, 18] = r[10, 18] * u, r[10, 18] * v, 0.5 * r[10, 18] * (u * u + v * v) - 5.0 * p[9:12, 17:20].max()
    s = gbr.Solver.for_case(c, **FORMS[form])
    s.set_state(Q)
    R = s.residual()
    for j, i in ((10, 18), (9, 18), (11, 18), (10, 17), (10, 19)):
        assert np.isnan(R[:, j, i]).all(), (j, i)
    s.step(1e-9)
    assert s.sync(allow=(gbr.GBR_ERR_NONPHYSICAL,)) == gbr.GBR_ERR_NONPHYSICAL
    s.close()
