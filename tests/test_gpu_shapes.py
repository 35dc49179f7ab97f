"""Every tile shape of the FP64 form, at sizes that the rule gives it on this
device: residual and flags against the oracle for each instance, the same bits
from each shape, halo rows and custom sides in the tiles that read filled ghost
cells, and ghost cells read through the boundary rules (8 x 4) against filled
ones."""
import dataclasses

import numpy as np
import pytest

from paper_2305_00762_gb300 import cases as C

from .parity import assert_residual_close, assert_state_close, tie_faces_ok
from .tile_rule import shape

pytestmark = pytest.mark.gpu

SHAPES = ["8x4", "16x8", "16x15"]
FORMS = {"plain": {}, "order4": {"order": 4}, "cons": {"cons": True}, "viscous": {}, "viscous_cons": {"cons": True}}
# ragged grids, the first that takes the shape
GRIDS = [(37, 21), (123, 101), (119, 133), (271, 239), (331, 303), (451, 417), (561, 537), (1021, 1013)]


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


def sms(torch):
    return torch.cuda.get_device_properties(0).multi_processor_count


def takes(torch, nx, ny, form="plain"):
    return shape(nx, ny, sms(torch), "cons" in form, form.startswith("viscous"))


def grid_of(torch, want, form="plain"):
    return next(g for g in GRIDS if takes(torch, *g, form) == want)


def make(form, nx, ny):
    if form.startswith("viscous"):
        return C.viscous_shock_tube(nx, ny)
    return C.riemann_2d(nx, ny, split=(0.55, 0.4))


@pytest.mark.parametrize("form", FORMS)
@pytest.mark.parametrize("want", SHAPES)
def test_residual_of_every_shape(env, want, form):
    torch, O, gbr = env
    nx, ny = grid_of(torch, want, form)
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
    assert_residual_close(R, Ro, Q, c, exclude=excl, what=f"{want} {form} {nx}x{ny}")
    s.timing(True)
    s.step(1e-6)
    ghosts = s.get_timing()[0]["ghost"][1]
    assert ghosts == (0 if want == "8x4" else 3)  # (the rule of the library is the one asked here)
    s.close()


@pytest.mark.parametrize("form", FORMS)
def test_the_same_bits_from_every_shape(env, form):
    torch, O, gbr = env
    grids = [grid_of(torch, w, form) for w in SHAPES]
    big = grids[-1]
    c = make(form, *big)
    out = []
    for nx, ny in grids:
        s = gbr.Solver(nx, ny, c.dx, c.dy, c.gamma, c.mu, c.Pr, c.bc, **FORMS[form])
        s.set_state(np.ascontiguousarray(c.Q[:, :ny, :nx]))
        out.append(s.residual()[:, :15, :31])  # cells whose stencils end inside the smallest grid
        s.close()
    assert np.array_equal(out[0], out[2]) and np.array_equal(out[1], out[2])


SLABS = [("riemann", lambda: C.riemann_2d(123, 101), 4), ("kh", lambda: C.kelvin_helmholtz(123, np.random.default_rng(3), ny=101), 4),
         ("wall", lambda: C.viscous_shock_tube(123, 101), 4), ("riemann", lambda: C.riemann_2d(450, 470), 2)]


@pytest.mark.parametrize("name,make_case,n", SLABS, ids=[f"{a}-{c}" for a, _, c in SLABS])
def test_halo_rows_read_and_filled(env, name, make_case, n):
    """A grid in tiles with filled ghost cells, cut into slabs that read theirs
    through the boundary rules (halo rows and their corners from memory), and one
    whose slabs fill them too: the single grid bit for bit, which the oracle
    checks."""
    torch, O, gbr = env
    from paper_2305_00762_gb300 import slab as S
    c = make_case()
    form = "viscous" if c.mu > 0 else "plain"
    assert takes(torch, c.nx, c.ny, form) != "8x4"
    assert (takes(torch, c.nx, (c.ny + n - 1) // n, form) == "8x4") == (n == 4)
    single = gbr.Solver.for_case(c)
    single.set_state(c.Q)
    slabs = S.LocalSlabs(c, n)
    slabs.set_state(c.Q)
    cfg = O.Config(c.nx, c.ny, c.dx, c.dy, c.gamma, c.mu, c.Pr, c.bc)
    Q = c.Q
    for _ in range(3):
        dt = 0.3 / single.max_wavespeed()
        single.step(dt)
        slabs.step(dt)
        Q, rc = O.rk3_step(cfg, Q, dt)
        assert rc == 0
    single.step_cfl(0.4)
    slabs.step_cfl(0.4)
    assert np.array_equal(slabs.get_state(), single.get_state()) and slabs.time() == single.time()
    slabs.close()
    single.set_state(c.Q)
    for _ in range(3):
        single.step(0.3 / single.max_wavespeed())
    assert_state_close(single.get_state(), Q, tol=1e-11, what=name)
    single.close()


@pytest.mark.parametrize("bc", [(0, 0, 0, 0), (1, 1, 1, 1), (2, 2, 2, 2), (3, 3, 3, 3), (1, 2, 3, 1), (2, 3, 0, 0)])
@pytest.mark.parametrize("mu", [0.0, 1e-3])
def test_ghost_cells_read_and_filled(env, bc, mu):
    """The 8 x 4 tile on one grid with ghost cells read through the rules (a
    solver's step) and filled before each stage (the static step)."""
    torch, O, gbr = env
    nx, ny = 37, 21
    assert takes(torch, nx, ny, "viscous" if mu else "plain") == "8x4"
    c = dataclasses.replace(C.riemann_2d(nx, ny, split=(0.5, 0.45)), mu=mu, bc=bc)
    s = gbr.Solver.for_case(c)
    s.set_state(c.Q)
    q = torch.from_numpy(c.Q).cuda()
    for _ in range(3):
        dt = 0.3 / s.max_wavespeed()
        s.step(dt)
        gbr.gbr_step_static(q, q, nx, ny, c.gamma, c.mu, c.Pr, bc, c.dx, c.dy, dt)
        torch.cuda.synchronize()
    assert np.array_equal(s.get_state(), q.cpu().numpy())
    s.close()


def test_custom_sides_read_and_filled(env):
    """Custom sides (fixed states, a kind that changes at a point, a moving one):
    a small grid, whose tiles read ghost cells through the rules, against the same
    cells of a longer one, whose tiles find them filled."""
    torch, O, gbr = env
    out = {}
    for nx in (70, 1400):
        c = C.double_mach(70, 19)
        dx, dy = c.dx, c.dy
        x = (np.arange(nx) + 0.5) * dx
        Q = np.empty((4, 19, nx))
        Q[:, :, :70] = c.Q
        Q[:, :, 70:] = c.Q[:, :, -1:]
        Q[0] *= 1.0 + 0.02 * np.sin(5.0 * x)
        s = gbr.Solver(nx, 19, dx, dy, c.gamma, 0.0, 0.72, c.bc)
        for k, side in enumerate(c.meta["sides"]):
            if side is not None:
                s.set_side(k, *side)
        s.set_state(Q)
        s.set_time(0.03)
        R = s.residual()
        s.timing(True)
        s.step(1e-4)
        assert s.get_timing()[0]["ghost"][1] == (0 if nx == 70 else 3)
        # (a residual reaches 6 cells, a step 18)
        out[nx] = (R[:, :, :64], s.get_state()[:, :, :52], s.time())
        s.close()
    for a, b in zip(out[70], out[1400]):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("cons,riemann", [(0, 0), (1, 0), (0, 1)])
def test_custom_sides_in_a_large_grid(env, cons, riemann):
    """The double Mach reflection in tiles with filled ghost cells against the
    oracle, step by step with the moving side."""
    torch, O, gbr = env
    nx, ny = 300, 75
    form = "cons" if cons else "plain"
    assert takes(torch, nx, ny, form) != "8x4"
    c = C.double_mach(nx, ny)
    cfg = O.Config(nx, ny, c.dx, c.dy, c.gamma, c.mu, c.Pr, c.bc, 7, cons, t=0.0, sides=c.meta["sides"], riemann=riemann)
    s = gbr.Solver.for_case(c, cons=bool(cons), riemann=riemann)
    s.set_state(c.Q)
    Q, t = c.Q.copy(), 0.0
    for _ in range(5):
        dt = 0.5 / O.max_wavespeed(cfg, Q)
        s.step(dt)
        Q, rc = O.rk3_step(dataclasses.replace(cfg, t=t), Q, dt)
        assert rc == 0
        t += dt
    assert_state_close(s.get_state(), Q, tol=1e-11, what=f"double Mach {nx}x{ny}")
    s.close()
