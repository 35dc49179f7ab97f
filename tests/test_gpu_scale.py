"""Residuals of flows in other units of mass (densities and pressures of 1e-6 to
1e-28) against the oracle: the MP test's threshold (Eq. mp5Condition, 1e-40) is
an absolute number, so a value is limited at one scale and not at another."""
import numpy as np
import pytest

from paper_2305_00762_gb300 import cases as C

from .parity import assert_residual_close, tie_faces_ok

pytestmark = pytest.mark.gpu

FORMS = {"plain": {}, "order4": {"order": 4}, "cons": {"cons": True}}


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


@pytest.mark.parametrize("form", FORMS)
@pytest.mark.parametrize("scale", [1e-6, 1e-12, 1e-20, 1e-28])
@pytest.mark.parametrize("size", [(61, 40), (123, 101), (271, 239)], ids=lambda s: f"{s[0]}x{s[1]}")
def test_residual_in_other_units(env, size, scale, form):
    torch, O, gbr = env
    nx, ny = size
    c, kw = C.riemann_2d(nx, ny, split=(0.55, 0.4)), FORMS[form]
    cfg = O.Config(nx, ny, c.dx, c.dy, c.gamma, c.mu, c.Pr, c.bc, order=kw.get("order", 7), cons=int(kw.get("cons", False)))
    Q = c.Q
    for _ in range(2):  # off the piecewise-constant data
        Q, rc = O.rk3_step(cfg, Q, 0.2 / O.max_wavespeed(cfg, Q))
        assert rc == 0
    Q = Q * scale
    s = gbr.Solver.for_case(c, **kw)
    s.record_flags(True)
    s.set_state(Q)
    R = s.residual()
    sx, sy = s.flags()
    s.close()
    Ro, sxo, syo = O.residual(cfg, Q, want_flags=True)
    excl = tie_faces_ok(O, cfg, Q, sx, sxo, sy, syo)
    assert_residual_close(R, Ro, Q, c, exclude=excl, what=f"{size} {form} at {scale:g}")
