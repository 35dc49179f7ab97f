"""CFL wavespeed of states at the ends of the FP64 range, against the formula in
numpy: a speed of sound whose square is subnormal or overflows, a subnormal
density, zero pressure. One such cell among ordinary ones must neither dominate
the maximum nor vanish from it."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

# rho, u, p of one cell in a gas at rest of c = 1.18
CELLS = {"c2 subnormal": (1e10, 0.0, 1e-300), "c2 overflows": (1e-300, 0.0, 1e12), "rho subnormal": (1e-308, 3.0, 1e-308),
         "rho subnormal, fast": (1e-308, 0.0, 1e-300), "no pressure": (2.0, 0.0, 0.0), "rho large": (1e308, 0.0, 1e200),
         "rho large, fast": (1e308, 0.0, 1e307)}


@pytest.mark.parametrize("name", CELLS)
@pytest.mark.parametrize("size", [(24, 18), (270, 240)], ids=["small", "large"])
def test_wavespeed_at_the_ends_of_the_range(name, size):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2305_00762_gb300 import build, gbr
    build.build()
    gbr.load()
    nx, ny = size
    r, u, p = np.ones((ny, nx)), np.zeros((ny, nx)), np.ones((ny, nx))
    r[5, 7], u[5, 7], p[5, 7] = CELLS[name]
    with np.errstate(over="ignore", under="ignore"):
        Q = np.stack([r, r * u, 0 * r, p / 0.4 + 0.5 * r * u * u])
        w = Q[1] / Q[0]
        ref = ((np.abs(w) + np.sqrt(1.4 * (0.4 * (Q[3] - 0.5 * Q[1] * w)) * (1.0 / Q[0]))) / 0.01).max()
    s = gbr.Solver(nx, ny, 0.01, 0.01, 1.4, 0.0, 0.72, (gbr.GBR_BC_PERIODIC,) * 4)
    s.set_state(Q)
    got = s.max_wavespeed()
    s.close()
    assert got == ref or abs(got - ref) <= 1e-12 * ref, (got, ref)
