"""Grids with more rows of tiles than one launch's y extent (65535) holds, in
the smallest FP64 tile and the largest: a flow of period 90 rows repeated along
y takes the same steps, bit for bit, as one period with periodic sides (the
result does not depend on the tile shape), with the scalars of a step (its time)
kept once."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

# columns and periods: 8 x 4 tiles above 4 * 65535 rows, 16 x 15 ones above 15 * 65535
GRIDS = [(6, 3000), (12, 11000)]


@pytest.mark.parametrize("nx,periods", GRIDS, ids=[f"{a}x{90 * b}" for a, b in GRIDS])
def test_rows_of_tiles_beyond_one_launch(nx, periods):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2305_00762_gb300 import build, gbr
    build.build()
    gbr.load()
    y, x = np.meshgrid((np.arange(90) + 0.5) / 90, (np.arange(nx) + 0.5) / nx, indexing="ij")
    r = 1.0 + 0.2 * np.sin(2 * np.pi * y) + 0.1 * np.cos(2 * np.pi * x)
    u, v, p = 0.3 * np.cos(2 * np.pi * (x + y)), 0.4 + 0.2 * np.sin(4 * np.pi * y), 1.0 + 0.1 * np.sin(2 * np.pi * (y - x))
    Q = np.stack([r, r * u, r * v, p / 0.4 + 0.5 * r * (u * u + v * v)])
    out = []
    for n in (1, periods):
        s = gbr.Solver(nx, 90 * n, 0.01, 0.01, 1.4, 0.0, 0.72, (gbr.GBR_BC_PERIODIC,) * 4)
        s.set_state(torch.from_numpy(Q).cuda().repeat(1, n, 1))
        for _ in range(3):
            s.step_cfl(0.4)
        s.step(1e-3)
        q = torch.empty(4, 90 * n, nx, dtype=torch.float64, device="cuda")
        s.get_state(q)
        s.sync()
        out.append((q, s.time()))
        s.close()
    assert out[0][1] == out[1][1]
    assert torch.equal(out[1][0].reshape(4, periods, 90, nx), out[0][0][:, None].expand(-1, periods, -1, -1))
