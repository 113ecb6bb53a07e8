"""The allocation-free overflow through every way of its scatter (dense to
spread, cells of many bins) and on grids of very few bins."""
import numpy as np
import pytest

from oracle import density as odens
from paper_2402_18311_gb300 import place

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny", [(1, 1), (2, 40), (7, 3), (128, 96)])
@pytest.mark.parametrize("sigma", [1e-3, 0.03, 0.3])
def test_noalloc_matches_oracle(nx, ny, sigma):
    torch = pytest.importorskip("torch")
    rng = np.random.default_rng(nx + ny)
    n, die, F, t = 3001, (0.0, 0.0, 8.0 * nx, 4.0 * ny), 18, 0.75
    w, h = rng.integers(1, 5, n) * 0.375, rng.integers(1, 4, n) * 0.5
    w[::701], h[::701] = 6.0 * nx, 3.0 * ny  # most of the die
    w, h = w.astype(np.float32), h.astype(np.float32)
    x = (die[2] * (0.5 + sigma * rng.standard_normal(n))).astype(np.float32)
    y = (die[3] * (0.5 + sigma * rng.standard_normal(n))).astype(np.float32)
    g = odens.Grid(die, nx, ny, F)
    q = lambda v: odens.quantize(v, F)  # noqa: E731
    M = odens.overlap_map(q(x), q(y), q(w), q(h), g)
    fixed = rng.integers(0, g.BW * g.BH, (nx, ny)) * (rng.random((nx, ny)) < 0.3)
    want = odens.overflow(M, fixed, np.float32(t), g, int(np.sum(q(w) * q(h))))
    up = lambda v: torch.from_numpy(np.ascontiguousarray(v)).cuda()  # noqa: E731
    tau = torch.zeros(1, dtype=torch.float64, device="cuda")
    out = torch.zeros(nx * ny, dtype=torch.int64, device="cuda")
    for _ in range(2):  # (the second call finds the scratch as the first left it)
        place.place_overflow_noalloc(up(x), up(y), up(w), up(h), n, die, (nx, ny, t), F, up(fixed.ravel()),
                                     tau, out)
        np.testing.assert_array_equal(out.cpu().numpy().reshape(nx, ny), M)  # integers
        assert tau.item() == pytest.approx(want, rel=1e-12)  # the exact excess, rounded once or twice
