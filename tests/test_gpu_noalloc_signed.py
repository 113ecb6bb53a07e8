"""The allocation-free overflow takes the fixed map's entries as the signed
integers that they are."""
import numpy as np
import pytest

from paper_2402_18311_gb300 import place

pytestmark = pytest.mark.gpu


def test_fixed_map_entries_are_signed():
    torch = pytest.importorskip("torch")
    rng = np.random.default_rng(8)
    nx, ny, n, F, t = 24, 16, 2000, 10, 0.75
    A = (4 << F) * (4 << F)
    q = lambda lo, hi: rng.integers(lo, hi, n)  # noqa: E731
    x, y, w, h = q(0, 4 * nx - 3), q(0, 4 * ny - 3), q(1, 4), q(1, 4)  # (whole units)
    M = np.zeros((nx, ny), dtype=object)
    for i in range(n):
        for bx in range(x[i] // 4, (x[i] + w[i] - 1) // 4 + 1):
            for by in range(y[i] // 4, (y[i] + h[i] - 1) // 4 + 1):
                M[bx, by] += ((int(min(x[i] + w[i], 4 * bx + 4) - max(x[i], 4 * bx)) << F)
                              * (int(min(y[i] + h[i], 4 * by + 4) - max(y[i], 4 * by)) << F))
    fixed = rng.integers(-A, A, (nx, ny))
    fixed[0] = [-(2 ** 40), -1, 0, 1] * 4
    # excess of the bins, times 4: integers
    excess = sum(max(0, 4 * int(M[i, j]) - 3 * (A - int(fixed[i, j]))) for i in range(nx) for j in range(ny))
    want = excess / (4 * int(np.sum(w * h) << (2 * F)))
    up = lambda v: torch.from_numpy(np.ascontiguousarray(v, np.float32)).cuda()  # noqa: E731
    tau = torch.zeros(1, dtype=torch.float64, device="cuda")
    place.place_overflow_noalloc(up(x), up(y), up(w), up(h), n, (0.0, 0.0, 4.0 * nx, 4.0 * ny), (nx, ny, t), F,
                                 torch.from_numpy(fixed.ravel()).cuda(), tau, None)
    # the exact excess rounded once, and one division
    assert abs(tau.item() - want) <= 2 * 2.0 ** -52 * want
