"""Cells of many bins (the warp-wide steps of the scatter and of the field
gather) in every way of the scatter, with and without stretching."""
import numpy as np
import pytest

from oracle import density as odens
from oracle import poisson as opois
from paper_2402_18311_gb300 import place, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("stretch", [0, 1])
@pytest.mark.parametrize("mode", [-1, 0, 1, 2])
@pytest.mark.parametrize("sigma", [1e-3, 0.25])
def test_maps_and_gradient_with_cells_of_many_bins(mode, stretch, sigma):
    # macros from 1 bin to 40 x 40 bins among 1000 cells (1000 is no multiple of
    # a warp), on the edges of 5 x 6 and 4 x 8 bins too
    d = synth.make_design(n_movable=1000, die=(0, 0, 512, 256), nx=128, ny=64, n_nets=500,
                          n_pads=16, target_density=0.9, seed=2, init_sigma_frac=sigma)
    sides = [(4, 4), (8, 8), (16, 20), (16, 24), (16, 28), (12, 32), (160, 160), (3, 200), (400, 2)]
    n = d.n_movable
    at = np.r_[0, 31, 32, 500:505, n - 1]
    for i, (w, h) in zip(at, sides):
        d.w[i], d.h[i] = w, h
        d.x[i] = min(d.x[i], 512 - w)
        d.y[i] = min(d.y[i], 256 - h)
    h = place.place_create(d, place.place_default_params(autotune=0, stretch=stretch, scatter_mode=mode))
    try:
        x, y = np.empty(d.n_cells, np.float32), np.empty(d.n_cells, np.float32)
        place.place_get_positions(h, 0, x, y)
        g = odens.Grid(d.die, d.nx, d.ny, place.place_get_info(h).frac_bits)
        q = lambda v: odens.quantize(v[:n], g.F)  # noqa: E731
        X, Y, W, H = q(x), q(y), q(d.w), q(d.h)
        M = odens.overlap_map(X, Y, W, H, g)
        gm = np.empty(d.nx * d.ny, np.int64)
        place.place_eval_density(h, 0, gm)
        np.testing.assert_array_equal(gm.reshape(d.nx, d.ny), M)  # integers
        weight = 1.0
        if stretch:
            X, Y, W, H, R, weight = odens.stretched(X, Y, W, H, g)
            M = odens.overlap_map_scaled(X, Y, W, H, R, g)
            place.place_get_stretched_map(h, 0, gm)
            np.testing.assert_array_equal(gm.reshape(d.nx, d.ny), M)
        qf = lambda v: odens.quantize(v[n:], g.F)  # noqa: E731
        F = odens.overlap_map(qf(d.x), qf(d.y), qf(d.w), qf(d.h), g)
        _, ex, ey = opois.poisson(odens.bin_density(M, F, np.float32(d.target_density), g), g.bin_w, g.bin_h)
        want = np.stack(odens.field_gather(X, Y, W, H, g, ex, ey)) * weight
        got = np.empty((2, n), np.float32)
        place.place_eval_density_grad(h, 0, got[0], got[1])
        # the gather's tolerance, over all cells and over the large ones
        for s in (slice(None), at):
            assert np.linalg.norm(got[:, s] - want[:, s]) < 1e-4 * np.linalg.norm(want[:, s])
    finally:
        place.place_destroy(h)
