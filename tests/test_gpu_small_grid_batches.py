"""Small grids: one cluster per copy up to 16 copies, the GEMM chain for more, and a
copy's bits are the same on either side of that line."""
import numpy as np
import pytest

from paper_2402_18311_gb300 import place, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny", [(16, 16), (64, 64), (48, 80), (128, 32)])
@pytest.mark.parametrize("opts", [{}, dict(fillers=1), dict(stretch=1)])
def test_copies_on_both_sides_of_the_line(nx, ny, opts):
    d = synth.make_design(n_movable=400, die=(0, 0, 4 * nx, 4 * ny), nx=nx, ny=ny, n_nets=440, n_pads=16,
                          target_density=0.9, seed=nx, init_sigma_frac=0.05)
    d.is_macro = np.zeros(d.n_cells, np.uint8)
    out = {}
    for K in (1, 16, 17, 130):
        h = place.place_create(d, place.place_default_params(tau_stop=-1.0, max_iters=1000, autotune=0, n_copies=K,
                                                             **opts))
        try:
            want = place.PLACE_SOLVE_CLUSTER if K <= 16 else place.PLACE_SOLVE_GEMM_FP32
            assert place.place_get_solve(h) == want
            place.place_step(h, 90)
            got = []
            for c in {0, K - 1}:
                p, f = np.empty((2, d.n_cells), np.float32), np.empty((3, nx * ny), np.float32)
                place.place_get_positions(h, c, p[0], p[1])
                place.place_eval_field(h, c, *f)
                got.append((p, f))
            out[K] = got
        finally:
            place.place_destroy(h)
    for K, got in out.items():
        for p, f in got:
            np.testing.assert_array_equal(p, out[1][0][0])
            np.testing.assert_array_equal(f, out[1][0][1])
