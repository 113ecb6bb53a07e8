"""Runs of iterations as one graph on the solves whose map, or stretched map, is
cleared inside every iteration, and with the fillers' doubled map: the same as one
by one.  And a placement between whose iterations every evaluation and measurement
runs: unchanged by them."""
import numpy as np
import pytest

from paper_2402_18311_gb300 import place, synth

pytestmark = pytest.mark.gpu
GEMM = dict(dct_mode=place.PLACE_DCT_BF16X3)
CASES = [(144, 112, {}), (128, 128, GEMM), (256, 256, GEMM), (64, 64, dict(stretch=1)),
         (128, 64, dict(stretch=1, wa_streams=2)), (128, 128, dict(GEMM, stretch=1)), (64, 48, dict(fillers=1)),
         (128, 128, dict(fillers=1)), (144, 112, dict(fillers=1, wa_streams=2))]


def _design(nx, ny):
    return synth.make_design(n_movable=1500, die=(0, 0, 2 * nx, 2 * ny), nx=nx, ny=ny, n_nets=1600, n_pads=16,
                             target_density=0.9, seed=5)


def _state(h, d, K):
    got = []
    for c in range(K):
        p = np.empty((2, d.n_cells), np.float32)
        place.place_get_positions(h, c, p[0], p[1])
        s = place.place_get_state(h, c)
        got += [p, np.array([s.iter, s.converged, s.lambda_, s.alpha, s.overflow, s.bins_effective])]
    return got


@pytest.mark.parametrize("nx,ny,opts", CASES)
def test_runs_equal_single_iterations(nx, ny, opts):
    d = _design(nx, ny)
    out = []
    for chunk in (1, 150):
        h = place.place_create(d, place.place_default_params(tau_stop=0.3, max_iters=290, autotune=0, n_copies=2,
                                                             **opts))
        try:
            got = []
            for r in range(2):
                for _ in range(300 // chunk):  # past both stops
                    place.place_step(h, chunk)
                got += _state(h, d, 2)
                place.place_perturb(h, place.PLACE_SHUFFLE_ALL, 0.5, 3 + r, -1)
            out.append(got)
        finally:
            place.place_destroy(h)
    for a, b in zip(*out):
        np.testing.assert_array_equal(a, b)


@pytest.mark.parametrize("nx,ny,opts", CASES + [(64, 64, {}), (128, 64, {})])
def test_evaluations_and_measurements_between_iterations_change_nothing(nx, ny, opts):
    d = _design(nx, ny)
    out = []
    for looks in (False, True):
        h = place.place_create(d, place.place_default_params(tau_stop=-1.0, autotune=0, n_copies=2, **opts))
        try:
            for n in (1, 30, 90, 20):
                place.place_step(h, n)
                if looks:
                    f, g = np.empty((3, nx * ny), np.float32), np.empty((2, d.n_movable), np.float32)
                    m, hp, tau = np.empty(nx * ny, np.int64), np.empty(2), np.empty(2)
                    place.place_measure_scatter_floor(h, 2)
                    place.place_measure_wa_floor(h, 2)
                    place.place_eval_density(h, 1, m)
                    place.place_eval_density(h, 0, None)
                    place.place_eval_field(h, 1, *f)
                    place.place_eval_density_grad(h, 0, g[0], g[1])
                    place.place_eval_wirelength(h, 1, 3.0, g[0], g[1])
                    place.place_eval_hpwl_overflow(h, hp, tau)
                    place.place_measure_scatter_floor(h, 1)
            out.append(_state(h, d, 2))
        finally:
            place.place_destroy(h)
    for a, b in zip(*out):
        np.testing.assert_array_equal(a, b)
