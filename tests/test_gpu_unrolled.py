"""Runs of iterations as one graph: the same as one by one, also across a stop
inside a run and a reset between runs."""
import numpy as np
import pytest

from paper_2402_18311_gb300 import place, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,opts", [(64, {}), (128, {"max_backtracks": 3}), (48, {"wa_streams": 3})])
def test_runs_equal_single_iterations(nx, opts):
    d = synth.make_design(n_movable=1500, die=(0, 0, 256, 256), nx=64, ny=64, n_nets=1600, n_pads=16,
                          target_density=0.9, seed=5)
    d.nx, d.die = nx, (0.0, 0.0, 4.0 * nx, 256.0)
    d.x = np.minimum(d.x, np.float32(4.0 * nx) - d.w)
    out = []
    for chunk in (1, 150):
        prm = place.place_default_params(tau_stop=0.3, max_iters=290, autotune=0, n_copies=2, **opts)
        h = place.place_create(d, prm)
        try:
            got = []
            for r in range(2):
                done = 0
                while done < 300:  # past both stops
                    place.place_step(h, chunk)
                    done += chunk
                for c in (0, 1):
                    x, y = np.empty(d.n_cells, np.float32), np.empty(d.n_cells, np.float32)
                    place.place_get_positions(h, c, x, y)
                    s = place.place_get_state(h, c)
                    got += [x, y, np.array([s.iter, s.converged, s.lambda_, s.alpha])]
                place.place_perturb(h, place.PLACE_SHUFFLE_ALL, 0.5, 3 + r, -1)
            out.append(got)
        finally:
            place.place_destroy(h)
    for a, b in zip(*out):
        np.testing.assert_array_equal(a, b)
