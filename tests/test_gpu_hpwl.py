"""The exact HPWL at the edges of the kernels' degree classes."""
import math

import numpy as np
import pytest

from paper_2402_18311_gb300 import place, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("weighted", [False, True])
@pytest.mark.parametrize("origin", [0.0, -512.0, 3000.0])
def test_hpwl_of_every_degree_class(weighted, origin):
    # pin coordinates and extents are exact on both sides and the sums round in
    # FP64: about 30 additions deep here, 30 2^-53 = 3.3e-15
    rng = np.random.default_rng(9)
    d = synth.make_design(n_movable=4000, die=(origin, origin, origin + 1024, origin + 1024), nx=64,
                          ny=64, n_nets=10, n_pads=16, seed=4, init_sigma_frac=0.2)
    deg = np.array(([0, 1, 2, 3, 4, 5, 8, 15, 16, 17, 33, 63, 64, 65, 255, 256, 257, 1500] * 9)[:-5])
    d.net_ptr = np.concatenate([[0], np.cumsum(deg)]).astype(np.int32)
    P = int(d.net_ptr[-1])
    d.pin_cell = rng.integers(0, d.n_cells, P).astype(np.int32)
    # offsets whose sum with a position needs more digits than FP32 has
    d.pin_dx = (rng.random(P) * d.w[d.pin_cell]).astype(np.float32)
    d.pin_dy = (rng.random(P) * 1e-3).astype(np.float32)
    if weighted:
        d.net_w = rng.choice(np.array([0.1, 1.0, 3.25], np.float32), deg.size)
    h = place.place_create(d, place.place_default_params(autotune=0, n_copies=2))
    try:
        hp = np.empty(2)
        place.place_eval_hpwl_overflow(h, hp)
        x, y = np.empty(d.n_cells, np.float32), np.empty(d.n_cells, np.float32)
        place.place_get_positions(h, 0, x, y)
        px = x[d.pin_cell].astype(np.float64) + d.pin_dx.astype(np.float64)
        py = y[d.pin_cell].astype(np.float64) + d.pin_dy.astype(np.float64)
        w = d.net_w.astype(np.float64) if weighted else np.ones(deg.size)
        cut = [slice(*d.net_ptr[e:e + 2]) for e in range(deg.size)]
        want = math.fsum(w[e] * (np.ptp(px[s]) + np.ptp(py[s])) for e, s in enumerate(cut) if deg[e])
        assert hp[0] == hp[1] and abs(hp[0] - want) <= 3.3e-15 * want
    finally:
        place.place_destroy(h)
