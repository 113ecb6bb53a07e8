"""Shuffle's bucketed selection against the oracle at the edges of its plan
(buckets, mask words, tiles) and over a batched handle's copies."""
import numpy as np
import pytest

from oracle import perturb as opt
from paper_2402_18311_gb300 import place, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 2, 32, 33, 96, 97, 8192, 8193, 30011])
@pytest.mark.parametrize("op,p", [(place.PLACE_SHUFFLE_ALL, 0.0), (place.PLACE_SHUFFLE_ALL, 0.01),
                                  (place.PLACE_SHUFFLE_ALL, 0.5), (place.PLACE_SHUFFLE_ALL, 1.0),
                                  (place.PLACE_SHUFFLE_MACRO, 0.5)])
def test_shuffle_matches_oracle(n, op, p):
    # integers and FP64 on both sides: the same positions bit for bit
    d = synth.make_design(n_movable=n, die=(0, 0, 512, 512), nx=64, ny=64, n_nets=max(1, n // 2),
                          n_pads=16, seed=n, init_sigma_frac=0.2)
    d.is_macro[:n] = np.random.default_rng(n).random(n) < 0.3
    K, seed = 3, 41
    h = place.place_create(d, place.place_default_params(n_copies=K, autotune=0))
    try:
        x0, y0 = np.empty(d.n_cells, np.float32), np.empty(d.n_cells, np.float32)
        place.place_get_positions(h, 0, x0, y0)
        cand = np.arange(n) if op == place.PLACE_SHUFFLE_ALL else np.flatnonzero(d.is_macro[:n])
        place.place_perturb(h, op, p, seed, -1)
        for c in range(K):
            want = opt.shuffle(x0, y0, d.w, d.h, cand, p, seed + c, d.die)
            got = np.empty((2, d.n_cells), np.float32)
            place.place_get_positions(h, c, got[0], got[1])
            np.testing.assert_array_equal(got, want)
    finally:
        place.place_destroy(h)
