"""place_state.bins_effective is an FP64 quotient: (sum M)^2 over the pass's FP32
sum of squares, not rounded to FP32 itself."""
import numpy as np
import pytest

from paper_2402_18311_gb300 import place, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny", [(64, 64), (128, 64), (144, 80)])  # one cluster, fast transforms, GEMMs
def test_bins_effective_is_fp64(nx, ny):
    d = synth.make_design(n_movable=3000, die=(0, 0, 4 * nx, 4 * ny), nx=nx, ny=ny, n_nets=3300, n_pads=16,
                          target_density=0.9, seed=6)
    h = place.place_create(d, place.place_default_params(tau_stop=-1.0, autotune=0))
    try:
        G = np.empty(nx * ny, np.int64)
        fp64 = 0
        for _ in range(12):
            # the map of the positions that the next iteration's density pass sees
            place.place_eval_density(h, 0, G)
            place.place_step(h, 1)
            got = place.place_get_state(h, 0).bins_effective
            m = G.astype(np.float64)
            want = m.sum() ** 2 / (m * m).sum()
            # an FP32 sum of nx ny squares of FP32 numbers, in chains of at most
            # nx ny / 256 additions, then a tree
            assert abs(got - want) <= 2.0 ** -24 * (nx * ny / 256 + 16) * want
            fp64 += float(np.float32(got)) != got
        assert fp64 >= 10  # (a quotient of 53 bits is an FP32 number by chance only)
    finally:
        place.place_destroy(h)
