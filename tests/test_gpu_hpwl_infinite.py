"""The exact HPWL with pin offsets that are not finite: an infinite coordinate is
an extent's end like any other, a coordinate that is not a number is left out."""
import numpy as np
import pytest

from paper_2402_18311_gb300 import place, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("deg", [2, 4, 9, 40, 120, 300])  # every degree class
@pytest.mark.parametrize("values,want", [((np.inf,), np.inf), ((-np.inf,), np.inf),
                                         ((np.inf, -np.inf), np.inf), ((np.nan,), None)])
def test_offsets_that_are_not_finite(deg, values, want):
    d = synth.make_design(n_movable=400, die=(0, 0, 1024, 1024), nx=64, ny=64, n_nets=10, n_pads=16,
                          seed=4, init_sigma_frac=0.2)
    rng = np.random.default_rng(deg)
    d.net_ptr = np.array([0, deg, 2 * deg], np.int32)
    d.pin_cell = rng.integers(0, d.n_cells, 2 * deg).astype(np.int32)
    d.pin_dx = rng.random(2 * deg).astype(np.float32)
    d.pin_dy = rng.random(2 * deg).astype(np.float32)
    d.pin_dx[deg - len(values):deg] = values  # the first net's last pins
    h = place.place_create(d, place.place_default_params(autotune=0))
    try:
        hp = np.empty(1)
        place.place_eval_hpwl_overflow(h, hp)
        if want is None:
            x, y = np.empty(d.n_cells, np.float32), np.empty(d.n_cells, np.float32)
            place.place_get_positions(h, 0, x, y)
            px = x[d.pin_cell].astype(np.float64) + d.pin_dx
            py = y[d.pin_cell].astype(np.float64) + d.pin_dy
            ext = lambda v: np.nanmax(v) - np.nanmin(v)  # noqa: E731
            want = sum(ext(px[s]) + ext(py[s]) for s in (slice(0, deg), slice(deg, 2 * deg)))
            # exact extents, and four of them added: a few roundings
            assert abs(hp[0] - want) <= 4 * 2.0 ** -52 * want
        else:
            assert hp[0] == want
    finally:
        place.place_destroy(h)
