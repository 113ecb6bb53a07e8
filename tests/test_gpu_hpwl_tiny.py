"""The exact HPWL of coordinates at both ends of FP32: subnormal extents to their
last bit, and sums beyond FP32's largest number."""
import numpy as np
import pytest

from paper_2402_18311_gb300 import place, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("deg", [2, 4, 9, 40, 120, 300])  # every degree class
@pytest.mark.parametrize("unit", [2.0 ** -149, 1e36])
def test_extents_at_the_ends_of_fp32(deg, unit):
    d = synth.make_design(n_movable=50, die=(0, 0, 1024, 1024), nx=64, ny=64, n_nets=10, n_pads=16, seed=4)
    d.x[0] = d.y[0] = 0.0
    d.net_ptr = np.array([0, deg], np.int32)
    d.pin_cell = np.zeros(deg, np.int32)
    k = np.arange(deg, dtype=np.float64)  # offsets in units: odd extents
    d.pin_dx = (unit * (k - 1)).astype(np.float32)
    d.pin_dy = (unit * np.where(k == deg - 1, 3, 0)).astype(np.float32)
    if unit > 1:
        d.pin_dx[:2] = -3e38, 3e38
    h = place.place_create(d, place.place_default_params(autotune=0))
    try:
        hp = np.empty(1)
        place.place_eval_hpwl_overflow(h, hp)
        want = np.ptp(d.pin_dx.astype(np.float64)) + np.ptp(d.pin_dy.astype(np.float64))
        assert want > 0 and hp[0] == want  # both exact but for the one addition
    finally:
        place.place_destroy(h)
