"""The density weight's factor mu_base^(1 - dHPWL / dref) keeps FP64 accuracy for
exponents far from 0, where a clamp wider than the default lets it through."""
import math

import numpy as np
import pytest

from paper_2402_18311_gb300 import place, synth

pytestmark = pytest.mark.gpu


def _two_iterations(d, **kw):
    h = place.place_create(d, place.place_default_params(tau_stop=-1.0, autotune=0, mu_lo=1e-30, mu_hi=1e30, **kw))
    try:
        place.place_step(h, 2)
        info = place.place_get_info(h)
        return place.place_get_history(h, 0), math.sqrt(info.bin_w * info.bin_h)
    finally:
        place.place_destroy(h)


@pytest.mark.parametrize("base", [1.1, 0.7, 2.0])
def test_lambda_factor(base):
    d = synth.make_design(n_movable=1000, die=(0, 0, 256, 256), nx=64, ny=64, n_nets=1100, n_pads=16, seed=2)
    lg = math.log2(np.float32(base))
    rec, w_bin = _two_iterations(d)
    dh = rec[1].hpwl_wa - rec[0].hpwl_wa  # (the same whatever hpwl_ref is)
    for e in (-90, -61.3, -17.1, 0.3, 5.9, 33.3, 71.7, 95):  # y log2 mu_base
        ref = dh / ((1.0 - e / lg) * d.n_nets * w_bin)
        if ref <= 0:  # the HPWL rises or falls: one sign of the exponent
            continue
        ref = np.float32(ref)
        rec, _ = _two_iterations(d, mu_base=base, hpwl_ref=ref)
        assert rec[1].hpwl_wa - rec[0].hpwl_wa == dh
        y = 1.0 - dh / (float(ref) * d.n_nets * w_bin)
        want = rec[0].lambda_ * math.pow(float(np.float32(base)), y)
        # two roundings of the series' sum, one of the product, one here
        assert abs(rec[1].lambda_ - want) <= 4 * 2.0 ** -52 * want, (e, rec[1].lambda_ / want - 1)
