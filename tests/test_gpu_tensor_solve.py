"""The tensor-core solve where it is asked for (PLACE_DCT_BF16X3): the library's
own choice on these grids is the fast transforms."""
import numpy as np
import pytest

from oracle import density as odens
from oracle import poisson as opois
from paper_2402_18311_gb300 import place, synth

pytestmark = pytest.mark.gpu


def _design(nx, ny, n=8000, seed=21):
    return synth.make_design(n_movable=n, die=(0, 0, 2 * nx, 2 * ny), nx=nx, ny=ny,
                             n_nets=int(n * 1.1), n_pads=16, target_density=0.9, seed=seed)


def _handle(d, **kw):
    return place.place_create(d, place.place_default_params(
        tau_stop=-1.0, max_iters=1000, dct_mode=place.PLACE_DCT_BF16X3, **kw))


@pytest.mark.parametrize("nx,ny,fold", [(128, 128, 1), (256, 256, 1), (512, 256, 1), (256, 512, 1),
                                        (256, 256, 0), (384, 256, 1)])
def test_field_matches_oracle(nx, ny, fold):
    # BF16x3's tolerance: 1e-4 in the 2-norm
    d = _design(nx, ny)
    h = _handle(d, autotune=0, dct_fold=fold)
    try:
        place.place_step(h, 100)
        x, y = np.empty(d.n_cells, np.float32), np.empty(d.n_cells, np.float32)
        place.place_get_positions(h, 0, x, y)
        n, g = d.n_movable, odens.Grid(d.die, nx, ny, place.place_get_info(h).frac_bits)
        q = lambda v: odens.quantize(v, g.F)  # noqa: E731
        M = odens.overlap_map(q(x[:n]), q(y[:n]), q(d.w[:n]), q(d.h[:n]), g)
        F = odens.overlap_map(q(d.x[n:]), q(d.y[n:]), q(d.w[n:]), q(d.h[n:]), g)
        want = opois.poisson(odens.bin_density(M, F, np.float32(0.9), g), g.bin_w, g.bin_h)
        got = [np.empty(nx * ny, np.float32) for _ in range(3)]
        place.place_eval_field(h, 0, *got)
        for a, b in zip(got, want):
            assert np.linalg.norm(a - b.ravel()) < 1e-4 * np.linalg.norm(b)
    finally:
        place.place_destroy(h)


def test_tuning_candidates_give_identical_results():
    # tile widths, split-K and the tuned choice: the same operations per element
    d = _design(256, 256, n=20000, seed=2)
    ref = None
    for cfg in (dict(autotune=0, gemm_bn=128), dict(autotune=0, gemm_bn=64),
                dict(autotune=0, gemm_bn=128, gemm_split=2), dict(autotune=1)):
        h = _handle(d, **cfg)
        try:
            place.place_step(h, 120)
            got = np.empty((2, d.n_cells), np.float32)
            place.place_get_positions(h, 0, got[0], got[1])
        finally:
            place.place_destroy(h)
        ref = got if ref is None else ref
        np.testing.assert_array_equal(got, ref)
