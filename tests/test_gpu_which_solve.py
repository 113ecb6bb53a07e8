"""place_get_solve names the solve that runs, where place_info.dct_mode names the
mode that a grid resolves to."""
import numpy as np
import pytest

from paper_2402_18311_gb300 import place, synth

pytestmark = pytest.mark.gpu
AUTO, FP32, BF16 = place.PLACE_DCT_AUTO, place.PLACE_DCT_FP32, place.PLACE_DCT_BF16X3


@pytest.mark.parametrize("nx,ny,opts,want", [
    (64, 64, dict(dct_mode=AUTO), place.PLACE_SOLVE_CLUSTER),
    (48, 80, dict(dct_mode=FP32), place.PLACE_SOLVE_CLUSTER),
    (144, 80, dict(dct_mode=AUTO), place.PLACE_SOLVE_GEMM_FP32),
    (384, 128, dict(dct_mode=FP32), place.PLACE_SOLVE_GEMM_FP32),
    (384, 128, dict(dct_mode=AUTO), place.PLACE_SOLVE_GEMM_BF16X3),
    (128, 128, dict(dct_mode=BF16), place.PLACE_SOLVE_GEMM_BF16X3),
    (256, 256, dict(dct_mode=AUTO, dct_fold=0), place.PLACE_SOLVE_GEMM_BF16X3),
    (256, 256, dict(dct_mode=AUTO), place.PLACE_SOLVE_FFT),
    (128, 64, dict(dct_mode=FP32), place.PLACE_SOLVE_FFT),
    (128, 128, dict(dct_mode=AUTO, gemm_bn=64, gemm_split=1), place.PLACE_SOLVE_FFT)])
def test_which_solve_runs(nx, ny, opts, want):
    d = synth.make_design(n_movable=500, die=(0, 0, 2 * nx, 2 * ny), nx=nx, ny=ny, n_nets=500, n_pads=16, seed=1)
    h = place.place_create(d, place.place_default_params(autotune=0, **opts))
    try:
        assert place.place_get_solve(h) == want
        # launches of an iteration: scatter, finish and four GEMMs; scatter and
        # three; scatter and one; then the wirelength's classes, gradient and update
        solve = {place.PLACE_SOLVE_FFT: 4, place.PLACE_SOLVE_CLUSTER: 2}.get(want, 6)
        classes = len({int(np.searchsorted([4, 16, 64, 256], k)) for k in np.diff(d.net_ptr)})
        assert place.place_get_info(h).kernels_per_iter == solve + classes + 2
    finally:
        place.place_destroy(h)
