"""The tensor cores' solve (PLACE_DCT_BF16X3) in whole placements, stage by stage,
batched, with every tile, and behind a wait that gave up: on grids where the
library itself would choose the fast transforms."""
import numpy as np
import pytest

from paper_2402_18311_gb300 import place, synth
from test_gpu_parity import (Handle, _fold_design, _tiny_128, chaos_horizon_check, check_stages, rel_l2,
                             spread)

pytestmark = pytest.mark.gpu


def _handle(d, **kw):
    kw = dict(dict(tau_stop=-1.0, max_iters=1000), **kw)
    h = Handle(d, dct_mode=place.PLACE_DCT_BF16X3, **kw)
    assert place.place_get_solve(h.h) == place.PLACE_SOLVE_GEMM_BF16X3
    return h


@pytest.mark.parametrize("make", [_tiny_128, lambda: synth.scaled(20000, 128, seed=2)])
def test_trajectory_to_its_chaos_horizon(make):
    # HPWL within 1e-3 up to iteration 220, from where the oracle leaves its own
    # twin one ulp away; shadowed from the oracle's states at 240 and 280
    d = make()
    h = _handle(d)
    try:
        chaos_horizon_check(h, d, make, 220, (240, 280))
    finally:
        h.close()


@pytest.mark.parametrize("nx,ny,die,fold", [
    (256, 256, None, 1), (512, 256, (-512, -256, 512, 256), 1), (256, 512, (1000, 3000, 1512, 4024), 1),
    (128, 384, (-128, 512, 128, 1280), 0), (512, 512, None, 1)])
def test_stages_match_oracle(nx, ny, die, fold):
    # square and oblong grids, dies away from zero, the start and once spread
    h = _handle(_fold_design(nx, ny, die))
    try:
        assert h.info.dct_fold == fold
        x, y = h.pos()
        check_stages(h, x, y, 2.0)
        x, y = spread(h, 150)
        check_stages(h, x, y, 2.0)
    finally:
        h.close()


def test_field_with_fillers_and_stretching():
    # the tensor cores' field and the fast transforms' (which the oracle checks with
    # either option) agree within the sum of their tolerances
    d = _fold_design(256, 256, n=6000, seed=8)
    for kw in (dict(fillers=1), dict(stretch=1), dict(stretch=1, dct_fold=0)):
        fields = []
        for mode in (place.PLACE_DCT_BF16X3, place.PLACE_DCT_FP32):
            h = Handle(d, tau_stop=-1.0, max_iters=1000, autotune=0, dct_mode=mode, **kw)
            try:
                f = np.empty((3, d.nx * d.ny), np.float32)
                place.place_eval_field(h.h, 0, *f)
                fields.append(f)
            finally:
                h.close()
        assert rel_l2(*fields) < 1e-4 + 1e-5


@pytest.mark.parametrize("nx,fold", [(128, 0), (256, 1), (256, 0)])
def test_candidates_give_identical_results(nx, fold):
    # tile widths, split-K, the scatter's ways, big-net cache sizes and WA
    # branches: the same operations in the same order per element
    d = synth.scaled(20000, 128, seed=2) if nx == 128 else _fold_design(256, 256, n=20000, seed=2)
    ref = None
    for cfg in (dict(gemm_bn=128, scatter_mode=0, wa_big_cap=256, wa_streams=1),
                dict(gemm_bn=64, scatter_mode=1, wa_big_cap=4096, wa_streams=2),
                dict(gemm_bn=128, gemm_split=2, scatter_mode=2, wa_streams=3), dict(autotune=1)):
        h = _handle(d, dct_fold=fold, **dict(dict(autotune=0), **cfg))
        try:
            got = []
            for n in (5, 100, 200):
                place.place_step(h.h, n)
                gm = np.empty(d.nx * d.ny, np.int64)
                place.place_eval_density(h.h, 0, gm)
                got += [*h.pos(), gm]
        finally:
            h.close()
        ref = ref or got
        for a, b in zip(got, ref):
            np.testing.assert_array_equal(a, b)


def test_split_matches_the_plain_gemms():
    # fields within 1e-5 of one another, and the same 100 iterations (HPWL 2e-5,
    # overflow 1e-5)
    d = _fold_design(256, 256, n=20000, seed=3)
    out = []
    for fold in (0, 1):
        h = _handle(d, dct_fold=fold)
        try:
            assert h.info.dct_fold == fold
            f = [np.empty(d.nx * d.ny, np.float32) for _ in range(3)]
            place.place_eval_field(h.h, 0, *f)
            place.place_step(h.h, 100)
            hp, tv = np.empty(1), np.empty(1)
            place.place_eval_hpwl_overflow(h.h, hp, tv)
            out.append((f, hp[0], tv[0]))
        finally:
            h.close()
    for a, b in zip(out[0][0], out[1][0]):
        assert rel_l2(b, a) < 1e-5
    assert out[1][1] == pytest.approx(out[0][1], rel=2e-5)
    assert out[1][2] == pytest.approx(out[0][2], abs=1e-5)


@pytest.mark.parametrize("nx,n", [(256, 6000), (128, 4000)])
def test_batched_copies_equal_solo_runs(nx, n):
    d, K = _fold_design(nx, nx, n=n, seed=4), 3
    hb = _handle(d, n_copies=K, autotune=0)
    try:
        place.place_step(hb.h, 40)
        x, y = hb.pos(0)
        place.place_set_positions(hb.h, -1, x, y)
        place.place_perturb(hb.h, place.PLACE_SHUFFLE_ALL, 0.5, 7, -1)
        place.place_step(hb.h, 50)
        finals = [hb.pos(c) for c in range(K)]
    finally:
        hb.close()
    for c in range(K):
        hs = _handle(d, autotune=0)
        try:
            place.place_set_positions(hs.h, 0, x, y)
            place.place_perturb(hs.h, place.PLACE_SHUFFLE_ALL, 0.5, 7 + c, 0)
            place.place_step(hs.h, 50)
            np.testing.assert_array_equal(finals[c], hs.pos())
        finally:
            hs.close()


def test_a_wait_that_gave_up_leaves_the_solve_usable():
    # (about two seconds)
    d = _tiny_128()
    h, ref = _handle(d, autotune=0), _handle(d, autotune=0)
    try:
        place.place_step(h.h, 5)
        place.place_step(ref.h, 5)
        assert place.place_test_wait_timeout(h.h) == place.PLACE_ETIMEOUT
        conv = np.zeros(1, np.int32)
        for x in (h, ref):
            place.place_step(x.h, 30, conv)
        np.testing.assert_array_equal(h.pos(), ref.pos())
    finally:
        h.close()
        ref.close()
