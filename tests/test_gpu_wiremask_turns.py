"""WireMask over more copies than its scratch is for at a time: every copy moves as
the copy alone does, and the scratch stays bounded."""
import numpy as np
import pytest

from paper_2402_18311_gb300 import place, synth

pytestmark = pytest.mark.gpu


def test_copies_in_turns_equal_one_copy():
    torch = pytest.importorskip("torch")
    # 400 macros on nets of 3159 pins: about 130 KB a copy, 540 MB for 4096 copies
    # at once, so that they take three turns
    d = synth.make_design(n_movable=400, die=(0, 0, 256, 256), nx=16, ny=16, n_nets=800, n_pads=16,
                          target_density=0.9, seed=11, init_sigma_frac=0.2)
    d.is_macro = (np.arange(d.n_cells) < 400).astype(np.uint8)
    want = None
    for K in (1, 4096):
        h = place.place_create(d, place.place_default_params(autotune=0, n_copies=K))
        try:
            torch.cuda.synchronize()
            free = torch.cuda.mem_get_info()[0]
            place.place_perturb(h, place.PLACE_WIREMASK, 0.0, 0, -1)
            for c in sorted({0, K // 3, K // 2, 2 * K // 3, K - 1}):
                got = np.empty((2, d.n_cells), np.float32)
                place.place_get_positions(h, c, got[0], got[1])
                want = got if want is None else want
                np.testing.assert_array_equal(got, want)
            # the scratch, its pool's rounding, and a graph of 2400 launches
            assert free - torch.cuda.mem_get_info()[0] < 400 << 20
        finally:
            place.place_destroy(h)
    assert not np.array_equal(want[0][:400], d.x[:400])
