"""WireMask where many macros share a net: bit for bit the oracle's corners, and
tables that grow with the pins, not with the square of a net's macros."""
import numpy as np
import pytest

from oracle import wiremask as owm
from paper_2402_18311_gb300 import place, synth

pytestmark = pytest.mark.gpu


def _positions(h, d, copy=0):
    x, y = np.empty(d.n_cells, np.float32), np.empty(d.n_cells, np.float32)
    place.place_get_positions(h, copy, x, y)
    return x, y


@pytest.mark.parametrize("macros", [2, 33, 300])
def test_nets_of_many_macros_match_oracle(macros):
    rng = np.random.default_rng(macros)
    d = synth.make_design(n_movable=600, die=(-256, 64, 256, 448), nx=64, ny=48, n_nets=40, n_pads=16,
                          target_density=0.9, seed=7, init_sigma_frac=0.3)
    d.is_macro = np.zeros(d.n_cells, np.uint8)
    mac = rng.choice(600, macros, replace=False)
    d.is_macro[mac] = 1
    # nets of all macros (some with several pins of one), of pairs, of one
    # macro alone, of macros and other cells, and of no macro
    other = np.setdiff1d(np.arange(d.n_cells), mac)
    nets = [mac, np.concatenate([mac, mac[: macros // 2], other[:40]]), np.concatenate([other[-300:], mac[:1]]),
            mac[:2], mac[-1:], other[:7]]
    nets += [rng.choice(d.n_cells, int(k), replace=False) for k in rng.integers(2, 500, 12)]
    deg = np.array([len(n) for n in nets])
    d.net_ptr = np.concatenate([[0], np.cumsum(deg)]).astype(np.int32)
    d.pin_cell = np.concatenate([rng.permutation(n) for n in nets]).astype(np.int32)
    P = int(d.net_ptr[-1])
    d.pin_dx = (rng.random(P) * d.w[d.pin_cell]).astype(np.float32)
    d.pin_dy = (rng.random(P) * d.h[d.pin_cell]).astype(np.float32)
    d.net_w = rng.uniform(0.5, 2.0, deg.size).astype(np.float32)
    h = place.place_create(d, place.place_default_params(autotune=0, n_copies=2))
    try:
        for rnd in range(2):  # (a second pass starts from the first one's places)
            before = [_positions(h, d, c) for c in (0, 1)]
            place.place_perturb(h, place.PLACE_WIREMASK, 0.0, 0, -1)
            for c, (x, y) in enumerate(before):
                want = owm.wiremask(x, y, d.w, d.h, d.net_ptr, d.pin_cell, d.pin_dx, d.pin_dy, 600,
                                    d.is_macro, d.die, d.nx, d.ny, net_w=d.net_w)
                np.testing.assert_array_equal(np.stack(_positions(h, d, c)), np.stack(want))
            place.place_perturb(h, place.PLACE_SHUFFLE_MACRO, 0.7, 3, 1)
    finally:
        place.place_destroy(h)


def _resident_kb():
    with open("/proc/self/status") as f:
        return next(int(line.split()[1]) for line in f if line.startswith("VmRSS"))


def test_tables_are_linear_in_the_pins():
    # one net of 6000 macros.  With every macro's copy of the net's pins the
    # handle would hold 6000^2 entries of 4 bytes (144 MB); a linear table is
    # below a megabyte, and 48 MB leave room for what else a handle allocates
    n = 6000
    d = synth.make_design(n_movable=n, die=(0, 0, 1024, 1024), nx=64, ny=64, n_nets=10, n_pads=16,
                          target_density=0.9, seed=1)
    d.net_ptr = np.array([0, n], np.int32)
    d.pin_cell = np.arange(n, dtype=np.int32)
    d.pin_dx = d.pin_dy = np.full(n, 0.5, np.float32)
    place.place_destroy(place.place_create(d, place.place_default_params(autotune=0)))
    d.is_macro = (np.arange(d.n_cells) < n).astype(np.uint8)
    start = _resident_kb()
    h = place.place_create(d, place.place_default_params(autotune=0))
    try:
        assert _resident_kb() - start < 48 * 1024
    finally:
        place.place_destroy(h)
