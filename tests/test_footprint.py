"""The footprint estimate of batches of small designs, by which a caller and the
job server admit: its reduction partials are bounded per copy."""
from paper_2402_18311_gb300 import place, synth


def test_footprint_of_many_small_copies():
    d = synth.make_design(n_movable=1000, die=(0, 0, 256, 256), nx=64, ny=64, n_nets=1000, n_pads=16,
                          target_density=0.9, seed=3)
    K = 4096
    got = place.place_estimate_device_bytes(d, place.place_default_params(n_copies=K))
    # per copy: nine ranges of partials (8 bytes, at most 4 x 1024 blocks of short nets
    # and 8192 of long ones) and the overflow's (20 bytes), the history (4096 records
    # of 48 bytes), 200 bytes a cell, 80 bytes a bin; 2% for the alignment and the rest
    per_copy = (9 * 8 + 20) * (4 * 1024 + 8192) + 4096 * 48 + 200 * 1016 + 80 * 4096
    assert got < 1.02 * K * per_copy
