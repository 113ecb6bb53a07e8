"""Positions in and out through every kind of memory."""
import numpy as np
import pytest

from paper_2402_18311_gb300 import place, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("fillers", [0, 1])
def test_positions_through_host_pinned_and_device_memory(fillers):
    torch = pytest.importorskip("torch")
    d = synth.make_design(n_movable=777, die=(0, 0, 512, 512), nx=64, ny=64, n_nets=400, n_pads=16,
                          target_density=0.9, seed=3)
    h = place.place_create(d, place.place_default_params(autotune=0, n_copies=2, fillers=fillers))
    n = d.n_cells
    try:
        x, y = (v + np.float32(3.25) for v in synth.random_start(d, 5, 0.2))
        want = np.stack([x, y])
        top = np.float32(512) - np.stack([d.w, d.h])
        want[:, :777] = np.clip(want[:, :777], 0, top[:, :777])
        want[:, 777:] = np.stack([d.x, d.y])[:, 777:]
        dev = torch.zeros(4 * n + 8, device="cuda")
        kinds = {
            "host": lambda: torch.zeros(2, n),
            "pinned": lambda: torch.zeros(2, n).pin_memory(),
            "device": lambda: torch.zeros(2, n, device="cuda"),
            # 4-byte aligned only
            "odd": lambda: dev[1:1 + 2 * n].view(2, n).zero_(),
        }
        for make_in in kinds.values():
            src = make_in()
            src[0].copy_(torch.from_numpy(x))
            src[1].copy_(torch.from_numpy(y))
            torch.cuda.synchronize()
            place.place_set_positions(h, -1, torch.from_numpy(d.x), torch.from_numpy(d.y))
            place.place_set_positions(h, 1, src[0], src[1])
            for make_out in kinds.values():
                out = make_out()
                place.place_get_positions(h, 1, out[0], out[1])
                np.testing.assert_array_equal(out.cpu().numpy(), want)
            only = torch.zeros(n, device="cuda")
            place.place_get_positions(h, 1, None, only)
            np.testing.assert_array_equal(only.cpu().numpy(), want[1])
        # the handle's own interleaved view as a source: read before it is written
        vx, _ = place.place_device_views(h, 1)
        flat = np.empty(2 * n, np.float32)
        flat[0::2], flat[1::2] = want
        if not fillers:
            class View:  # (n contiguous floats from the view's start)
                def data_ptr(self):
                    return vx

                def is_contiguous(self):
                    return True
            place.place_set_positions(h, 1, View(), View())
            out = np.empty((2, n), np.float32)
            place.place_get_positions(h, 1, out[0], out[1])
            np.testing.assert_array_equal(out[:, :777], np.clip(flat[:777], 0, top[:, :777]))
    finally:
        place.place_destroy(h)
