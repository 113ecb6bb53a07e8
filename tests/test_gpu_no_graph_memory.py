"""Without memory for the graph of several iterations a handle runs one iteration
at a time: no error, the same results."""
import numpy as np
import pytest

from paper_2402_18311_gb300 import place, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("step", [1, 2])  # at the graph's instantiation, at its upload
def test_iterations_without_memory_for_their_graph(step):
    d = synth.tiny_1k(3)
    out = []
    for fail in (0, step):
        h = place.place_create(d, place.place_default_params(tau_stop=-1.0, max_iters=1000, autotune=0))
        try:
            place.place_test_no_graph_memory(h, fail)
            for n in (100, 77, 60):
                place.place_step(h, n)
            got = np.empty((2, d.n_cells), np.float32)
            place.place_get_positions(h, 0, got[0], got[1])
            assert place.place_get_state(h, 0).iter == 237
            out.append(got)
        finally:
            place.place_destroy(h)
    np.testing.assert_array_equal(out[0], out[1])


def test_the_failure_is_asked_for_by_step():
    h = place.place_create(synth.tiny_1k(0), place.place_default_params(autotune=0))
    try:
        with pytest.raises(RuntimeError):
            place.place_test_no_graph_memory(h, 3)
    finally:
        place.place_destroy(h)
