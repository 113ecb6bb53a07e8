"""The fused Poisson solves against the FP64 oracle (fast transforms at every
length, the one-cluster kernel of small grids at the edges of its range) and
their bookkeeping of the map."""
import numpy as np
import pytest

from oracle import density as odens
from oracle import poisson as opois
from paper_2402_18311_gb300 import place, synth

pytestmark = pytest.mark.gpu

# Field error against FP64 in the 2-norm.  One FP32 transform of n points adds
# about log2(n) rounding errors of 2^-24 to the norm of its input; three of
# them per direction at n <= 4096 and 2 directions stay below 72 2^-24 =
# 4.3e-6 of the density's norm, and the density's constant part, which the
# solve drops, is at most about twice its varying part on these designs.
FIELD_TOL = 1e-5


def _design(nx, ny, seed=5, n=3000, die=None):
    return synth.make_design(n_movable=n, die=die or (0, 0, 2 * nx, 2 * ny), nx=nx, ny=ny,
                             n_nets=int(1.1 * n), n_pads=16, target_density=0.9, seed=seed)


def _rel(a, b):
    return float(np.linalg.norm(a - b) / np.linalg.norm(b))


def _fields(d, info, x, y):
    n, g = d.n_movable, odens.Grid(d.die, d.nx, d.ny, info.frac_bits)
    q = lambda v: odens.quantize(v, g.F)  # noqa: E731
    W, H = q(d.w), q(d.h)
    M = odens.overlap_map(q(x[:n]), q(y[:n]), W[:n], H[:n], g)
    F = odens.overlap_map(q(d.x[n:]), q(d.y[n:]), W[n:], H[n:], g)
    rho = odens.bin_density(M, F, np.float32(d.target_density), g)
    psi, ex, ey = opois.poisson(rho, g.bin_w, g.bin_h)
    grad = odens.field_gather(q(x[:n]), q(y[:n]), W[:n], H[:n], g, ex, ey)
    return psi.ravel(), ex.ravel(), ey.ravel(), np.concatenate(grad)


@pytest.mark.parametrize("nx,ny,mode", [
    (16, 16, place.PLACE_DCT_AUTO), (48, 80, place.PLACE_DCT_FP32),
    (128, 32, place.PLACE_DCT_AUTO), (16, 128, place.PLACE_DCT_AUTO),
    (64, 64, place.PLACE_DCT_AUTO), (64, 128, place.PLACE_DCT_AUTO),
    (128, 64, place.PLACE_DCT_FP32), (256, 512, place.PLACE_DCT_AUTO),
    (512, 256, place.PLACE_DCT_FP32), (1024, 64, place.PLACE_DCT_AUTO),
    (64, 1024, place.PLACE_DCT_AUTO), (2048, 128, place.PLACE_DCT_AUTO),
    (128, 2048, place.PLACE_DCT_FP32), (4096, 64, place.PLACE_DCT_AUTO),
    (64, 4096, place.PLACE_DCT_AUTO)])
def test_field_and_gradient_match_oracle(nx, ny, mode):
    d = _design(nx, ny)
    h = place.place_create(d, place.place_default_params(tau_stop=-1.0, autotune=0, dct_mode=mode))
    try:
        place.place_step(h, 40)
        x, y = np.empty(d.n_cells, np.float32), np.empty(d.n_cells, np.float32)
        place.place_get_positions(h, 0, x, y)
        want = _fields(d, place.place_get_info(h), x, y)
        got = [np.empty(nx * ny, np.float32) for _ in range(3)]
        place.place_eval_field(h, 0, *got)
        # the planes (with psi) and, through the gradient, the pairs
        assert _rel(got[0], want[0]) < FIELD_TOL
        assert _rel(np.concatenate(got[1:]), np.concatenate(want[1:3])) < FIELD_TOL
        g = np.empty((2, d.n_movable), np.float32)
        place.place_eval_density_grad(h, 0, g[0], g[1])
        assert _rel(g.ravel(), want[3]) < 1e-4  # the gather's own tolerance
    finally:
        place.place_destroy(h)


@pytest.mark.parametrize("nx", [32, 64, 48])  # one cluster; fast transforms; GEMMs
@pytest.mark.parametrize("opts", [{}, {"fillers": 1}, {"stretch": 1}, {"max_backtracks": 5}])
def test_evaluations_between_iterations_change_nothing(nx, opts):
    # an iteration leaves the map zero and an evaluation does not: iterations
    # with every kind of evaluation in between equal those without, also for a
    # copy that is reset meanwhile
    d = _design(nx, 128, seed=8)
    out = []
    for ask in (False, True):
        prm = place.place_default_params(tau_stop=-1.0, autotune=0, n_copies=2, **opts)
        h = place.place_create(d, prm)
        try:
            for k in range(4):
                place.place_step(h, 3)
                if ask:
                    place.place_eval_density(h, k % 2)
                    place.place_step(h, 1)
                    place.place_eval_hpwl_overflow(h)
                    place.place_step(h, 1)
                    place.place_eval_field(h, 0)
                    place.place_step_timed(h, 1, np.zeros(5, np.float32))
                    place.place_eval_density_grad(h, 1)
                else:
                    place.place_step(h, 3)
                if k == 1:
                    place.place_perturb(h, place.PLACE_SHUFFLE_ALL, 0.5, 3, 1)
            pos = np.empty((4, d.n_cells), np.float32)
            place.place_get_positions(h, 0, pos[0], pos[1])
            place.place_get_positions(h, 1, pos[2], pos[3])
            out.append(pos)
        finally:
            place.place_destroy(h)
    np.testing.assert_array_equal(out[0], out[1])


@pytest.mark.parametrize("nx,ny", [(144, 112), (48, 176)])  # sides of 32 k + 16
def test_gemm_tiles_agree(nx, ny):
    # one copy takes the GEMMs' small tiles, forty the wide ones: the same
    # chain of multiply-adds per element, so the same bits
    d = _design(nx, ny, seed=12)
    got = []
    for copies in (1, 40):
        h = place.place_create(d, place.place_default_params(
            tau_stop=-1.0, autotune=0, n_copies=copies, dct_mode=place.PLACE_DCT_FP32))
        try:
            place.place_step(h, 15)
            for c in {0, copies - 1}:
                x, y = np.empty(d.n_cells, np.float32), np.empty(d.n_cells, np.float32)
                place.place_get_positions(h, c, x, y)
                e = np.empty((2, nx * ny), np.float32)
                place.place_eval_field(h, c, None, e[0], e[1])
                got.append((x, y, e))
        finally:
            place.place_destroy(h)
    for other in got[1:]:
        for a, b in zip(got[0], other):
            np.testing.assert_array_equal(a, b)
