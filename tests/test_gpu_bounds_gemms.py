"""The bounds-checking build on the GEMM solves (the tensor cores' with every tile,
split-K and the even/odd split, the FP32 ones with both tile sizes) and on
WireMask's tables of shared nets: every check passes, and the results are those of
the normal build bit for bit.  Each build runs in a child process."""
import json
import os
import subprocess
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SCRIPT = r"""
import hashlib, json, sys
import numpy as np
sys.path.insert(0, sys.argv[1])
from paper_2402_18311_gb300 import place, synth

def design(nx, ny, n=4000):
    return synth.make_design(n_movable=n, die=(0, 0, 2 * nx, 2 * ny), nx=nx, ny=ny, n_nets=n + n // 10,
                             n_pads=16, target_density=0.9, seed=5)

def hsh(*arrs):
    return hashlib.sha1(b"".join(np.ascontiguousarray(a).tobytes() for a in arrs)).hexdigest()

def evals(h, d):
    n, G = d.n_movable, d.nx * d.ny
    pos, f, g = np.empty((2, d.n_cells), np.float32), np.empty((3, G), np.float32), np.empty((4, n), np.float32)
    hp, m = np.empty(place.place_get_info(h).n_copies), np.empty(G, np.int64)
    place.place_eval_hpwl_overflow(h, hp)
    place.place_eval_density(h, 0, m)
    place.place_eval_field(h, 0, *f)
    place.place_eval_wirelength(h, 0, 4.0, g[0], g[1])
    place.place_eval_density_grad(h, 0, g[2], g[3])
    place.place_get_positions(h, 0, *pos)
    return hsh(pos, f, g, hp, m)

out, checked = {}, []
B, F = place.PLACE_DCT_BF16X3, place.PLACE_DCT_FP32
cases = [(128, 128, B, dict(autotune=1, fillers=1)), (128, 128, B, dict(gemm_bn=64, gemm_split=1)),
         (128, 256, B, dict(gemm_bn=128, gemm_split=2)), (256, 256, B, dict(gemm_bn=128, gemm_split=2)),
         (256, 256, B, dict(gemm_bn=64, stretch=1)), (256, 256, B, dict(dct_fold=0, n_copies=2)),
         (144, 80, F, {}), (80, 112, F, dict(stretch=1, n_copies=3)), (496, 752, F, {})]
for i, (nx, ny, mode, kw) in enumerate(cases):
    d = design(nx, ny)
    h = place.place_create(d, place.place_default_params(**dict(dict(
        tau_stop=-1.0, max_iters=10**6, autotune=0, dct_mode=mode), **kw)))
    want = place.PLACE_SOLVE_GEMM_BF16X3 if mode == B else place.PLACE_SOLVE_GEMM_FP32
    assert place.place_get_solve(h) == want
    checked.append(place.place_get_info(h).bounds_checked)
    place.place_step(h, 60)
    out[f"{i}"] = evals(h, d)
    place.place_destroy(h)

# nets of many macros
d = design(64, 48, n=900)
d.is_macro = np.zeros(d.n_cells, np.uint8)
d.is_macro[:300] = 1
rng = np.random.default_rng(1)
nets = [np.arange(300), np.concatenate([np.arange(280, 900), np.arange(290, 300)])]
nets += [rng.choice(d.n_cells, k, replace=False) for k in rng.integers(2, 300, 20)]
d.net_ptr = np.concatenate([[0], np.cumsum([len(v) for v in nets])]).astype(np.int32)
d.pin_cell = np.concatenate(nets).astype(np.int32)
d.pin_dx = rng.random(d.pin_cell.size).astype(np.float32)
d.pin_dy = rng.random(d.pin_cell.size).astype(np.float32)
h = place.place_create(d, place.place_default_params(tau_stop=-1.0, autotune=0, n_copies=2))
place.place_step(h, 20)
place.place_perturb(h, place.PLACE_WIREMASK, 0.0, 0, -1)
out["wiremask"] = evals(h, d)
place.place_destroy(h)
print(json.dumps({"checked": checked, "out": out}))
"""


@pytest.mark.gpu
def test_bounds_build_agrees_on_the_gemms():
    runs = {}
    for bounds in (0, 1):
        env = dict(os.environ, HYBRO_PLACE_BOUNDS=str(bounds))
        r = subprocess.run([sys.executable, "-c", SCRIPT, ROOT], env=env, capture_output=True, text=True,
                           timeout=900)
        assert r.returncode == 0, r.stderr[-3000:]
        runs[bounds] = json.loads(r.stdout.strip().splitlines()[-1])
        assert runs[bounds]["checked"] == [bounds] * 9
    assert runs[0]["out"] == runs[1]["out"]
