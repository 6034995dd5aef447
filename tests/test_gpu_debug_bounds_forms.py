"""The index-checked build over every form of the step: each case forces one (environment) and asserts that it is
the one that runs, so that a change of the dispatch cannot empty the test.  Cut tiles, lattices narrower than
the halo, single planes, slabs of one plane, chunks of one row; no access outside, and the bits of the
ordinary build (the binary march: its rounding, eight float32 roundings a step, since the compiler fuses its
packed multiplications and additions as the code around them allows)."""
import json
import os
import subprocess
import sys

import numpy as np
import pytest

from tests.helpers import drop_populations, library, make_ctx, oracle_model

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
F, E = "forcing", "equilibrium"
FORCED = ("LB_D3_FIELD", "LB_D3_VARIANT", "LB_D2_VARIANT", "LB_D2_ROWS", "LB_F64_SLAB", "LB_WIDE", "LB_B3_MARCH")
# lattice, scheme, shape, storage, environment, part of the form's name
CASES = (
    # D3Q19 forcing, 32-bit arithmetic: fused pairs, fused one-site kernel, density field
    [("D3Q19", F, s, st, {"LB_D3_FIELD": "0"}, form) for s, st, form in (
        ((68, 20, 12), 2, "pairs 32x8"), ((64, 16, 9), 2, "interleaved"), ((2, 3, 3), 2, "pairs 32x8"),
        ((38, 13, 11), 1, "pairs 32x8"), ((38, 13, 11), 3, "pairs 32x8"), ((96, 20, 7), 3, "interleaved"),
        ((37, 13, 11), 1, "tile, one site"), ((37, 13, 11), 2, "tile, one site"), ((1, 2, 3), 3, "tile, one site"))]
    + [("D3Q19", F, s, st, {"LB_D3_FIELD": "1"}, form) for s, st, form in (
        ((68, 20, 12), 1, "pairs 32x8, density field"), ((64, 16, 9), 2, "density field, interleaved"),
        ((2, 3, 3), 3, "pairs 32x8, density field"), ((37, 13, 11), 1, "density field, one site"),
        ((33, 5, 9), 2, "density field, one site"), ((1, 1, 1), 2, "density field, one site"), ((3, 9, 1), 3, "density field, one site"))]
    + [("D3Q19", sc, (38, 13, 11), st, {"LB_D3_VARIANT": "0"}, "tile, two sites") for sc in (F, E) for st in (1, 2)]
    # D3Q19 float64: fused, whole lattice, slabs
    + [("D3Q19", sc, s, 0, {} if n is None else {"LB_F64_SLAB": n}, "tile" if n == "0" else "passes")
       for sc in (F, E) for s in ((22, 20, 18), (5, 2, 4), (1, 1, 1)) for n in (None, "0", "1", "3")]
    # D3Q19 equilibrium tiles
    + [("D3Q19", E, s, st, {"LB_WIDE": w}, "64x4" if w == "1" else "32x8")
       for w in "01" for s, st in (((38, 13, 11), 1), ((38, 13, 11), 2), ((64, 16, 9), 3), ((130, 10, 5), 2), ((2, 3, 3), 1))]
    + [("D3Q19", E, (37, 13, 11), st, {}, "tile, one site") for st in (1, 2)]
    # D2Q9: tiles, pairs, marching strips
    + [("D2Q9", sc, s, st, {"LB_D2_VARIANT": "0"}, "tile") for sc in (F, E) for s, st in (((46, 37), 2), ((45, 37), 1))]
    + [("D2Q9", sc, s, st, {"LB_D2_ROWS": "0"}, "pairs") for sc in (F, E) for s, st in (((46, 37), 2), ((45, 37), 3), ((2, 5), 1))]
    + [("D2Q9", E, s, st, {"LB_D2_ROWS": n}, "marching")
       for n in "18" for s, st in (((60, 12), 2), ((62, 13), 3), ((2, 5), 2), ((178, 9), 2))]
    + [("D2Q9", sc, s, 0, {}, "tile") for sc in (F, E) for s in ((66, 20), (230, 220), (3, 2))]
    # binary D3Q19 float32, marching
    + [("binary", sc, s, 1, {"LB_B3_MARCH": "1"}, "") for sc in (F, E) for s in ((34, 10, 9), (33, 9, 8), (2, 3, 3), (1, 1, 1))])
STEPS = 5


def run_cases():
    lb = library()
    out, saved = {}, {k: os.environ.pop(k, None) for k in FORCED}
    try:
        for n, (lat, scheme, shape, storage, env, form) in enumerate(CASES):
            os.environ.update(env)
            if lat == "binary":
                rng = np.random.default_rng(n)
                with lb.BinaryContext(shape, -0.04, 0.04, 0.08, 0.7, 0.8, 0.9, scheme=lb.FORCING if scheme == F else lb.EQUILIBRIUM,
                                      storage=lb.F32) as c:
                    c.init_fields(1 + 0.01 * rng.uniform(-1, 1, c.shape), rng.uniform(-1, 1, c.shape))
                    c.step(STEPS)
                    out[f"case{n}"] = np.stack(c.get_populations())
            else:
                f0 = drop_populations(oracle_model(lat, scheme), shape, 0.3 * max(shape), perturb=1e-3, seed=6)
                with make_ctx(lb, lat, scheme, shape, storage=storage) as ctx:
                    assert form in ctx.kernel_info()["form"], (CASES[n], ctx.kernel_info())
                    ctx.set_populations(f0)
                    ctx.step(STEPS)
                    out[f"case{n}"] = ctx.get_populations()
            for k in env:
                del os.environ[k]
    finally:
        os.environ.update({k: v for k, v in saved.items() if v is not None})
    return out


CHILD = """
import json, sys
import numpy as np
sys.path.insert(0, {root!r})
from tests import test_gpu_debug_bounds_forms as T
from paper_0710_5470_gb300 import lb
out = T.run_cases()
np.savez({npz!r}, **out)
print(json.dumps(lb.debug_bounds()))
"""


def test_every_form_stays_in_bounds_and_matches(tmp_path):
    from paper_0710_5470_gb300 import build
    npz = str(tmp_path / "checked.npz")
    r = subprocess.run([sys.executable, "-c", CHILD.format(root=ROOT, npz=npz)], cwd=ROOT,
                       env=dict(os.environ, LB_LIBRARY=build.build(debug=True)), capture_output=True, text=True, timeout=900)
    assert r.returncode == 0, r.stderr[-3000:]
    checked, violation = json.loads(r.stdout.strip().splitlines()[-1])
    assert checked is True
    assert violation == 0, hex(violation)
    got, want = np.load(npz), run_cases()
    assert len(want) == len(CASES)
    for n, case in enumerate(CASES):
        a, b = got[f"case{n}"], want[f"case{n}"]
        if case[0] == "binary":
            assert np.abs(a - b).max() <= STEPS * 8 * 2.0 ** -24 * np.abs(b).max(), case
        else:
            assert np.array_equal(a, b, equal_nan=True), case
