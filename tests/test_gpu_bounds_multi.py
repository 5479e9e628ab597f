"""The debug build's index checks (tests/test_gpu_bounds.py) over the kernels
that take several steps per launch: rows and tiles of single lattices, whole
and ragged, with a point source too; rows of batches; resident members of
both kinds, their smallest and largest; and the single-step kernels in every
launch variant, which calls of one step reach.  The checks redirect what they
find, and the word must stay zero."""
import json
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SCRIPT = r'''
import json, sys
sys.path.insert(0, ROOT)
import lbm_inputs as inp
from paper_1107_4543_gb300 import build, lbm as L
L.load(build.build(debug=True))
L.lbm_debug_bounds(reset=True)
S = inp.s_ll(inp.rates("OPT"))
T = {"f32": L.LBM_F32DEV, "f16": L.LBM_F16DEV, "bf16": L.LBM_BF16DEV}
out = {"rows": 0, "tiles": 0}
def lattice(nx, ny, t):
    h = L.lbm_create(nx, ny, S, 1.0, (0.05, -0.02), T[t])
    L.lbm_init_analytic(h, L.LBM_INIT_GAUSSIAN, (1e-3, 4.0, nx / 2.0, ny / 2.0))
    return h
for nx, ny, t, kind in ((1203, 1101, "f32", "rows"), (4098, 3001, "f16", "rows"),
                        (4097, 3001, "bf16", "rows"), (3, 2, "f32", "tiles"),
                        (101, 101, "f32", "tiles"), (512, 16, "f16", "tiles"),
                        (5, 3000, "f32", "tiles"), (333, 257, "bf16", "tiles")):
    h = lattice(nx, ny, t)
    assert L.lbm_step_plan(h)[0] == (L.LBM_PLAN_ROWS if kind == "rows" else L.LBM_PLAN_TILES), (nx, ny)
    for n in (1, 2, 3, 5, 71):
        L.lbm_step(h, n)
    if kind == "tiles":
        L.lbm_set_source(h, nx - 1, ny // 2, 1e-3, 20.0)
        for n in (1, 4, 71):
            L.lbm_step(h, n)
    L.lbm_destroy(h)
    out[kind] |= L.lbm_debug_bounds()
for t, sizes in (("f32", ((8, 4000), (1997, 1613), (1301, 9), (16, 24), (3, 3), (46, 70), (56, 56))),
                 ("f16", ((9, 4001), (2000, 1500), (1999, 1501), (80, 80), (5, 5))),
                 ("bf16", ((9, 4001), (2000, 1500), (1999, 1501), (80, 80), (5, 5)))):
    hs = [lattice(nx, ny, t) for nx, ny in sizes]
    b = L.lbm_batch_create(hs)
    assert L.lbm_batch_plan(b, T[t])[0] == L.LBM_PLAN_ROWS, t
    for n in (3, 1, 2, 73):
        L.lbm_batch_step(b, n)
    for v in range(L.LBM_BATCH_TUNE_VARIANTS):
        L.lbm_batch_set_variant(b, v)
        for n in (1, 1, 1):
            L.lbm_batch_step(b, n)
    L.lbm_batch_drift(b, len(hs))
    L.lbm_batch_destroy(b)
    for h in hs:
        L.lbm_destroy(h)
    out["batch_" + t] = L.lbm_debug_bounds()
print("BOUNDS " + json.dumps(out))
'''


def test_index_checks_of_several_steps_per_launch_stay_clean():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1107_4543_gb300 import build

    build.build(debug=True)
    r = subprocess.run([sys.executable, "-c", SCRIPT.replace("ROOT", repr(ROOT), 1)],
                       capture_output=True, text=True, timeout=900)
    assert r.returncode == 0, r.stdout[-2000:] + r.stderr[-2000:]
    res = json.loads([x for x in r.stdout.splitlines() if x.startswith("BOUNDS ")][-1][7:])
    assert sorted(res) == ["batch_bf16", "batch_f16", "batch_f32", "rows", "tiles"]
    assert all(v == 0 for v in res.values()), res
