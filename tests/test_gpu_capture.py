"""lbm_step on a stream that its owner captures into a graph: a call of an
even number of steps leaves the buffers as it found them, so that every replay
advances the lattice by as many steps, whatever the plan of uncaptured calls;
and a forced call reads nothing from the host once it has returned."""
import numpy as np
import pytest

import lbm_inputs as inp

pytestmark = pytest.mark.gpu

RATES = inp.s_ll(inp.rates("OPT"))


@pytest.fixture(scope="module")
def L():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1107_4543_gb300 import build, lbm

    build.build()
    lbm.load()
    return lbm


def lattice(L, nx, ny, dtype, source):
    h = L.lbm_create(nx, ny, RATES, 1.0, (0.0, 0.0), L.DTYPES[dtype])
    L.lbm_init_analytic(h, L.LBM_INIT_GAUSSIAN, (1e-3, 4.0, nx / 3.0, ny / 2.0))
    if source:
        L.lbm_set_source(h, nx // 2, ny // 3, 1e-4, 20.0)
    return h


@pytest.mark.parametrize("nx,ny,dtype,plan,source", [
    (101, 101, "f32", "TILES", False), (101, 101, "f32", "TILES", True),
    (512, 16, "f16", "TILES", False), (1203, 1101, "f32", "ROWS", False),
    (1024, 1024, "f16", "SINGLE", False), (64, 64, "f64", "SINGLE", True)])
@pytest.mark.parametrize("n", [2, 4, 6, 70])
def test_captured_calls_replay(L, nx, ny, dtype, plan, source, n):
    import torch

    replays = 1 if source else 3
    if plan == "SINGLE" and n >= 64:
        pytest.skip("64 single steps replay a graph of their own")
    want = lattice(L, nx, ny, dtype, source)
    L.lbm_step(want, n * replays)
    h = lattice(L, nx, ny, dtype, source)
    assert L.lbm_step_plan(h)[0] == getattr(L, "LBM_PLAN_" + plan)
    if plan != "TILES":  # tuning, if any, before the capture
        L.lbm_step(h, 1)
        L.lbm_init_analytic(h, L.LBM_INIT_GAUSSIAN, (1e-3, 4.0, nx / 3.0, ny / 2.0))
    st = torch.cuda.Stream()
    L.lbm_set_stream(h, st)
    a, b = torch.ones(1024, device="cuda"), torch.zeros(1024, device="cuda")
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=st):
        b.copy_(a)  # something other than a step before the first one
        L.lbm_step(h, n)
    with torch.cuda.stream(st):
        for _ in range(replays):
            g.replay()
    torch.cuda.synchronize()
    assert np.array_equal(L.lbm_get_populations(h), L.lbm_get_populations(want))
    L.lbm_set_stream(h, None)
    del g
    for x in (h, want):
        L.lbm_destroy(x)
