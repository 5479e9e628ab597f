"""Batches whose resident members are of both kinds, those of which two share
an SM and those a few nodes larger, which take a launch of their own beside
the others' (csrc/resident.cuh): every member equals its standalone run bit
for bit, over calls of odd and even length."""
import numpy as np
import pytest

import lbm_inputs as inp

pytestmark = pytest.mark.gpu

RATES = inp.s_ll(inp.rates("OPT"))
# both sides of 3208 (FP32) and 6421 (16 bits) nodes, the largest resident
# ones (3228, 6456), small ones, and one that is not resident
PAIRS = [("f32", 8, 401), ("f32", 20, 20), ("f16", 6, 1070), ("bf16", 33, 31)]
ALONE = [("f32", 46, 70), ("f32", 12, 269), ("f16", 92, 70), ("bf16", 12, 538)]
OTHER = [("f32", 70, 60)]
# FP32 members stepped one node per thread (up to 384 nodes), and the next size
TINY = [("f32", 2, 2), ("f32", 3, 3), ("f32", 2, 31), ("f32", 33, 2), ("f32", 11, 11),
        ("f32", 8, 16), ("f32", 43, 3), ("f32", 24, 16), ("f32", 35, 11)]


@pytest.mark.parametrize("members", [PAIRS + ALONE + OTHER, ALONE, PAIRS, TINY])
def test_both_kinds_of_resident_members_equal_alone(members):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1107_4543_gb300 import build, lbm as L

    build.build()
    L.load()
    hs, b, want = [], None, []
    try:
        for dt, nx, ny in members:
            f = inp.gaussian_pulse(nx, ny, 1e-3, 3.0, xc=1.0, yc=ny - 2.0)
            h = L.lbm_create(nx, ny, RATES, 1.0, (0.0, 0.0), L.DTYPES[dt])
            g = L.lbm_create(nx, ny, RATES, 1.0, (0.0, 0.0), L.DTYPES[dt])
            L.lbm_init_field(h, *f)
            L.lbm_init_field(g, *f)
            L.lbm_step(g, 104)
            want.append(L.lbm_get_populations(g))
            L.lbm_destroy(g)
            hs.append(h)
        b = L.lbm_batch_create(hs)
        assert list(L.lbm_batch_resident(b)) == [m not in OTHER for m in members]
        for n in (37, 1, 64, 2):
            L.lbm_batch_step(b, n)
        got = [L.lbm_get_populations(h) for h in hs]
    finally:
        if b is not None:
            L.lbm_batch_destroy(b)
        for h in hs:
            L.lbm_destroy(h)
    for m, g, w in zip(members, got, want):
        assert np.array_equal(g, w), m
