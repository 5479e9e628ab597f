"""Lattices in tiles whose last few steps, and calls of few steps, run as
single-step launches (plan.h, tile_least): populations equal the storage
type's single-step kernel (one slab) bit for bit over calls of every such
length."""
import numpy as np
import pytest

import lbm_inputs as inp

pytestmark = pytest.mark.gpu

RATES = inp.s_ll(inp.rates("OPT"))


@pytest.mark.parametrize("dtype,nx,ny", [("bf16", 700, 700), ("f32", 512, 512), ("f32", 5, 3000),
                                         ("bf16", 5, 3000)])
def test_short_calls_and_rests_equal_single_steps(dtype, nx, ny):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1107_4543_gb300 import build, lbm as L

    build.build()
    L.load()
    f = inp.random_populations(nx, ny, 9, amp=1e-3)
    h = L.lbm_create(nx, ny, RATES, 1.0, (0.05, -0.02), L.DTYPES[dtype])
    s = L.lbm_slabs_create(nx, ny, RATES, 1.0, (0.05, -0.02), L.DTYPES[dtype], 1)
    try:
        L.lbm_set_populations(h, f)
        L.lbm_slabs_set_populations(s, f)
        for n in (1, 2, 3, 4, 5, 7, 9, 10, 11, 67, 130, 1):
            L.lbm_step(h, n)
            L.lbm_slabs_step(s, n)
            assert np.array_equal(L.lbm_get_populations(h),
                                  L.lbm_slabs_get_populations(s, ny, nx)), n
    finally:
        L.lbm_destroy(h)
        L.lbm_slabs_destroy(s)
