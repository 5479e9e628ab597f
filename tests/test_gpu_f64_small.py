"""The plain FP64 step of small lattices, shared by four warps per 32 nodes,
against the oracle bit for bit: one node group and less, ragged ends, both
sides of the size where one warp per 32 nodes takes over (two blocks per SM:
9728 nodes on 152 SMs), and populations so large that the quotients take the
ordinary division."""
import os

import numpy as np
import pytest

import lbm_inputs as inp
import oracle as orc

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("scale", [1.0, 2.0 ** 502])
@pytest.mark.parametrize("nx,ny", [(2, 2), (5, 3), (31, 2), (2, 33), (8, 4), (33, 31), (64, 64),
                                   (97, 100), (152, 64), (139, 70)])
def test_small_lattices_bit_identical(nx, ny, scale):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1107_4543_gb300 import lbm

    orc.set_threads(os.cpu_count() or 1)
    r = inp.rates("OPT")
    rng = np.random.default_rng(nx * 1000 + ny)
    x = np.arange(nx) * 2 * np.pi / nx
    f = orc.init_eq(1.0 + 1e-3 * np.cos(x)[None, :] * np.ones((ny, 1)), np.full((ny, nx), 0.1),
                    np.zeros((ny, nx)))
    f = f * (1.0 + 1e-4 * rng.standard_normal(f.shape)) * scale
    h = lbm.lbm_create(nx, ny, inp.s_ll(r), 1.0, (0.0, 0.0), lbm.LBM_F64)
    try:
        lbm.lbm_set_populations(h, f)
        lbm.lbm_step(h, 131)
        got = lbm.lbm_get_populations(h)
    finally:
        lbm.lbm_destroy(h)
    assert np.array_equal(got, orc.run(f.copy(), inp.s_paper(r), 131))
