"""What the kernels that take several steps per launch left untested in the
single-step path: the launch variants of the single-step kernel, and the
forcing of a point source, whose node values lattices in tiles get from the
host and single steps from a kernel.  lbm_step_plan says which path a lattice
takes."""
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


@pytest.mark.parametrize("dtype,nx,ny,single", [("f32", 700, 700, True), ("f32", 1201, 1101, False),
                                                ("f16", 1024, 1024, True),
                                                ("bf16", 1500, 1111, True),
                                                ("f64dev", 131, 70, True)])
def test_every_launch_variant_gives_the_same_populations(L, dtype, nx, ny, single):
    """Lattices planned as single steps, and one in rows stepped one by one."""
    f = inp.random_populations(nx, ny, 4, amp=1e-3)
    got = []
    for v in range(L.LBM_TUNE_VARIANTS):
        h = L.lbm_create(nx, ny, RATES, 1.0, (0.05, -0.02), L.DTYPES[dtype])
        try:
            kind, steps = L.lbm_step_plan(h)
            assert (kind == L.LBM_PLAN_SINGLE and steps == 1) if single else kind == L.LBM_PLAN_ROWS
            L.lbm_set_variant(h, v)
            L.lbm_set_populations(h, f)
            for n in ((9,) if single else (1,) * 9):
                L.lbm_step(h, n)
            assert L.lbm_get_variant(h) == v
            got.append(L.lbm_get_populations(h))
        finally:
            L.lbm_destroy(h)
    for g in got[1:]:
        assert np.array_equal(got[0], g)


def forced(L, dtype, nx, ny, x, y, patch, chunks):
    """Populations after the chunks' forced steps from rest, but for a square
    patch of given populations around the source (x, y), with the plan."""
    r = patch.shape[1] // 2
    h = L.lbm_create(nx, ny, RATES, 1.0, (0.0, 0.0), L.DTYPES[dtype])
    try:
        f = L.lbm_get_populations(h)
        f[:, y - r:y + r + 1, x - r:x + r + 1] += patch
        L.lbm_set_source(h, x, y, 0.01, 17.0)
        L.lbm_set_populations(h, f)
        plan = L.lbm_step_plan(h)[0]
        for n in chunks:
            L.lbm_step(h, n)
        return L.lbm_get_populations(h), plan
    finally:
        L.lbm_destroy(h)


@pytest.mark.parametrize("dtype", ["f32", "f16", "bf16"])
@pytest.mark.parametrize("x,y", [(140, 145), (147, 141), (150, 150), (149, 139)])
def test_forced_tiles_equal_single_forced_steps(L, dtype, x, y):
    """The same source and surroundings in a lattice in tiles and in one so
    large that its forced steps go one by one: until the disturbance has
    crossed the smaller lattice, both hold the same numbers around the source
    (bit for bit, at rest elsewhere), through replayed graphs (64 steps and
    more) and remainders."""
    r, steps = 3, 125  # reaches 128 nodes from the source
    patch = 1e-3 * np.random.default_rng(x).standard_normal((9, 2 * r + 1, 2 * r + 1))
    small, plan = forced(L, dtype, 300, 290, x, y, patch, (steps,))
    assert plan == L.LBM_PLAN_TILES
    parts, _ = forced(L, dtype, 300, 290, x, y, patch, (3, 70, 52))
    large, plan = forced(L, dtype, 1024, 1024, 512, 512, patch, (steps,))
    assert plan == L.LBM_PLAN_SINGLE
    w = 130
    a = small[:, y - w:y + w + 1, x - w:x + w + 1]
    assert np.array_equal(a, large[:, 512 - w:512 + w + 1, 512 - w:512 + w + 1])
    assert np.array_equal(small, parts)
    assert np.abs(a - large[:, :1, :1]).max() > 1e-3  # the source has acted
