"""Moments of the 32- and 16-bit deviation types: rho = rho0 + the FP64 sum of
the stored deviations from left to right, likewise j, and u = j (1 / rho) with
the correctly rounded reciprocal, bit for bit -- for deviations of one size,
of sizes too far apart for a sum in fewer bits, for zeros, subnormals, values
whose FP32 sum overflows, and infinities (a lattice that has diverged)."""
import numpy as np
import pytest

import lbm_inputs as inp

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def L():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1107_4543_gb300 import build, lbm

    build.build()
    lbm.load()
    return lbm


def spread(kind, shape, rng):
    """Deviations (9, ny, nx) of the given kind."""
    sign = rng.choice([-1.0, 1.0], shape)
    if kind == "even":
        return 1e-3 * rng.standard_normal(shape)
    if kind == "tiny":  # a density of one to the last bits
        return 1e-16 * rng.standard_normal(shape)
    if kind == "mixed":  # 2^-60 .. 1, a fifth of them zero
        return sign * 2.0 ** rng.uniform(-60, 0, shape) * (rng.uniform(size=shape) < 0.8)
    if kind == "cancel":  # large values that cancel but for small ones
        d = 2.0 ** rng.uniform(-24, -10, shape)
        d[2] = 0.3 * sign[0]
        d[4] = -d[2] + 2.0 ** -30 * sign[1]
        return d
    if kind == "subnormal":
        return sign * 2.0 ** rng.uniform(-149, -100, shape)
    if kind == "huge":  # FP32 sums overflow, FP64 ones do not
        return sign * 3.0e38 * rng.uniform(0.5, 1.0, shape)
    d = 1e-3 * rng.standard_normal(shape)  # infinite: some populations past FP32's range
    d[rng.uniform(size=shape) < 0.02] = 1e300
    d[rng.uniform(size=shape) < 0.02] = -1e300
    return d


def stored(L, dtype, d, scale):
    """The deviations as the storage type holds them, in FP64."""
    import torch

    with np.errstate(over="ignore"):
        v = torch.from_numpy((d * scale).astype(np.float32))
    v = v if dtype == "f32" else v.to({"f16": torch.float16, "bf16": torch.bfloat16}[dtype])
    return v.to(torch.float64).numpy() / scale


@pytest.mark.parametrize("u0", [(0.0, 0.0), (0.125, -0.0625)])
@pytest.mark.parametrize("kind", ["even", "tiny", "mixed", "cancel", "subnormal", "huge", "infinite"])
@pytest.mark.parametrize("dtype", ["f32", "bf16", "f16"])
def test_moments_equal_the_fp64_sums(L, dtype, kind, u0):
    nx, ny = 67, 41
    rng = np.random.default_rng(11)
    args = (nx, ny, inp.s_ll(inp.rates("OPT")), 1.0, u0)
    e = L.lbm_create(*args, L.LBM_F64DEV)  # its populations are the base (u0 exact in FP32)
    h = L.lbm_create(*args, L.DTYPES[dtype])
    try:
        base = L.lbm_get_populations(e)
        f = base + spread(kind, (9, ny, nx), rng)
        L.lbm_set_populations(h, f)
        d = stored(L, dtype, f - base, L.lbm_info(h)["qscale"])
        got = L.lbm_moments(h)
    finally:
        L.lbm_destroy(h)
        L.lbm_destroy(e)
    with np.errstate(all="ignore"):
        r = 1.0 + (((((((d[0] + d[1]) + d[2]) + d[3]) + d[4]) + d[5]) + d[6]) + d[7] + d[8])
        jx = u0[0] + (d[1] - d[3] + d[5] - d[6] - d[7] + d[8])
        jy = u0[1] + (d[2] - d[4] + d[5] + d[6] - d[7] - d[8])
        inv = 1.0 / r
        want = (r, jx * inv, jy * inv)
    if kind == "huge" and dtype != "f16":
        assert np.isfinite(r).all() and np.abs(r).max() > 3.5e38
    if kind == "infinite":
        assert np.isinf(r).any()
    for g, w in zip(got, want):
        assert np.array_equal(g, w, equal_nan=True), (np.abs(g - w).max(), (g != w).sum())
