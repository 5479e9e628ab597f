"""GPU checks of the kernels that advance several steps per launch
(csrc/step_multi.cuh) against the single-step kernel: the same arithmetic
with the same storage rounding between steps, so populations are equal bit
for bit, at sizes where tiles, strips and the periodic wrap can go wrong."""
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


RATES = inp.s_ll(inp.rates("OPT"))


def noisy(nx, ny, seed):
    """Random populations: every direction of every node differs."""
    return inp.random_populations(nx, ny, seed, amp=1e-3)


# one row, one column, around a pair, a chunk, a tile (44 .. 60 columns) and
# several tiles; the storage type's single-step kernel runs in one slab
TILE_SIZES = [(2, 2), (3, 2), (5, 3), (8, 2), (9, 7), (44, 5), (45, 40), (59, 8), (64, 64),
              (65, 97), (101, 101), (131, 23), (512, 16), (300, 290)]


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("nx,ny", TILE_SIZES)
def test_tiles_equal_single_steps(L, nx, ny, dtype):
    f = noisy(nx, ny, 3)
    for steps in (1, 5, 67, 131):
        h = L.lbm_create(nx, ny, RATES, 1.0, (0.05, -0.02), L.DTYPES[dtype])
        s = L.lbm_slabs_create(nx, ny, RATES, 1.0, (0.05, -0.02), L.DTYPES[dtype], 1)
        try:
            L.lbm_set_populations(h, f)
            L.lbm_slabs_set_populations(s, f)
            L.lbm_step(h, steps)
            L.lbm_slabs_step(s, steps)
            assert np.array_equal(L.lbm_get_populations(h), L.lbm_slabs_get_populations(s, ny, nx))
        finally:
            L.lbm_destroy(h)
            L.lbm_slabs_destroy(s)


# lattices that take the rows kernel (tests/native/plan_check.cu checks that
# they do): whole rows, a partial last chunk of every kind, few rows
ROW_SIZES = [("f32", nx, ny) for nx, ny in [(1200, 1101), (1201, 1101), (1202, 1101), (1203, 1101),
                                            (700001, 2), (420003, 3)]]
ROW_SIZES += [("f16", 2496 + k, 2101) for k in range(8)] + [("bf16", 2501, 2101)]


@pytest.mark.parametrize("dtype,nx,ny", ROW_SIZES)
def test_rows_equal_single_steps(L, dtype, nx, ny):
    f = noisy(nx, ny, 5)
    h = L.lbm_create(nx, ny, RATES, 1.0, (0.05, -0.02), L.DTYPES[dtype])
    g = L.lbm_create(nx, ny, RATES, 1.0, (0.05, -0.02), L.DTYPES[dtype])
    try:
        for x in (h, g):
            L.lbm_set_variant(x, 2)
            L.lbm_set_populations(x, f)
        for steps in (3, 7, 2, 4):
            L.lbm_step(h, steps)
            for _ in range(steps):
                L.lbm_step(g, 1)  # the single-step kernel
        a = L.lbm_get_populations(h)
        assert np.array_equal(a, L.lbm_get_populations(g))
    finally:
        L.lbm_destroy(h)
        L.lbm_destroy(g)


@pytest.mark.parametrize("dtype", ["f32", "f16", "bf16"])
def test_forced_tiles_follow_the_single_forced_steps(L, dtype):
    """A point source inside the tiles' halos: runs of many steps equal runs
    of one step at a time, across replays and remainders."""
    nx, ny = 53, 31
    got = []
    for chunks in ((140,), (1,) * 140, (3, 70, 67)):
        h = L.lbm_create(nx, ny, RATES, 1.0, (0.0, 0.0), L.DTYPES[dtype])
        try:
            L.lbm_set_source(h, 52, 0, 0.01, 17.0)
            L.lbm_init_field(h, *inp.gaussian_pulse(nx, ny, 1e-3, 4.0))
            for n in chunks:
                L.lbm_step(h, n)
            got.append(L.lbm_get_populations(h))
        finally:
            L.lbm_destroy(h)
    assert np.array_equal(got[0], got[1]) and np.array_equal(got[0], got[2])


@pytest.mark.parametrize("u0", [(0.0, 0.0), (0.125, -0.0625)])
@pytest.mark.parametrize("amp", [0.0, 1e-9, 1e-3, 0.3])
def test_init_rounds_the_fp64_deviations_once(L, amp, u0):
    """The FP32 init (float-float combinations of FP64 differences) stores
    the FP64 deviations of LBM_F64DEV rounded once: within 2^-24 of each,
    plus the roundings of adding the base, which a lattice holds after its
    creation (u0 exact in FP32, so both types have the same one).  The FP32
    moments are then those sums' errors away from the fields."""
    nx, ny = 61, 37
    rng = np.random.default_rng(7)
    rho = 1.0 + amp * rng.uniform(-1, 1, (ny, nx))
    ux = u0[0] + amp * rng.uniform(-1, 1, (ny, nx))
    uy = u0[1] + amp * rng.uniform(-1, 1, (ny, nx))
    h = L.lbm_create(nx, ny, RATES, 1.0, u0, L.LBM_F32DEV)
    d = L.lbm_create(nx, ny, RATES, 1.0, u0, L.LBM_F64DEV)
    try:
        base = L.lbm_get_populations(d)
        for x in (h, d):
            L.lbm_init_field(x, rho, ux, uy)
        want = L.lbm_get_populations(d)
        err = 2.0 ** -24 * np.abs(want - base)
        assert np.all(np.abs(L.lbm_get_populations(h) - want) <= err + 2.0 ** -51)
        r, u, v = L.lbm_moments(h)
        e = err.sum(axis=0) + 2.0 ** -47
        assert np.all(np.abs(r - rho) <= e)
        assert np.all(np.abs(u - ux) <= (1 + np.abs(ux)) * e / rho)
        assert np.all(np.abs(v - uy) <= (1 + np.abs(uy)) * e / rho)
    finally:
        L.lbm_destroy(h)
        L.lbm_destroy(d)


# members whose groups take three steps per launch in FP32 and FP16 (one large
# member each, and narrow ones around a chunk, three chunks and a warp); the
# BF16 pair steps one by one, one member is resident
BATCH = [("f32", 2000, 1001), ("f32", 9, 3001), ("f32", 10, 3001), ("f32", 11, 3001),
         ("f32", 109, 901), ("f32", 119, 903), ("f32", 121, 905), ("f32", 333, 1201),
         ("f32", 20, 20), ("f16", 2600, 2103), ("f16", 17, 4001), ("f16", 22, 3001),
         ("f16", 239, 501), ("f16", 241, 503), ("bf16", 130, 90), ("bf16", 61, 200)]


def alone(L, dtype, nx, ny, f, steps):
    h = L.lbm_create(nx, ny, RATES, 1.0, (0.0, 0.0), L.DTYPES[dtype])
    try:
        L.lbm_init_field(h, *f)
        L.lbm_step(h, steps)
        return L.lbm_get_populations(h), L.lbm_moments(h)
    finally:
        L.lbm_destroy(h)


def test_batch_rows_equal_alone(L):
    """Groups of three-step launches, of single steps and a resident member
    in one batch, from either buffer and over calls of every remainder."""
    fields = [inp.gaussian_pulse(nx, ny, 1e-3, 5.0, xc=3.0, yc=ny - 2.0) for _, nx, ny in BATCH]
    hs, b = [], None
    try:
        for (dt, nx, ny), f in zip(BATCH, fields):
            h = L.lbm_create(nx, ny, RATES, 1.0, (0.0, 0.0), L.DTYPES[dt])
            L.lbm_init_field(h, *f)
            hs.append(h)
        L.lbm_step(hs[1], 1)  # one member starts on its other buffer
        b = L.lbm_batch_create(hs)
        for n in (1, 2, 3, 7, 69):
            L.lbm_batch_step(b, n)
        got = [L.lbm_get_populations(h) for h in hs]
    finally:
        if b is not None:
            L.lbm_batch_destroy(b)
        for h in hs:
            L.lbm_destroy(h)
    for k, ((dt, nx, ny), f) in enumerate(zip(BATCH, fields)):
        want, _ = alone(L, dt, nx, ny, f, 82 + (k == 1))
        assert np.array_equal(got[k], want), (k, dt, nx, ny)


def test_served_generations_of_rows_equal_alone(L):
    """A server's ragged generations: members stop after step counts of every
    remainder, some inside a generation's last three-step launch."""
    import time

    steps = [5, 22, 23, 24, 9, 11, 31, 3, 1, 12, 10, 2, 33, 32, 7, 4]
    fields = [inp.gaussian_pulse(nx, ny, 1e-3, 5.0, xc=2.0, yc=1.0) for _, nx, ny in BATCH]
    s = L.lbm_server_create(2 ** 33, 11)
    try:
        ids, keep = [], []
        for (dt, nx, ny), f, n in zip(BATCH, fields, steps):
            req, kept = L.make_request(nx, ny, RATES, n, dtype=dt, init_kind=L.LBM_INIT_FIELDS,
                                       fields=f)
            keep.append(kept)
            ids.append(L.lbm_submit(s, req))
        got, t0 = {}, time.time()
        while len(got) < len(ids) and time.time() - t0 < 120:
            for k, rid in enumerate(ids):
                if k not in got:
                    rc, *out = L.lbm_poll(s, rid, BATCH[k][1], BATCH[k][2])
                    if rc == L.LBM_OK:
                        got[k] = out[:3]
            time.sleep(0.01)
    finally:
        L.lbm_server_destroy(s)
    assert len(got) == len(ids)
    for k, ((dt, nx, ny), f) in enumerate(zip(BATCH, fields)):
        _, want = alone(L, dt, nx, ny, f, steps[k])
        for a, w in zip(got[k], want):
            assert np.array_equal(a, w), (k, dt, nx, ny)
