"""The plain FP64 collision's shared-reciprocal quotients (collide_f64,
k_step_f64_split) where the reciprocal is hardest to round: densities just
below a power of two (1 - 2^-53 is the largest FP64 number below one, its
significand all ones), with momenta whose products are powers of two, so that
a quotient lies next to the middle of two FP64 numbers.  One step against the
oracle bit for bit, with all rates but s_nu so small that the quotients reach
the populations unrounded."""
import numpy as np
import pytest

import lbm_inputs as inp
import oracle as orc

pytestmark = pytest.mark.gpu

TINY = 2.0 ** -300
RATES = dict(s_e=TINY, s_eps=TINY, s_q=TINY, s_nu=1.0)


def uniform(j, axes, scale):
    """Populations of density 1 - j 2^-53 (summed left to right without
    rounding), times scale: momentum 2^-4 along x and no p_xx, or along x and
    y and no p_xy, so that the quotient alone makes that moment relax."""
    f = np.zeros(9)
    if axes == 1:
        f[5] = f[8] = 2.0 ** -5
    else:
        f[1] = f[2] = 2.0 ** -4
    f[0] = (1.0 - j * 2.0 ** -53) - f[1:].sum()
    assert f.sum() == 1.0 - j * 2.0 ** -53
    return f * scale


@pytest.mark.parametrize("nx,ny", [(8, 4), (152, 70)])  # four warps per 32 nodes, and one
@pytest.mark.parametrize("scale", [1.0, 2.0 ** 9, 2.0 ** -7])
def test_quotients_by_densities_below_a_power_of_two(nx, ny, scale):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1107_4543_gb300 import lbm

    bad = []
    for j in (1, 2, 3, 5, 7, 9, 101, 1001, 4095, 8191):
        for axes in (1, 2):
            f = np.empty((9, ny, nx))
            f[:] = uniform(j, axes, scale)[:, None, None]
            h = lbm.lbm_create(nx, ny, inp.s_ll(RATES), 1.0, (0.0, 0.0), lbm.LBM_F64)
            try:
                lbm.lbm_set_populations(h, f)
                lbm.lbm_step(h, 1)
                got = lbm.lbm_get_populations(h)
            finally:
                lbm.lbm_destroy(h)
            if not np.array_equal(got, orc.run(f.copy(), inp.s_paper(RATES), 1)):
                bad.append((j, axes))
    assert not bad, bad
