"""The von Neumann kernel (section 4.1) where its QR sweeps are hardest.

Close to k = 0 the three hydrodynamic eigenvalues lie within |k| of one
another and the shift has to come from differences far smaller than the
entries: every case has to converge (lbm_vn_eigs raises otherwise) to the
eigenvalues numpy finds.  The tolerance: about 225 rotations (25 sweeps of 9)
of eps ||G||, ||G|| < 3, times an eigenvalue condition of up to 14 (numpy's
eigenvectors on these cases): 2e-12.
"""
import numpy as np
import pytest

import lbm_inputs as inp
from oracle import vn

pytestmark = pytest.mark.gpu


def match_err(a, b):
    """Largest distance between the eigenvalue multisets a and b."""
    b = list(b)
    err = 0.0
    for x in a:
        j = int(np.argmin([abs(x - y) for y in b]))
        err = max(err, abs(x - b.pop(j)))
    return err


@pytest.mark.parametrize("n", [1, 31, 33, 257])
@pytest.mark.parametrize("k_lo", [-12, -5, -2])
def test_small_wavenumbers_converge(n, k_lo):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1107_4543_gb300 import lbm

    rng = np.random.default_rng(100 * n - k_lo)
    k = 10.0 ** rng.uniform(k_lo, k_lo + 2, n)
    th = rng.choice([0.0, np.pi / 4, 0.3, 1.1], n)
    kx, ky = k * np.cos(th), k * np.sin(th)
    U = rng.choice([0.0, 0.1], n)
    V = U * rng.choice([0.0, 1.0], n)
    sets = [inp.rates(["LL", "OPT", "OPT-Z", "LL*", "OPT-B"][i % 5], nu=1e-3) for i in range(n)]
    got = lbm.lbm_vn_eigs(kx, ky, U, V, np.array([inp.s_ll(r) for r in sets]))
    worst = max(match_err(got[c], vn.eigs(kx[c], ky[c], U[c], V[c], inp.s_paper(sets[c])))
                for c in range(n))
    assert worst < 2e-12
