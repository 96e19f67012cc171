"""The delta_tol sweep on the standard grid takes every unordered pair once and squares kernel values down
the octaves: its sums equal the oracle's to the rounding of FP64 sums, at tile edges too.  Tolerance:
a term is within 16 ulp (an exp, up to three squarings), the sums of up to 10^6 positive terms
within 10^6 ulp at worst, so 1e-9 is far outside what rounding can do and far inside one lost or extra pair
of the smaller clouds (1 / n^2)."""
import numpy as np
import pytest
import torch

from oracle import method as M
from oracle import radius as R

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,m", [(2, 1), (63, 2), (64, 3), (65, 2), (128, 4), (129, 9), (1000, 3)])
@pytest.mark.parametrize("scale,tol", [(1.0, 0.01), (4.0, 0.3), (1e-4, 0.001)])
def test_sweep_sums(n, m, scale, tol):
    import paper_2104_15124_gb300 as vb
    r = np.random.default_rng(n + m)
    x = r.uniform(-1.0, 1.0, (n, m)).astype(np.float32)
    x[-1] = x[0]                                  # a duplicate: t = 0 off the diagonal
    rho = r.uniform(0.05, 2.0, n)
    ref = R.radius_sweep(x, rho, scale, M.xi_grid(), tol)
    chi, _, _ = vb.radius_sweep(torch.from_numpy(x).cuda(), torch.from_numpy(rho).cuda(), scale, tol)
    np.testing.assert_allclose(chi.cpu().numpy(), ref, rtol=1e-9)
