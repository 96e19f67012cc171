"""The sweep on 57-point grids at the ends of the FP64 range: where 2^xi is zero no pair is kept, where
every t / 2^xi vanishes all are, each worth 1."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lo,all_kept", [(-1100.0, False), (-974.0, None), (946.0, True), (1012.0, True)])
def test_range(lo, all_kept):
    import paper_2104_15124_gb300 as vb
    n = 200
    x = torch.from_numpy(np.random.default_rng(1).standard_normal((n, 3)).astype(np.float32)).cuda()
    rho = torch.ones(n, dtype=torch.float64, device="cuda")
    chi, _, _ = vb.radius_sweep(x, rho, 1.0, 0.5, (lo, lo + 14.0, 0.25))
    chi = chi.cpu().numpy()
    want = {False: 0.0, None: float(n), True: float(n * n)}[all_kept]   # None: the diagonal alone
    assert np.all(chi == want)
