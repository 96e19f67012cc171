"""The bandwidth at the edges of its 128-row, 16-column chunks: the rank-order sum, bit for bit."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 7, 127, 128, 129, 1000])
@pytest.mark.parametrize("k,k_bw", [(1, 1), (15, 15), (16, 16), (17, 17), (33, 20), (64, 64), (130, 129)])
def test_rank_order_sum(n, k, k_bw):
    import paper_2104_15124_gb300 as vb
    d2 = np.sort(np.random.default_rng(n * 1000 + k).random((n, k)) + 1e-3, axis=1)
    s = d2[:, 0].copy()
    for r in range(1, k_bw):
        s = s + d2[:, r]
    b = vb.bandwidth(torch.from_numpy(d2).cuda(), k_bw)
    torch.cuda.synchronize()
    assert np.array_equal(b.cpu().numpy(), np.sqrt(s))
