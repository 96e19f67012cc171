"""Gradient sums over many samples: n equal samples, whose mean gradient is the gradient of one.  With n
a power of two each sample's share is exactly 1 / n of it, so what is left is the sum: a block adds 128
samples, then these sums, of which it has at most n / (152 * 128) + 1, and the blocks' sums are added in
FP64.  The relative error is below (128 + n / 19456 + 2) 2^-24."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1 << 12, 1 << 21])
@pytest.mark.parametrize("m", [4, 16])
def test_equal_samples(n, m):
    import paper_2104_15124_gb300 as vb
    r = np.random.default_rng(m)
    x = torch.from_numpy(r.standard_normal((1, m)).astype(np.float32)).cuda()
    y = torch.full((1,), 0.7, dtype=torch.float32, device="cuda")
    net = vb.Mlp(m, seed=9)
    one, loss1 = net.gradient(x, y)
    g, loss = net.gradient(x.expand(n, m).contiguous(), y.expand(n).contiguous())
    bound = (128 + n / 19456 + 2) * 2.0 ** -24
    one, g = one.cpu().numpy().astype(np.float64), g.cpu().numpy().astype(np.float64)
    assert np.all(np.abs(g - one) <= bound * np.abs(one) + 1e-30)
    assert abs(loss.item() - loss1.item()) <= bound * loss1.item()
