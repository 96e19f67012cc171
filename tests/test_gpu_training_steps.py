"""Gradients of the radius network at the edges of the training kernel's sample blocks (32 samples) and
input widths, against the FP64 chain rule.  Tolerance: FP32 sums of n terms and of 64-wide dot
products, about sqrt(n) 2^-24 of the terms' magnitude (1e-5 at n = 1,000); 1e-3 of the gradient's norm
allows for its cancellation."""
import numpy as np
import pytest
import torch

from oracle import mlp as OM

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 31, 32, 33, 1000, 4897])
@pytest.mark.parametrize("m", [1, 4, 7, 16])
def test_gradient(n, m):
    import paper_2104_15124_gb300 as vb
    r = np.random.default_rng(100 * m + n)
    x = r.standard_normal((n, m + 2)).astype(np.float32)       # rows longer than the network's inputs
    y = (r.standard_normal(n) * 0.3 - 2.0).astype(np.float32)
    net = vb.Mlp(m, seed=7)
    net.set_standardisation(np.full(m, 0.1), np.full(m, 1.1), -2.0, 0.3)
    g, loss = net.gradient(torch.from_numpy(x).cuda(), torch.from_numpy(y).cuda())
    theta = net.bf16_weights().cpu().numpy().astype(np.float64)
    Xs = (x[:, :m].astype(np.float64) - np.float32(0.1)) / np.float32(1.1)
    ref_loss, ref_g = OM.loss_and_grad(theta, Xs, (y.astype(np.float64) + 2.0) / np.float32(0.3))
    assert abs(loss.item() - ref_loss) <= 1e-4 * ref_loss
    assert np.linalg.norm(g.cpu().numpy() - ref_g) <= 1e-3 * np.linalg.norm(ref_g)


def test_epoch_follows_its_gradients():
    # one minibatch per epoch: a first Adam step from zero moments moves every weight by lr g / (|g| + eps)
    import paper_2104_15124_gb300 as vb
    r = np.random.default_rng(3)
    x = torch.from_numpy(r.standard_normal((333, 3)).astype(np.float32)).cuda()
    y = torch.from_numpy(r.standard_normal(333).astype(np.float32)).cuda()
    net = vb.Mlp(3, seed=5)
    w0 = net.master.clone()
    g, loss = net.gradient(x, y)
    l2 = net.train_epoch(x, y, batch=512, lr=1e-2)
    step = -1e-2 * g / (g.abs() + 1e-8)
    assert torch.equal(loss, l2)
    assert torch.allclose(net.master - w0, step, rtol=1e-3, atol=1e-6)
