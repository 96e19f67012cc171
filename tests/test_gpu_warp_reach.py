"""Large clouds in which a query reaches most tiles go on to the tiled search, others do not; the lists are
the full-key tiled search's bit for bit either way."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("what", ["plain", "radius", "batch", "near"])
def test_reach(what):
    import paper_2104_15124_gb300 as vb
    n, m, k = 100000, 3 if what == "near" else 8, 24
    if what == "batch":
        n = 2 * 60001
    x = torch.from_numpy(np.random.default_rng(8).standard_normal((n, m)).astype(np.float32)).cuda()
    halves = [x[: n // 2], x[n // 2:]] if what == "batch" else [x]
    ref = [vb.knn(h, k, heap_keys="full") for h in halves]
    nbr = torch.cat([r[0] + i * (n // 2) for i, r in enumerate(ref)])
    d2 = torch.cat([r[1] for r in ref])
    vb.report_reset()
    if what == "batch":
        out = vb.Builder(n, m, k, d=m, c=1.0, cloud_ptr=[0, n // 2, n])(x)
        got = out.nbr, out.nbr_d2
    elif what == "radius":
        got = vb.knn(x, k, radius=d2[:, -1].sqrt().float(), inflate=1.1)
    else:
        got = vb.knn(x, k)
    torch.cuda.synchronize()
    rep = vb.raise_on_device_error()
    assert torch.equal(got[0], nbr.int()) and torch.equal(got[1], d2)
    if what == "near":
        assert rep["knn_retry_tiles"] == 0
    elif what == "plain":
        assert rep["knn_retry_tiles"] > 0.5 * n / 64
