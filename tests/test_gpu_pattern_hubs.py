"""Rows of the symmetric pattern with few, exactly 32, more than 32 (second pass), more than 256
(block path) reverse entries, at every list length class: columns and distances as the oracle's."""
import numpy as np
import pytest
import torch

from oracle import knn as OK
from oracle import method as M

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("k", [1, 7, 32, 33, 64, 65, 128, 129])
@pytest.mark.parametrize("n", [300, 900])
def test_hubs(n, k):
    import paper_2104_15124_gb300 as vb
    r = np.random.default_rng(k)
    # clusters of points on small spheres in R^12 around a hub each: the hub is everybody's neighbour
    sizes = np.array([20, 33, 34, 60, 150, n - 297])
    parts = []
    for s in sizes:
        c = r.standard_normal(12) * 50.0
        v = r.standard_normal((s, 12))
        parts.append(c + np.concatenate([np.zeros((1, 12)), v[1:] / np.linalg.norm(v[1:], axis=1, keepdims=True)]))
    x = np.concatenate(parts).astype(np.float32)[r.permutation(n)]
    nbr, d2 = OK.knn(x, k)
    p = M.sym_pattern(x, nbr)
    vb.report_reset()
    g = vb.graph(torch.from_numpy(nbr.astype(np.int32)).cuda(), torch.from_numpy(d2).cuda())
    torch.cuda.synchronize()
    vb.raise_on_device_error()
    z = g.nnz
    assert z == p.nnz
    assert np.array_equal(g.row_ptr.cpu().numpy(), p.row_ptr)
    assert np.array_equal(g.col[:z].cpu().numpy(), p.col.astype(np.int32))
    assert np.array_equal(g.ed2[:z].cpu().numpy(), p.d2.astype(np.float32))
