"""The symmetric pattern where reverse entries fill a row's 64 slots (63 to 66 of them), and where more
overflow than are listed (65,536): columns and distances as the oracle's."""
import numpy as np
import pytest
import torch

from oracle import knn as OK
from oracle import method as M

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("what", ["edges", "overflow"])
def test_pattern(what):
    import paper_2104_15124_gb300 as vb
    r = np.random.default_rng(9)
    if what == "edges":   # a hub at the centre of a sphere in R^24 is in every list of its cluster
        k = 5
        parts = []
        for s in (33, 34, 64, 65, 66, 67, 68, 69, 70, 71, 72, 73):
            v = r.standard_normal((s, 24))
            v[0] = 0.0
            v[1:] /= np.linalg.norm(v[1:], axis=1, keepdims=True)
            parts.append(v + 100.0 * r.standard_normal(24))
        x = np.concatenate(parts)
    else:
        k = 64
        x = r.standard_normal((12000, 24))
    x = x[r.permutation(len(x))].astype(np.float32)
    nbr, d2 = OK.knn(x, k)
    p = M.sym_pattern(x, nbr)
    rev = np.diff(p.row_ptr) - 1 - k
    if what == "edges":
        assert {63, 64, 65, 66} <= set(rev.tolist())
    else:
        assert np.maximum(rev - 64, 0).sum() > 1 << 16
    vb.report_reset()
    g = vb.graph(torch.from_numpy(nbr.astype(np.int32)).cuda(), torch.from_numpy(d2).cuda())
    torch.cuda.synchronize()
    vb.raise_on_device_error()
    z = g.nnz
    assert z == p.nnz
    assert np.array_equal(g.row_ptr.cpu().numpy(), p.row_ptr)
    assert np.array_equal(g.col[:z].cpu().numpy(), p.col.astype(np.int32))
    assert np.array_equal(g.ed2[:z].cpu().numpy(), p.d2.astype(np.float32))
