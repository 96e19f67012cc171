"""The difference-form product L-hat x over the range of z = x / S that FP64 differences allow: z beyond
the largest FP32 number with differences inside it, z far below, and x constant but for its last digits.
Tolerance: four FP32 roundings a term (S, val S, the difference, the product) and a sum of at most `len`
of them, (len + 4) 2^-24 of the sum of the terms' magnitudes."""
import ctypes

import numpy as np
import pytest
import torch

from paper_2104_15124_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("zscale,rel", [(1.0, 1.0), (1e40, 1e-5), (1e38, 1e-3), (1e-30, 1e-3), (1.0, 1e-6)])
@pytest.mark.parametrize("entry", ["spmv", "noalloc"])
def test_range(entry, zscale, rel):
    import paper_2104_15124_gb300 as vb
    out = vb.build(torch.from_numpy(W.circle(3001, 5)).cuda(), 24, d=1, c=0.0)
    g, n = out.graph, out.graph.n
    z = g.nnz
    r = np.random.default_rng(7)
    S = out.S * (1e-12 if zscale > 1 else 1.0)
    x = (zscale * (1.0 + rel * r.standard_normal(n)) * S.cpu().numpy()).astype(np.float32)
    xt = torch.from_numpy(x).cuda()
    if entry == "spmv":
        y = vb.spmv(g, out.val, xt, S=S, laplacian=True)
    else:
        y = torch.zeros(n, dtype=torch.float32, device="cuda")
        gc = g.c()
        p = lambda t: ctypes.c_void_p(t.data_ptr())
        assert vb.lib().vb_spmv_laplacian_noalloc(ctypes.c_void_p(torch.cuda.current_stream().cuda_stream), ctypes.byref(gc),
                                                  p(out.val), p(S), 1.0, p(xt), 0.0, p(y)) == 0
    torch.cuda.synchronize()
    ptr, col = g.row_ptr.cpu().numpy(), g.col[:z].cpu().numpy()
    row = np.repeat(np.arange(n), np.diff(ptr))
    off = row != col
    row, col = row[off], col[off]
    S64 = S.cpu().numpy()
    zz = x.astype(np.float64) / S64
    t = out.val[:z].cpu().numpy().astype(np.float64)[off] * S64[col] * (zz[col] - zz[row])
    ref, mag = np.bincount(row, t, n), np.bincount(row, np.abs(t), n)
    err = np.abs(y.cpu().numpy().astype(np.float64) - ref)
    assert np.all(err <= (np.diff(ptr).max() + 4) * 2.0 ** -24 * mag)
