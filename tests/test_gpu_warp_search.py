"""The warp search (m <= 8, k <= 128) at the edges of its lists, tiles and clouds: the lists and
distances equal the FP64 brute force bit for bit, as every search's must."""
import numpy as np
import pytest
import torch

from oracle import knn as OK

pytestmark = pytest.mark.gpu


def _check(x, k, **kw):
    import paper_2104_15124_gb300 as vb
    ref_nbr, ref_d2 = OK.knn(x, k)
    vb.report_reset()
    nbr, d2 = vb.knn(torch.from_numpy(x).cuda(), k, **kw)
    torch.cuda.synchronize()
    rep = vb.raise_on_device_error()
    assert np.array_equal(nbr.cpu().numpy(), ref_nbr)
    assert np.array_equal(d2.cpu().numpy(), ref_d2)
    return rep, ref_d2


@pytest.mark.parametrize("n,k", [(2, 1), (33, 32), (34, 33), (63, 62), (65, 64), (129, 128), (130, 127), (641, 31),
                                 (4097, 65), (6000, 96), (6001, 128), (9000, 1), (9001, 129)])
@pytest.mark.parametrize("m", [1, 2, 3, 4, 5, 8])
def test_sizes(n, k, m):
    _check(np.random.default_rng(n + 13 * k + m).standard_normal((n, m)).astype(np.float32), k)


@pytest.mark.parametrize("m", [2, 3, 4, 7])
@pytest.mark.parametrize("what", ["outliers", "clusters", "scales", "lattice", "far"])
def test_shapes(what, m):
    # thresholds that change abruptly from one query to the next, exact ties, wide ranges of scale
    r = np.random.default_rng(m)
    x = r.standard_normal((5000, m))
    if what == "outliers":
        x[::97] *= 1e3
    elif what == "clusters":
        x = np.concatenate([x[:1500] * 1e-4, x[1500:3000] * 1e-2 + 5.0, x[3000:]])
    elif what == "scales":
        x *= 10.0 ** r.uniform(-6, 6, (5000, 1))
    elif what == "lattice":
        x = np.round(x * 4.0)
    else:
        x = x * 1e-3 + 1000.0
    _check(x.astype(np.float32), 40)


@pytest.mark.parametrize("tc", [None, "bf16", "fp16"])
def test_radius_guesses_of_every_quality(tc):
    x = np.random.default_rng(3).standard_normal((7000, 3)).astype(np.float32)
    _, d2 = OK.knn(x, 48)
    rk = np.sqrt(d2[:, 47])
    scale = 10.0 ** np.random.default_rng(4).uniform(-2, 2, 7000)   # from far too small to far too large
    _check(x, 48, radius=torch.from_numpy((rk * scale).astype(np.float32)).cuda(), inflate=1.0, tensor_cores=tc)


@pytest.mark.parametrize("m", [2, 3, 4, 6])
def test_clouds_that_share_tiles(m):
    # clouds far below and just above a tile's 64 points, so tiles and groups of queries straddle them
    import paper_2104_15124_gb300 as vb
    r = np.random.default_rng(50 + m)
    sizes = [18, 19, 64, 65, 200, 17, 1000, 40, 63, 2500]
    ptr = np.concatenate([[0], np.cumsum(sizes)])
    x = np.concatenate([r.standard_normal((s, m)) * r.uniform(0.1, 3.0) + r.standard_normal(m) for s in sizes]).astype(np.float32)
    b = vb.Builder(len(x), m, 16, d=2, c=1.0, cloud_ptr=ptr)
    out = b(torch.from_numpy(x).cuda())
    torch.cuda.synchronize()
    vb.raise_on_device_error()
    for lo, hi in zip(ptr[:-1], ptr[1:]):
        ref_nbr, ref_d2 = OK.knn(x[lo:hi], 16)
        assert np.array_equal(out.nbr[lo:hi].cpu().numpy() - lo, ref_nbr)
        assert np.array_equal(out.nbr_d2[lo:hi].cpu().numpy(), ref_d2)
