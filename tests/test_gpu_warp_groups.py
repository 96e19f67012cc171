"""The warp search where one warp takes groups of 8 and 16 points (clouds of more than 38,912 and 77,824
points): with per-point radius guesses that differ by more than a group's extent, on clouds whose
thresholds change abruptly, and in a batch.  Lists and distances equal the FP64 brute force bit for bit."""
import functools

import numpy as np
import pytest
import torch

from oracle import knn as OK

pytestmark = pytest.mark.gpu


@functools.lru_cache(maxsize=1)
def _uniform(n, m):
    x = np.random.default_rng(n + m).uniform(0.0, 1.0, (n, m)).astype(np.float32)
    return x, *OK.knn(x, 128)


def _check(x, ref_nbr, ref_d2, **kw):
    import paper_2104_15124_gb300 as vb
    vb.report_reset()
    nbr, d2 = vb.knn(torch.from_numpy(x).cuda(), ref_nbr.shape[1], **kw)
    torch.cuda.synchronize()
    vb.raise_on_device_error()
    wrong = np.any(nbr.cpu().numpy() != ref_nbr, axis=1)
    assert not wrong.any(), f"{wrong.sum()} rows differ"
    assert np.array_equal(d2.cpu().numpy(), ref_d2)


@pytest.mark.parametrize("n,m", [(41000, 2), (41000, 3), (83000, 2), (83000, 3)])
@pytest.mark.parametrize("k", [64, 128])
@pytest.mark.parametrize("guess", ["0.5-1.2", "0.5-1.5", "0.56 or 1.6", "any"])
def test_uneven_radius_guesses(n, m, k, guess):
    x, nbr, d2 = _uniform(n, m)
    r = np.random.default_rng(k)
    f = {"0.5-1.2": r.uniform(0.5, 1.2, n), "0.5-1.5": r.uniform(0.5, 1.5, n),
         "0.56 or 1.6": r.choice([0.56, 1.6], n), "any": 10.0 ** r.uniform(-0.5, 1.0, n)}[guess]
    radius = torch.from_numpy((np.sqrt(d2[:, k - 1]) * f).astype(np.float32)).cuda()
    _check(x, nbr[:, :k], d2[:, :k], radius=radius, inflate=1.0)


@pytest.mark.parametrize("what,m", [("outliers", 3), ("clusters", 2), ("scales", 4), ("lattice", 2), ("gauss", 6)])
def test_shapes(what, m):
    r = np.random.default_rng(m)
    x = r.standard_normal((41000, m))
    if what == "outliers":
        x[::97] *= 1e3
    elif what == "clusters":
        x = np.concatenate([x[:15000] * 1e-4, x[15000:30000] * 1e-2 + 5.0, x[30000:]])
    elif what == "scales":
        x *= 10.0 ** r.uniform(-4, 4, (41000, 1))
    elif what == "lattice":
        x = np.round(x * 40.0)
    x = x.astype(np.float32)
    nbr, d2 = OK.knn(x, 40)
    _check(x, nbr, d2)
    f = r.uniform(0.5, 1.5, 41000)
    _check(x, nbr, d2, radius=torch.from_numpy((np.sqrt(d2[:, 39]) * f).astype(np.float32)).cuda(), inflate=1.0)


def test_batch_of_uneven_clouds():
    import paper_2104_15124_gb300 as vb
    r = np.random.default_rng(5)
    sizes = [30000, 70, 33, 15001, 640, 29000, 5003, 100, 4000]   # 83,847 points: groups of 16
    ptr = np.concatenate([[0], np.cumsum(sizes)])
    x = np.concatenate([r.standard_normal((s, 3)) * r.uniform(0.1, 3.0) + r.standard_normal(3) for s in sizes]).astype(np.float32)
    refs = [OK.knn(x[lo:hi], 32) for lo, hi in zip(ptr[:-1], ptr[1:])]
    rk = np.concatenate([np.sqrt(d[:, 31]) for _, d in refs])
    radius = torch.from_numpy((rk * r.uniform(0.5, 1.3, len(x))).astype(np.float32)).cuda()
    b = vb.Builder(len(x), 3, 32, d=2, c=1.0, cloud_ptr=ptr, radius=radius, inflate=1.0)
    out = b(torch.from_numpy(x).cuda())
    torch.cuda.synchronize()
    vb.raise_on_device_error()
    for lo, hi, (nbr, d2) in zip(ptr[:-1], ptr[1:], refs):
        assert np.array_equal(out.nbr[lo:hi].cpu().numpy() - lo, nbr)
        assert np.array_equal(out.nbr_d2[lo:hi].cpu().numpy(), d2)
