"""vb_profile_read's launch count equals the kernel nodes of the same call recorded in a CUDA graph, on the
one-block order (n <= 4,096, m <= 8) and the general one."""
import ctypes

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


def _kernel_nodes(call):
    g = torch.cuda.CUDAGraph(keep_graph=True)
    with torch.cuda.graph(g, capture_error_mode="thread_local"):
        keep = call()
    rt = ctypes.CDLL("libcudart.so.13")
    graph, num = ctypes.c_void_p(g.raw_cuda_graph()), ctypes.c_size_t(0)
    assert rt.cudaGraphGetNodes(graph, None, ctypes.byref(num)) == 0
    nodes = (ctypes.c_void_p * num.value)()
    assert rt.cudaGraphGetNodes(graph, nodes, ctypes.byref(num)) == 0
    kernels = 0
    for nd in nodes:
        ty = ctypes.c_int(-1)
        assert rt.cudaGraphNodeGetType(ctypes.c_void_p(nd), ctypes.byref(ty)) == 0
        kernels += ty.value == 0
    del keep
    return kernels


@pytest.mark.parametrize("n,m", [(2000, 2), (4096, 6), (4097, 3), (4097, 6), (2000, 20)])
@pytest.mark.parametrize("what", ["knn", "radius_sweep"])
def test_count(what, n, m):
    import paper_2104_15124_gb300 as vb
    x = torch.from_numpy(np.random.default_rng(n + m).standard_normal((n, m)).astype(np.float32)).cuda()
    rho = torch.ones(n, dtype=torch.float64, device="cuda")
    call = (lambda: vb.knn(x, 16)) if what == "knn" else (lambda: vb.radius_sweep(x, rho, 1.0, 0.5, (-14.0, 0.0, 0.25)))
    call()
    torch.cuda.synchronize()
    vb.profile_enable(True)
    call()
    _, launches = vb.profile_read()
    vb.profile_enable(False)
    assert launches == _kernel_nodes(call)
