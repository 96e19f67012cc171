"""A build streams the products t = ed2 / (rho_i rho_j) that one pass has formed (into the room of
L-hat's values); the step-by-step calls gather per entry.  Both do the same arithmetic per entry in
the same order, so their results agree bit for bit, whatever the row lengths and alignments."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,m,k", [(3, 2, 1), (33, 3, 2), (257, 2, 7), (2000, 3, 33), (4099, 4, 64), (1500, 6, 128)])
@pytest.mark.parametrize("c", [0.0, 1.0])
def test_build_equals_its_steps(n, m, k, c):
    import paper_2104_15124_gb300 as vb
    x = torch.from_numpy(np.random.default_rng(n + k).standard_normal((n, m)).astype(np.float32)).cuda()
    d, beta = 2.0, -0.25
    out = vb.build(x, k, d=d, c=c, beta=beta)
    g = out.graph
    b = vb.bandwidth(out.nbr_d2)
    eps2, chi, dim = vb.epsilon_tune(g, b, 1.0)
    psi, P = vb.density(g, b, eps2, d, beta)
    xi_c = vb.operator_centre(g, b, P)
    eps2_op, chi_op, _ = vb.epsilon_tune(g, P, 4.0, xi_c=xi_c, warn_bit=2)
    val, q, D, S = vb.kernel_csr(g, psi, P, eps2_op, c, beta, d)
    torch.cuda.synchronize()
    nnz = g.nnz
    for name, a, e in (("b", out.b, b), ("eps2", out.eps2_den, eps2), ("chi", out.chi_den, chi), ("dim", out.dim_den, dim),
                       ("psi", out.psi, psi), ("P", out.P, P), ("xi_c", out.xi_c, xi_c), ("eps2_op", out.eps2_op, eps2_op),
                       ("chi_op", out.chi_op, chi_op), ("val", out.val[:nnz], val[:nnz]), ("q", out.q, q), ("D", out.D, D),
                       ("S", out.S, S)):
        assert torch.equal(a, e), name
    # the bandwidth's sums in rank order
    ref = np.zeros(n)
    for r in range(k):
        ref = ref + out.nbr_d2[:, r].cpu().numpy()
    assert np.array_equal(b.cpu().numpy(), np.sqrt(ref))


@pytest.mark.parametrize("offset", [0, 1, 3])
def test_difference_form_product_at_any_alignment(offset):
    # rows of one to many entries, arrays that do and do not start on 16 bytes, and an infinite input:
    # FP64 sums of the same FP32 entries within the rounding of FP32 sums of 2 k + 1 terms
    import paper_2104_15124_gb300 as vb
    r = np.random.default_rng(offset)
    n = 1003
    x = torch.from_numpy(r.standard_normal((n, 3)).astype(np.float32)).cuda()
    out = vb.build(x, 20, d=2.0, c=1.0)
    z = out.graph.nnz
    col = torch.empty(z + 4, dtype=torch.int32, device="cuda")[offset:offset + z].copy_(out.graph.col[:z])
    val = torch.empty(z + 4, dtype=torch.float32, device="cuda")[offset:offset + z].copy_(out.val[:z])
    g = vb.Graph(n, out.graph.row_ptr, col, out.graph.ed2, out.graph.nnz_dev)
    v = torch.from_numpy(r.standard_normal(n).astype(np.float32)).cuda()
    row = torch.repeat_interleave(torch.arange(n, device="cuda"), g.row_ptr[1:] - g.row_ptr[:-1])
    j = col.long()
    zz = v.double() / out.S
    t = val.double() * out.S[j] * (zz[j] - zz[row])
    ref = torch.zeros(n, dtype=torch.float64, device="cuda").index_add_(0, row, t)
    mag = torch.zeros(n, dtype=torch.float64, device="cuda").index_add_(0, row, t.abs())
    y = vb.spmv(g, val, v, S=out.S, laplacian=True)
    assert bool(((y.double() - ref).abs() <= 8 * 2.0 ** -24 * mag + 1e-30).all())
    v[5] = float("inf")
    y = vb.spmv(g, val, v, S=out.S, laplacian=True)
    touched = torch.zeros(n, dtype=torch.bool, device="cuda")
    touched[row[j == 5]] = True
    assert not bool(y[~touched].isinf().any()) and bool(y[touched].isinf().all())
