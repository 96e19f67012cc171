"""Performance cases: the work that a user of this library has it do.

Each case is one call, or one training epoch, through the public Python entry points, on the
synthetic manifold samples of paper_2104_15124_gb300/workloads.py.  `prepare` holds what a
program keeps between calls (a Builder with its buffers, the samples on the GPU, a trained
radius network); `run` is the call itself and returns every output of it.

The outputs of a build include the CSR arrays at their allocated size, n (2k + 1) entries, of
which the first nnz are used; `prepare` clears them, so the unused tail is zero.
"""
import math

import numpy as np
import torch

import paper_2104_15124_gb300 as vb
from paper_2104_15124_gb300 import workloads as W

BETA = -0.25


def listed():
    return [
        # the smallest build: the unit circle of the parity configuration; latency and launches count
        {"name": "circle_2k", "kind": "build", "cloud": "circle", "n": 2000, "m": 2, "k": 32, "d": 1, "c": 0.0, "tc": ""},
        # an ordinary build in three dimensions with a varying density, BF16 tiles
        {"name": "sphere_50k_bf16", "kind": "build", "cloud": "vmf", "n": 50000, "m": 3, "k": 64, "d": 2, "c": 1.0,
         "tc": "bf16"},
        # an odd size in more dimensions than the space-filling curve takes: principal-axis order, 8-wide rows
        {"name": "gauss8_20011", "kind": "build", "cloud": "gauss", "n": 20011, "m": 8, "k": 48, "d": 8, "c": 1.0, "tc": ""},
        # the large single cloud, plain call
        {"name": "torus_1m", "kind": "build", "cloud": "torus", "n": 1000000, "m": 4, "k": 64, "d": 2, "c": 1.0, "tc": ""},
        # the large single cloud in its configured form: learned radius and BF16 tiles
        {"name": "torus_1m_learned_bf16", "kind": "build", "cloud": "torus", "n": 1000000, "m": 4, "k": 64, "d": 2, "c": 1.0,
         "tc": "bf16", "learned": True},
        # wide coordinates: a 5-dimensional Gaussian in R^100, FP16 tiles, the largest k
        {"name": "gauss100_200k_fp16", "kind": "build", "cloud": "gauss100", "n": 200000, "m": 100, "k": 128, "d": 5, "c": 1.0,
         "tc": "fp16"},
        # 256 clouds of uneven size in one launch sequence, replayed from a CUDA graph
        {"name": "ellipsoids_256_graph", "kind": "batch", "clouds": 256, "lo": 2000, "hi": 40000, "m": 3, "k": 32, "d": 2,
         "c": 1.0, "tc": "bf16", "learned": True, "graph": True},
        # the product L-hat x in difference form that an iterative solver calls again and again
        {"name": "spmv_torus_1m", "kind": "spmv", "cloud": "torus", "n": 1000000, "m": 4, "k": 64, "d": 2, "c": 1.0},
        # 32 eigenpairs and the spectral solve of L f = g
        {"name": "solve_sphere_50k", "kind": "solve", "cloud": "vmf", "n": 50000, "m": 3, "k": 64, "d": 2, "c": 1.0, "ell": 32},
        # one step of the particle evolution (build, solve, gradient, update), the whole call
        {"name": "evolve_4k", "kind": "evolve", "n": 4000, "m": 2, "k": 128, "ell": 8},
        # the epsilon sweep over the delta_tol pattern of every grid point, a cloud with its own bandwidths
        {"name": "radius_sweep_5003", "kind": "radius", "cloud": "vmf", "n": 5003, "m": 3, "k": 32, "tol": 0.01},
        # training of the radius network: one epoch, forward, backward and Adam
        {"name": "train_radius_100k", "kind": "train", "cloud": "torus", "n": 100000, "m": 4, "batch": 4096},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


_CLOUDS = {"circle": (2, 1, 0.0), "vmf": (3, 2, 1.0), "sphere": (3, 2, 1.0), "torus": (4, 2, 1.0)}


def draw(rng):
    kind = rng.choice(["build", "build", "build", "build", "wide", "batch", "spmv", "solve", "evolve", "radius", "train"])
    if kind == "build":
        cloud = rng.choice(["circle", "vmf", "sphere", "torus", "gauss"])
        k = rng.choice([8, 16, 31, 32, 48, 64, 100, 128])
        if cloud == "gauss":
            m = rng.randint(2, 12)
            n = _log_int(rng, 1000, 200000 if m <= 4 else 30000)
            d, c = m, rng.choice([0.0, 1.0])
        else:
            m, d, c = _CLOUDS[cloud]
            n = _log_int(rng, 1000, 1000000 if k <= 64 else 300000)
        return {"kind": "build", "cloud": cloud, "n": n, "m": m, "k": k, "d": d, "c": c,
                "tc": rng.choice(["", "", "bf16", "fp16"]),
                "learned": cloud in ("vmf", "torus") and n >= 20000 and rng.random() < 0.3}
    if kind == "wide":
        return {"kind": "build", "cloud": "gauss100", "n": _log_int(rng, 2000, 150000), "m": rng.choice([24, 50, 64, 100, 128]),
                "k": rng.choice([32, 64, 100, 128]), "d": 5, "c": 1.0, "tc": "fp16"}
    if kind == "batch":
        return {"kind": "batch", "clouds": rng.randint(2, 200), "lo": 500, "hi": rng.randint(2000, 30000), "m": 3,
                "k": rng.choice([16, 32, 48]), "d": 2, "c": 1.0, "tc": rng.choice(["", "bf16", "fp16"]),
                "learned": rng.random() < 0.5, "graph": rng.random() < 0.5}
    if kind in ("spmv", "solve"):
        cloud = rng.choice(["circle", "vmf", "torus"])
        m, d, c = _CLOUDS[cloud]
        case = {"kind": kind, "cloud": cloud, "n": _log_int(rng, 2000, 1000000 if kind == "spmv" else 50000), "m": m,
                "k": rng.choice([24, 32, 64]), "d": d, "c": c}
        if kind == "solve":
            case["ell"] = rng.choice([8, 16, 32])
        return case
    if kind == "evolve":
        return {"kind": "evolve", "n": _log_int(rng, 1500, 8000), "m": rng.randint(2, 3), "k": rng.choice([48, 64, 128]),
                "ell": rng.choice([6, 8, 12])}
    if kind == "radius":
        cloud = rng.choice(["vmf", "sphere", "torus"])
        return {"kind": "radius", "cloud": cloud, "n": _log_int(rng, 1000, 5000), "m": _CLOUDS[cloud][0], "k": 32,
                "tol": rng.choice([0.001, 0.01, 0.1])}
    return {"kind": "train", "cloud": "torus", "n": _log_int(rng, 20000, 200000), "m": 4, "batch": rng.choice([1024, 2048, 4096])}


# ----------------------------------------------------------------------------- inputs
def _sample(case, seed):
    n, cloud = case["n"], case["cloud"]
    seed = 7919 * seed + 11
    if cloud == "circle":
        return W.circle(n, seed)
    if cloud == "vmf":
        return W.sphere_vmf(n, 2.0, seed)
    if cloud == "sphere":
        return W.sphere_uniform(n, seed)
    if cloud == "torus":
        return W.torus4(n, 0.01, seed)
    if cloud == "gauss":
        return W.gaussian(n, case["m"], None, seed)
    return W.gauss_embedded(n, 5, case["m"], 1e-3, seed).x


def _batch_ptr(case):
    """Offsets of the clouds: their sizes are the case's, whatever the seed of the samples."""
    r = np.random.default_rng(case["clouds"])
    sizes = np.floor(r.uniform(case["lo"], case["hi"] + 1, case["clouds"])).astype(np.int64)
    return np.concatenate([np.zeros(1, dtype=np.int64), np.cumsum(sizes)])


def _batch(case, seed):
    """The clouds of workloads.ellipsoids() at those sizes: ellipsoids with semi-axes U[0.5, 2],
    samples uniform in the polar and the azimuthal angle, drawn on the GPU."""
    ptr = _batch_ptr(case)
    g = torch.Generator(device="cuda").manual_seed(7919 * seed + 11)
    axes = torch.rand((case["clouds"], 3), generator=g, device="cuda", dtype=torch.float64) * 1.5 + 0.5
    sizes = torch.from_numpy(np.diff(ptr)).cuda()
    a = axes.repeat_interleave(sizes, dim=0)
    u = torch.rand((int(ptr[-1]), 2), generator=g, device="cuda", dtype=torch.float64)
    th, ph = math.pi * u[:, 0], 2.0 * math.pi * u[:, 1]
    x = torch.stack([th.sin() * ph.cos(), th.sin() * ph.sin(), th.cos()], dim=1) * a
    return x.float().contiguous(), ptr


def _gpu(a):
    return torch.from_numpy(np.ascontiguousarray(a, dtype=np.float32)).cuda()


def _radius_net(x, target):
    """The radius network fitted to (x, log r), with the shift and the inflation its residual gives."""
    net = vb.train_radius_model(x, target, epochs=6, batch=4096, seed=103)
    resid = target - net.predict(x)
    return net, float(resid.mean()), math.exp(3.0 * float(resid.std()))


def _learned(case, seed):
    """Builder arguments of the learned radius, trained on a separate smaller draw of the same law."""
    if case["kind"] == "batch":
        n_ref = 0.5 * (case["lo"] + case["hi"])
        bt = W.ellipsoids(3, case["lo"], case["hi"], 104729 + seed)
        x = _gpu(bt.x)
        parts = []
        for lo, hi in zip(bt.cloud_ptr[:-1], bt.cloud_ptr[1:]):
            _, d2 = vb.knn(x[lo:hi].contiguous(), case["k"])
            parts.append(0.5 * torch.log(d2[:, case["k"] - 1]) + math.log((hi - lo) / n_ref) / case["d"])
        net, shift, inflate = _radius_net(x, torch.cat(parts).float())
        sizes = np.diff(_batch_ptr(case)).astype(np.float64)
        return {"mlp": net, "log_shift": shift, "inflate": inflate,
                "cloud_log_shift": (np.log(n_ref / sizes) / case["d"]).astype(np.float32)}
    n = max(case["n"] // 10, 10000)
    kp = max(1, round(case["k"] * n / case["n"]))
    x = _gpu(_sample(dict(case, n=n), 104729 + seed))
    _, d2 = vb.knn(x, kp)
    net, shift, inflate = _radius_net(x, (0.5 * torch.log(d2[:, kp - 1])).float())
    return {"mlp": net, "log_shift": shift, "inflate": inflate}


def _cleared(builder):
    for t in (builder.out.graph.col, builder.out.graph.ed2, builder.out.val):
        t.zero_()
    return builder


def _operator(case, seed):
    """The operator of a cloud, as a solver has it in hand."""
    x = _gpu(_sample(case, seed))
    b = vb.Builder(case["n"], case["m"], case["k"], d=case["d"], c=case["c"], beta=BETA)
    out = b(x)
    nnz = out.graph.nnz
    g = vb.Graph(case["n"], out.graph.row_ptr, out.graph.col[:nnz].clone(), out.graph.ed2[:nnz].clone(), out.graph.nnz_dev)
    return x, g, out.val[:nnz].clone(), out.S


def prepare(case, seed):
    kind = case["kind"]
    if kind in ("build", "batch"):
        kw = {"tensor_cores": case["tc"] or None}
        if kind == "batch":
            x, kw["cloud_ptr"] = _batch(case, seed)
            n = x.shape[0]
        else:
            x, n = _gpu(_sample(case, seed)), case["n"]
        if case.get("learned"):
            kw.update(_learned(case, seed))
        b = _cleared(vb.Builder(n, case["m"], case["k"], d=case["d"], c=case["c"], beta=BETA, **kw))
        s = {"kind": kind, "x": x, "builder": b}
        if case.get("graph"):
            s["graph"] = b.graph(x)
        return s
    if kind == "spmv":
        _, g, val, S = _operator(case, seed)
        v = torch.from_numpy(np.random.default_rng(seed).standard_normal(case["n"]).astype(np.float32)).cuda()
        return {"kind": kind, "g": g, "val": val, "S": S, "v": v}
    if kind == "solve":
        x, g, val, S = _operator(case, seed)
        return {"kind": kind, "g": g, "val": val, "S": S, "ell": case["ell"], "rhs": x[:, 0].contiguous()}
    if kind == "evolve":
        r = np.random.default_rng(seed)
        n, m = case["n"], case["m"]
        x = r.standard_normal((n, m)).astype(np.float32)
        return {"kind": kind, "x": _gpu(x), "sigma": _gpu(np.eye(m)), "W": _gpu(r.standard_normal((n, m))),
                "g": _gpu(x[:, 0]), "k": case["k"], "ell": case["ell"], "d": float(m)}
    if kind == "radius":
        x = _gpu(_sample(case, seed))
        _, d2 = vb.knn(x, case["k"])
        return {"kind": kind, "x": x, "rho": vb.bandwidth(d2), "tol": case["tol"]}
    x = _gpu(_sample(case, seed))
    _, d2 = vb.knn(x, 8)
    y = (0.5 * torch.log(d2[:, 7])).float()
    net = vb.Mlp(case["m"], seed=seed)
    net.fit_standardisation(x, y)
    return {"kind": kind, "x": x, "y": y, "net": net, "batch": case["batch"]}


# ----------------------------------------------------------------------------- the call
_BUILD = ("nbr", "nbr_d2", "b", "eps2_den", "chi_den", "dim_den", "psi", "P", "xi_c", "eps2_op", "chi_op", "dim_op", "val",
          "q", "D", "S")


def _outputs(out):
    r = {f: getattr(out, f) for f in _BUILD}
    r.update(row_ptr=out.graph.row_ptr, col=out.graph.col, ed2=out.graph.ed2, nnz=out.graph.nnz_dev)
    return r


def run(s):
    kind = s["kind"]
    if kind in ("build", "batch"):
        if "graph" in s:
            s["graph"].replay()
            return _outputs(s["builder"].out)
        return _outputs(s["builder"](s["x"]))
    if kind == "spmv":
        return vb.spmv(s["g"], s["val"], s["v"], S=s["S"], laplacian=True)
    if kind == "solve":
        e = vb.solve(s["g"], s["val"], s["S"], s["ell"], rhs=s["rhs"])
        return {"evals": e.evals, "phi": e.phi, "f": e.f}
    if kind == "evolve":
        st = vb.evolve_step(s["x"], 0.01, s["sigma"], s["W"], s["g"], k=s["k"], ell=s["ell"], d=s["d"])
        return {"x_next": st.x_next, "grad_f": st.grad_f, "f": st.f, "S": st.build.S, "psi": st.build.psi}
    if kind == "radius":
        chi, eps2, dim = vb.radius_sweep(s["x"], s["rho"], 1.0, s["tol"])
        return {"chi": chi, "eps2": eps2, "dim": dim}
    loss = s["net"].train_epoch(s["x"], s["y"], batch=s["batch"], lr=3e-3, seed=1)
    return {"loss": loss, "master": s["net"].master}


# ----------------------------------------------------------------------------- what a pass cannot do without
def work(case):
    kind, m = case["kind"], case["m"]
    if kind == "batch":
        n = case["clouds"] * (case["lo"] + case["hi"]) // 2
    else:
        n = case["n"]
    if kind in ("build", "batch"):
        # samples in; lists, pattern, L-hat and the per-point vectors out; per entry 2 x 57 sweep
        # terms and four kernel evaluations, per neighbour one distance
        k = case["k"]
        nnz = int(1.15 * n * k) + n
        return {"bytes": 4 * n * m + 12 * n * k + 12 * nnz + 8 * (n + 1) + 56 * n,
                "flops": 3 * m * n * k + nnz * (2 * 57 * 2 + 4 * 10)}
    if kind == "spmv":
        nnz = int(1.15 * n * case["k"]) + n
        return {"bytes": 8 * nnz + 8 * (n + 1) + 16 * n, "flops": 4 * nnz}
    if kind == "solve":
        # the operator and the right-hand side in, the eigenpairs and f out; about ten filters of degree 30
        nnz, cols = int(1.15 * n * case["k"]) + n, case["ell"] + 1
        return {"bytes": 8 * nnz + 20 * n + 4 * n * (cols + 1), "flops": 300 * 3 * nnz * cols}
    if kind == "evolve":
        k, cols = case["k"], case["ell"] + 1
        nnz = int(1.15 * n * k) + n
        return {"bytes": 4 * n * (5 * m + 3) + 12 * nnz + 12 * n * k, "flops": 300 * 3 * nnz * cols}
    if kind == "radius":
        # at the largest epsilon of the grid nearly every pair counts: one distance, and about 25
        # kernel values of some 20 operations each over the grid points that keep it
        return {"bytes": 4 * n * m + 8 * n + 8 * 59, "flops": n * n * (3 * m + 2 + 25 * 20)}
    H = 64
    return {"bytes": n * (4 * m + 4) + 12 * (H * (m + H + 3) + 1), "flops": 6 * n * (H * m + H * H + H)}


# ----------------------------------------------------------------------------- the same in 64 bits
def _knn64(x, k):
    """Exact neighbour lists of FP64 points on the GPU, by brute force: (indices, squared distances)."""
    n, m = x.shape
    idx, d2 = [], []
    step = max(1, (1 << 27) // n)
    for lo in range(0, n, step):
        q = x[lo:lo + step]
        d = torch.zeros((q.shape[0], n), dtype=torch.float64, device=x.device)
        for r in range(m):
            d += (q[:, r:r + 1] - x[None, :, r]).square_()
        d[torch.arange(q.shape[0]), torch.arange(lo, lo + q.shape[0])] = math.inf
        v, i = torch.topk(d, k, dim=1, largest=False, sorted=True)
        idx.append(i)
        d2.append(v)
    return torch.cat(idx), torch.cat(d2)


def _build64(x, k, d, c):
    """The build in FP64 from its definition, as a dict like run()'s."""
    n = x.shape[0]
    dev = x.device
    nbr, d2 = _knn64(x, k)
    b = d2.sum(1).sqrt()
    ar = torch.arange(n, device=dev)
    own = ar.repeat_interleave(k)
    key = torch.unique(torch.cat([ar * n + ar, own * n + nbr.reshape(-1), nbr.reshape(-1) * n + own]))
    row, col = key // n, key % n
    e2 = torch.zeros(row.shape[0], dtype=torch.float64, device=dev)
    for r in range(x.shape[1]):
        e2 += (x[row, r] - x[col, r]).square()
    off = row != col
    grid = torch.arange(57, dtype=torch.float64, device=dev) * 0.25 - 10.0

    def rows(v):
        return torch.zeros(n, dtype=torch.float64, device=dev).index_add_(0, row, v)

    def sweep(t, centre):
        chi = torch.stack([torch.exp(-t / 2.0 ** float(g + centre)).sum() for g in grid])
        slope = (chi[1:].log() - chi[:-1].log()) / (0.25 * math.log(2.0))
        g = int(slope.argmax())
        return 2.0 ** float(grid[g] + centre), chi, 2.0 * slope[g]

    eps2, chi, dim = sweep(e2 / (b[row] * b[col]), 0.0)
    psi = rows(torch.exp(-e2 / (eps2 * b[row] * b[col]))) / (n * (math.pi * eps2 * b * b) ** (d / 2.0))
    P = psi ** BETA
    arg = e2 / (4.0 * P[row] * P[col])
    xc = math.floor(4.0 * math.log2(float(arg[off].sum() / (e2 / (b[row] * b[col]))[off].sum())) + 0.5) / 4.0
    eps2o, chio, dimo = sweep(arg, xc)
    alpha = (2.0 - c + (d + 2) * BETA) / 2.0
    K = torch.exp(-arg / eps2o)
    q = psi ** (-BETA * d) * rows(K)
    K = K / (q[row] * q[col]) ** alpha
    D = rows(K)
    S = P * D.sqrt()
    val = (K / (S[row] * S[col]) - (~off).double() / P[row] ** 2) / eps2o
    nnz = row.shape[0]

    def padded(v):
        w = torch.zeros(n * (2 * k + 1), dtype=torch.float64, device=dev)
        w[:nnz] = v
        return w

    def one(v):
        return torch.tensor([float(v)], dtype=torch.float64, device=dev)

    return {"nbr": None, "nbr_d2": d2, "b": b, "eps2_den": one(eps2), "chi_den": chi, "dim_den": one(dim), "psi": psi, "P": P,
            "xi_c": one(xc), "eps2_op": one(eps2o), "chi_op": chio, "dim_op": one(dimo), "val": padded(val), "q": q, "D": D,
            "S": S, "row_ptr": None, "col": None, "ed2": padded(e2), "nnz": None}


def exact(case, seed):
    kind = case["kind"]
    if kind == "build" and case["n"] * case["n"] * case["m"] <= 1e10:
        x = _gpu(_sample(case, seed)).double()
        return _build64(x, case["k"], case["d"], case["c"])
    if kind == "spmv":
        s = prepare(case, seed)
        g, n = s["g"], case["n"]
        row = torch.repeat_interleave(torch.arange(n, device="cuda"), g.row_ptr[1:] - g.row_ptr[:-1])
        col = g.col.long()
        z = s["v"].double() / s["S"]
        t = s["val"].double() * s["S"][col] * (z[col] - z[row])
        return torch.zeros(n, dtype=torch.float64, device="cuda").index_add_(0, row, t)
    if kind == "solve" and case["n"] <= 4000:
        s = prepare(case, seed)
        g, n = s["g"], case["n"]
        row = torch.repeat_interleave(torch.arange(n, device="cuda"), g.row_ptr[1:] - g.row_ptr[:-1])
        col, S = g.col.long(), s["S"]
        # L z = sum_j w_ij (z_j - z_i): the symmetric matrix with that diagonal
        off = row != col
        A = torch.zeros((n, n), dtype=torch.float64, device="cuda")
        A[row[off], col[off]] = s["val"].double()[off]
        w = s["val"].double()[off] * S[col[off]] / S[row[off]]
        A.diagonal().copy_(-torch.zeros(n, dtype=torch.float64, device="cuda").index_add_(0, row[off], w))
        ev, v = np.linalg.eigh(A.cpu().numpy())
        ev, v = ev[::-1][:case["ell"] + 1].copy(), v[:, ::-1][:, :case["ell"] + 1] * math.sqrt(n)
        Sn = S.cpu().numpy()
        phi = v / Sn[:, None]
        gt = phi[:, 1:].T @ (Sn * Sn * s["rhs"].cpu().numpy().astype(np.float64)) / n
        return {"evals": ev, "phi": None, "f": phi[:, 1:] @ (gt / ev[1:])}
    if kind == "radius":
        s = prepare(case, seed)
        x, rho, n = s["x"].double(), s["rho"], case["n"]
        tau = -math.log(case["tol"])
        chi = torch.zeros(57, dtype=torch.float64, device="cuda")
        for lo in range(0, n, 2048):
            d = torch.zeros((min(2048, n - lo), n), dtype=torch.float64, device="cuda")
            for r in range(case["m"]):
                d += (x[lo:lo + 2048, r:r + 1] - x[None, :, r]).square_()
            t = d / (rho[lo:lo + 2048, None] * rho[None, :])
            for g in range(57):
                u = t / 2.0 ** (-10.0 + 0.25 * g)
                chi[g] += torch.where(u < tau, torch.exp(-u), 0.0).sum()
        slope = (chi[1:].log() - chi[:-1].log()) / (0.25 * math.log(2.0))
        g = int(slope.argmax())
        return {"chi": chi, "eps2": torch.tensor([2.0 ** (-10.0 + 0.25 * g)], dtype=torch.float64), "dim": 2.0 * slope[g:g + 1]}
    return None   # larger ones take too long; the order of a training epoch's samples is the library's own
