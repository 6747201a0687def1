"""Measured workloads of the eigensolver: what its users call, over the sizes they call it with.

``listed()`` names the cases; ``draw(rng)`` gives one more of the same ranges;
``prepare(case, seed)`` builds the matrix, the decomposition handle and the
vectors; ``run(state)`` is one pass through the public entry points;
``work(case)`` its unavoidable bytes and operations; ``exact(case, seed)`` the
outputs computed by plain torch in 64 bits.

Matrices (the kinds and sizes of this repository's configurations, tests and
benchmark):

* ``fd2d``, ``fd3d``: cell-centred finite-difference operators -div(a grad u)
  with Dirichlet boundary, a per cell = 10^U(lo, hi), in 3D with boxes set to
  1e4 (the high-contrast operators);
* ``torus``: symmetric 10-nearest-neighbour graph Laplacian of points on a
  torus, weights exp(-d^2 / sigma^2), + 1e-6 I (the point-cloud graphs);
* ``rgg``: random geometric graph Laplacian in the unit square, mean degree
  10, weights U(0.5, 2), + 1e-6 I (``step``: its largest component).

The seed draws the coefficients, points or weights and the vectors.  The
points of an ``rgg``, and of a ``torus`` whose coarse levels are called, go
with the size alone: one graph, many weights or right-hand sides.

Entry points (``"call"``):

* ``spmv``: y = A x (``MMD.level_spmv``);
* ``op``: y = A^(k)^{-1} M^(k) x by (preconditioned) conjugate gradients, the
  operator of every Lanczos step (``MMD.level_op``);
* ``bsolve``: the complement solve that starts a refinement (``MMD.level_bsolve``);
* ``block``: the same operator on a block of columns, the refinement's solve
  (``MMD.level_op_block``), in FP64 or mixed precision;
* ``eig``: the N leftmost eigenpairs (``MMD.eig_leftmost``);
* ``batch``: many small eigenproblems at once (``eig_leftmost_batched``);
* ``step``: forward and backward of a loss on eigenvalues and the Fiedler
  vector (``eigsh_leftmost``), gradients with respect to the matrix values.

Solver tolerances are those that the eigensolver itself asks for: a tenth of
the residual target.  Targets are 1e-10 (the finite-difference configuration)
to 1e-12 (eigenvectors that gradients are taken through).
"""
import math

import numpy as np
import torch

import paper_1804_03415_gb300 as G

PRECISION = {"fp64": G.MMD_FP64, "mixed": G.MMD_MIXED}


def listed():
    return [
        # the smallest call: one product with the 64 x 64 finite-difference operator, all latency
        {"name": "spmv_fd2d_64", "call": "spmv", "matrix": "fd2d", "size": 64},
        # the memory-bound product: the 128^3 high-contrast operator, 175 MB of matrix
        {"name": "spmv_fd3d_128", "call": "spmv", "matrix": "fd3d", "size": 128},
        # one Lanczos step's solve on a small, badly conditioned operator (config: 64 x 64, a = 10^U(-2,2))
        {"name": "op_fd2d_64", "call": "op", "matrix": "fd2d", "size": 64, "level": 0, "tol": 1e-11},
        # the same on a mid-sized graph (the differentiation config's 50k nodes)
        {"name": "op_rgg_50k", "call": "op", "matrix": "rgg", "size": 50000, "level": 0, "tol": 1e-12},
        # the same on the benchmark's point-cloud graph: where its eigensolve spends its time
        {"name": "op_torus_200k", "call": "op", "matrix": "torus", "size": 200000, "level": 0, "tol": 1e-11},
        # a Lanczos step on a coarse level: PCG on A^(1) with an inner CG on M^(1)
        {"name": "op_level1_torus_100k", "call": "op", "matrix": "torus", "size": 100000, "level": 1, "tol": 1e-11},
        # the complement solve that starts the refinement of the benchmark's finest level
        {"name": "bsolve_torus_200k", "call": "bsolve", "matrix": "torus", "size": 200000, "level": 1, "tol": 1e-11},
        # a refinement's block of solves in FP64, a ragged last tile
        {"name": "block_torus_50k", "call": "block", "matrix": "torus", "size": 50000, "level": 0, "m": 11,
         "tol": 1e-11, "precision": "fp64"},
        # the same in mixed precision, the benchmark's block width
        {"name": "block_mixed_torus_50k", "call": "block", "matrix": "torus", "size": 50000, "level": 0, "m": 50,
         "tol": 1e-11, "precision": "mixed"},
        # a whole eigensolve on a point-cloud graph with the default options
        {"name": "eig_torus_20k", "call": "eig", "matrix": "torus", "size": 20000, "n_eig": 16, "tol": 1e-12,
         "precision": "fp64"},
        # many small graphs of uneven sizes at once
        {"name": "batch_torus_6x", "call": "batch", "matrix": "torus", "size": 6000, "count": 6, "n_eig": 8,
         "tol": 1e-12},
        # one training step on edge weights: eigenpairs, loss on 8 eigenvalues and the Fiedler vector, backward
        {"name": "step_rgg_1500", "call": "step", "matrix": "rgg", "size": 1500, "n_eig": 8, "tol": 1e-12},
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["spmv", "spmv3", "op_fd", "op_graph", "op_coarse", "bsolve", "block", "block_mixed", "eig",
                       "batch", "step"])
    if kind == "spmv":
        return {"call": "spmv", "matrix": rng.choice(["torus", "rgg"]), "size": _logint(rng, 2000, 200000)}
    if kind == "spmv3":
        return {"call": "spmv", "matrix": "fd3d", "size": rng.randint(17, 127)}
    if kind == "op_fd":
        return {"call": "op", "matrix": "fd2d", "size": rng.randint(16, 63), "level": 0,
                "tol": rng.choice([1e-11, 1e-12])}
    if kind == "op_graph":
        return {"call": "op", "matrix": rng.choice(["torus", "rgg"]), "size": _logint(rng, 2000, 150000), "level": 0,
                "tol": rng.choice([1e-11, 1e-12])}
    if kind == "op_coarse":
        return {"call": "op", "matrix": "torus", "size": _logint(rng, 6000, 90000), "level": 1, "tol": 1e-11}
    if kind == "bsolve":
        return {"call": "bsolve", "matrix": "torus", "size": _logint(rng, 6000, 190000), "level": rng.choice([1, 2]),
                "tol": rng.choice([1e-11, 1e-12])}
    if kind == "block":
        return {"call": "block", "matrix": "torus", "size": _logint(rng, 3000, 49000), "level": 0,
                "m": rng.randint(2, 11), "tol": 1e-11, "precision": "fp64"}
    if kind == "block_mixed":
        return {"call": "block", "matrix": "torus", "size": _logint(rng, 3000, 49000), "level": 0,
                "m": rng.randint(8, 50), "tol": 1e-11, "precision": "mixed"}
    if kind == "eig":
        return {"call": "eig", "matrix": "torus", "size": _logint(rng, 3000, 19000), "n_eig": rng.randint(6, 16),
                "tol": 1e-12, "precision": rng.choice(["fp64", "mixed"])}
    if kind == "batch":
        return {"call": "batch", "matrix": "torus", "size": rng.randint(2500, 5900), "count": rng.randint(2, 6),
                "n_eig": rng.randint(4, 8), "tol": 1e-12}
    return {"call": "step", "matrix": "rgg", "size": rng.randint(500, 1450), "n_eig": rng.randint(4, 8), "tol": 1e-12}


# ------------------------------------------------------------------ matrices
def _laplacian(n, i, j, w, shift):
    """CSR (row pointers, columns, values) on the GPU of the Laplacian of the edges i < j, plus shift I."""
    ih, jh, wh = i.cpu().numpy(), j.cpu().numpy(), w.cpu().numpy()
    # degrees on the host: one order of addition, so the same seed gives the same bits
    deg = np.bincount(ih, weights=wh, minlength=n) + np.bincount(jh, weights=wh, minlength=n)
    d = torch.arange(n, device=i.device)
    key, order = torch.sort(torch.cat([i, j, d]) * n + torch.cat([j, i, d]))
    val = torch.cat([-w, -w, torch.from_numpy(deg + shift).to(w.device)])[order]
    rowptr = torch.zeros(n + 1, dtype=torch.int64, device=i.device)
    rowptr[1:] = torch.cumsum(torch.bincount(key // n, minlength=n), 0)
    return rowptr.to(torch.int32), (key % n).to(torch.int32), val


def _near(pts, r, chunk=20000):
    """Every ordered pair (i, j, distance), i != j, of points within r of each other (cells of side r)."""
    n, dim = pts.shape
    cell = torch.floor((pts - pts.min(0).values) / r).to(torch.int64) + 1
    ext = (cell.max(0).values + 2).tolist()
    mul = torch.tensor([math.prod(ext[:a]) for a in range(dim)], device=pts.device)
    key = (cell * mul).sum(1)
    skey, order = torch.sort(key, stable=True)
    around = torch.cartesian_prod(*[torch.arange(-1, 2, device=pts.device)] * dim)
    wanted = key[:, None] + (around * mul).sum(1)[None]
    first = torch.searchsorted(skey, wanted)
    count = torch.searchsorted(skey, wanted, right=True) - first
    out = []
    for c0 in range(0, n, chunk):
        cnt, a = count[c0:c0 + chunk].reshape(-1), first[c0:c0 + chunk].reshape(-1)
        src = torch.arange(c0, min(c0 + chunk, n), device=pts.device).repeat_interleave(count.shape[1])
        i = src.repeat_interleave(cnt)
        pos = torch.arange(i.numel(), device=pts.device) - (torch.cumsum(cnt, 0) - cnt).repeat_interleave(cnt)
        j = order[a.repeat_interleave(cnt) + pos]
        d = ((pts[i] - pts[j]) ** 2).sum(1).sqrt()
        keep = (d <= r) & (i != j)
        out.append((i[keep], j[keep], d[keep]))
    return tuple(torch.cat(t) for t in zip(*out))


def _torus(n, seed, k=10, big=1.0, small=0.3, jitter=1e-3, shift=1e-6):
    rng = np.random.default_rng(seed)
    th = np.empty(0)
    while th.size < n:  # uniform on the surface: rejection on big + small cos(theta)
        t = rng.uniform(0, 2 * math.pi, 2 * n)
        th = np.concatenate([th, t[rng.uniform(0, 1, 2 * n) < (big + small * np.cos(t)) / (big + small)]])
    th, ph = th[:n], rng.uniform(0, 2 * math.pi, n)
    ring = big + small * np.cos(th)
    pts = np.stack([ring * np.cos(ph), ring * np.sin(ph), small * np.sin(th)], 1) + rng.normal(0, jitter, (n, 3))
    # a radius that holds about 5 k points on the surface of area 4 pi^2 big small
    i, j, d = _near(torch.from_numpy(pts).cuda(), math.sqrt(20 * k * math.pi * big * small / n))
    for by in (d, i):  # each point's neighbours, nearest first
        o = torch.argsort(by, stable=True)
        i, j, d = i[o], j[o], d[o]
    cnt = torch.bincount(i, minlength=n)
    keep = torch.arange(i.numel(), device=i.device) - (torch.cumsum(cnt, 0) - cnt)[i] < k
    i, j, d = i[keep], j[keep], d[keep]
    key, at = torch.unique(torch.minimum(i, j) * n + torch.maximum(i, j), return_inverse=True)
    dist = torch.empty(key.numel(), dtype=torch.float64, device=d.device)
    dist[at] = d  # a pair met from both ends has the same distance twice
    sigma = float(np.mean(d.cpu().numpy()))
    return _laplacian(n, key // n, key % n, torch.exp(-(dist / sigma) ** 2), shift)


def _rgg(n, seed, whole, deg=10.0, weights=(0.5, 2.0), shift=1e-6):
    pts = torch.from_numpy(np.random.default_rng(n).uniform(0, 1, (n, 2))).cuda()
    i, j, _ = _near(pts, math.sqrt(deg / (math.pi * n)))
    label = torch.arange(n, device=i.device)
    while not whole:  # connected components: smallest label of the neighbours, then pointer jumping
        new = label.scatter_reduce(0, i, label[j], "amin")
        new = new[new]
        if torch.equal(new, label):
            break
        label = new
    keep = torch.ones_like(label, dtype=torch.bool) if whole else label == torch.bincount(label).argmax()
    number = torch.cumsum(keep, 0) - 1
    e = keep[i] & (i < j)
    i, j, n = number[i[e]], number[j[e]], int(keep.sum())
    key = torch.sort(i * n + j).values
    w = torch.from_numpy(np.random.default_rng(seed).uniform(weights[0], weights[1], key.numel())).cuda()
    return _laplacian(n, key // n, key % n, w, shift)


def _fd(dim, m, seed, lo, hi, box=0.0):
    rng = np.random.default_rng(seed)
    a = 10.0 ** rng.uniform(lo, hi, (m,) * dim)
    if box:  # axis-aligned boxes of sides 4 .. 16 over a tenth of the cells
        inside = np.zeros(a.shape, bool)
        while inside.sum() < 0.1 * a.size:
            side = np.minimum(rng.integers(4, 17, dim), m)
            org = [int(rng.integers(0, m - s + 1)) for s in side]
            inside[tuple(slice(o, o + s) for o, s in zip(org, side))] = True
        a[inside] = box
    a = torch.from_numpy(a).cuda()
    diag, below, above = torch.zeros_like(a), [], []
    for ax in range(dim):
        f = 2 * a.narrow(ax, 0, m - 1) * a.narrow(ax, 1, m - 1) / (a.narrow(ax, 0, m - 1) + a.narrow(ax, 1, m - 1))
        prev, nxt = torch.zeros_like(a), torch.zeros_like(a)
        nxt.narrow(ax, 0, m - 1).copy_(f)
        prev.narrow(ax, 1, m - 1).copy_(f)
        diag += prev + nxt
        for edge in (0, m - 1):
            diag.narrow(ax, edge, 1).add_(a.narrow(ax, edge, 1))
        below.append((-(m ** (dim - 1 - ax)), -prev))
        above.append((m ** (dim - 1 - ax), -nxt))
    entries = below + [(0, diag)] + above[::-1]  # ascending columns
    row = torch.arange(a.numel(), device=a.device)
    col = torch.stack([row + o for o, _ in entries], 1)
    val = torch.stack([v.reshape(-1) for _, v in entries], 1)
    keep = val != 0
    rowptr = torch.zeros(a.numel() + 1, dtype=torch.int64, device=a.device)
    rowptr[1:] = torch.cumsum(keep.sum(1), 0)
    return rowptr.to(torch.int32), col[keep].to(torch.int32), val[keep]


def _matrix(case, seed, size=None):
    size = size or case["size"]
    if case["matrix"] == "fd2d":
        return _fd(2, size, seed, -2.0, 2.0)
    if case["matrix"] == "fd3d":
        return _fd(3, size, seed, -3.0, 3.0, box=1e4)
    if case["matrix"] == "rgg":
        return _rgg(size, seed, whole=case["call"] != "step")
    return _torus(size, size if case.get("level", 0) else seed)


def _batch_sizes(case):
    """Uneven sizes, from the case's largest down to a third of it."""
    return [max(2000, int(case["size"] * (1 - 2 * b / (3 * case["count"])))) for b in range(case["count"])]


def _randn(seed, *shape):
    return torch.randn(*shape, dtype=torch.float64, device="cuda", generator=torch.Generator("cuda").manual_seed(seed))


# ------------------------------------------------------------------ one pass
def prepare(case, seed):
    call, s = case["call"], {"case": case}
    if call == "batch":
        mats = [_matrix(case, seed * 64 + b, n) for b, n in enumerate(_batch_sizes(case))]
        s["handles"] = [G.MMD(*A) for A in mats]
        return s
    A = _matrix(case, seed)
    n = A[0].numel() - 1
    if call == "step":
        # the graph's pattern, its values as the trained tensor, the loss's weights
        s["A"] = A[0], A[1], A[2].requires_grad_(True)
        s["t"] = _randn(seed, n)
        return s
    # products and level-0 solves alone need no levels: the decomposition stops at once
    no_levels = call == "spmv" or (call in ("op", "block") and case["level"] == 0)
    h = s["h"] = G.MMD(*A, k_max=0) if no_levels else G.MMD(*A)
    if call == "eig":
        s["out"] = (torch.zeros(case["n_eig"], dtype=torch.float64, device="cuda"),
                    torch.zeros((case["n_eig"], n), dtype=torch.float64, device="cuda"))
        return s
    if call == "op":
        n = h.level_size(case["level"])
    elif call == "bsolve":
        n = h.level_size(case["level"] - 1)
    s["x"] = _randn(seed, case["m"], n) if call == "block" else _randn(seed, n)
    s["y"] = torch.zeros_like(s["x"])
    return s


def run(s):
    case = s["case"]
    call = case["call"]
    stream = torch.cuda.current_stream().cuda_stream
    if call == "batch":
        return [(lam, V) for lam, V, _ in G.eig_leftmost_batched(s["handles"], case["n_eig"], case["tol"], streams=3)]
    if call == "step":
        rowptr, col, val = s["A"]
        val.grad = None
        lam, V = G.eigsh_leftmost(rowptr, col, val, case["n_eig"], case["tol"], stream=stream)
        (lam.sum() + 0.5 * (s["t"] * V[:, 1] ** 2).sum()).backward()
        return lam.detach(), V.detach(), val.grad
    h = s["h"]
    if call == "eig":
        lam, V, _ = h.eig_leftmost(case["n_eig"], case["tol"], out=s["out"], stream=stream,
                                   precision=PRECISION[case["precision"]])
        return lam, V
    if call == "spmv":
        h.level_spmv(0, 0, s["x"], s["y"], stream=stream)
    elif call == "op":
        h.level_op(case["level"], s["x"], s["y"], case["tol"], stream=stream)
    elif call == "bsolve":
        h.level_bsolve(case["level"], s["x"], s["y"], case["tol"], stream=stream)
    else:
        h.level_op_block(case["level"], s["x"], s["y"], case["tol"], precision=PRECISION[case["precision"]],
                         stream=stream)
    return s["y"]


# ------------------------------------------------------------------ work
def _sizes(case, size=None):
    """(n, nnz) of the case's matrix (graphs: their mean row lengths)."""
    m = size or case["size"]
    if case["matrix"] in ("fd2d", "fd3d"):
        dim = int(case["matrix"][2])
        return m ** dim, m ** dim + 2 * dim * (m - 1) * m ** (dim - 1)
    return m, int((12.4 if case["matrix"] == "torus" else 10.9) * m)


def _cg(case, n):
    """About how many CG iterations one solve on the level-0 matrix takes at these tolerances."""
    return (34 if case["matrix"] == "fd2d" else 7 if case["matrix"] == "torus" else 20) * math.sqrt(n)


def work(case):
    call = case["call"]
    if call == "batch":
        parts = [work({**case, "call": "eig", "size": n}) for n in _batch_sizes(case)]
        return {k: sum(p[k] for p in parts) for k in ("bytes", "flops")}
    n, nnz = _sizes(case)
    matrix = 12 * nnz + 4 * n  # values and columns, row pointers, once
    iteration = 2 * nnz + 10 * n  # one product, two dot products and three updates
    if call == "spmv":
        return {"bytes": matrix + 16 * n, "flops": 2 * nnz}
    if call == "bsolve":  # on U^T A^(k-1) U, whose conditioning the decomposition bounds: about 100 iterations
        shrink = 11 ** (case["level"] - 1)
        return {"bytes": (matrix + 16 * n) / shrink, "flops": 100 * (iteration + 4 * n) / shrink}
    if call == "op" and case["level"] >= 1:  # A^(1), M^(1) on n / 11 rows of about 55 entries: 230 x 11 products
        nk = n / 11
        return {"bytes": nk * (2 * 12 * 55 + 16), "flops": 230 * 11 * nk * (2 * 55 + 10)}
    if call in ("op", "block"):
        m = case.get("m", 1)
        return {"bytes": matrix + 16 * n * m, "flops": m * _cg(case, n) * iteration}
    # eigensolves: about four Lanczos steps a pair, each a solve (a third of a random vector's iterations saved)
    solves = 4 * case["n_eig"] + (30 if call == "step" else 0)
    return {"bytes": matrix * (2 if call == "step" else 1) + 8 * n * case["n_eig"] * (2 if call == "step" else 1),
            "flops": solves * 0.65 * _cg(case, n) * iteration}


# ------------------------------------------------------------------ 64-bit results
def _csr(A):
    return torch.sparse_csr_tensor(A[0].to(torch.int64), A[1].to(torch.int64), A[2], (A[0].numel() - 1,) * 2)


def _solve(A, B):
    """A^{-1} B, B (n, m): dense Cholesky and refinement, or above 12,000 rows restarted conjugate gradients."""
    S, n = _csr(A), A[0].numel() - 1
    if n <= 12000:
        L = torch.linalg.cholesky(S.to_dense())
        X = torch.cholesky_solve(B, L)
        for _ in range(3):
            X = X + torch.cholesky_solve(B - S @ X, L)
        return X
    X = torch.zeros_like(B)
    for tol in (1e-13, 1e-3, 1e-3):  # the residual itself is solved for again
        R = B - S @ X
        P, rr = R.clone(), (R * R).sum(0)
        goal = tol * tol * rr
        for it in range(20000):
            Q = S @ P
            al = rr / (P * Q).sum(0)
            X += al * P
            R -= al * Q
            new = (R * R).sum(0)
            P = R + (new / rr) * P
            rr = new
            if it % 50 == 0 and bool((rr <= goal).all()):
                break
    return X


def _lowest(A, N):
    """(lambda ascending, V with a positive largest entry) of the N leftmost pairs: subspace iteration with A^{-1}."""
    D = _csr(A).to_dense()
    n = D.shape[0]
    L = torch.linalg.cholesky(D)
    S = _csr(A)
    Q = torch.linalg.qr(_randn(7, n, min(n, 4 * N + 16))).Q
    old = None
    for _ in range(200):
        Q = torch.linalg.qr(torch.cholesky_solve(Q, L)).Q
        w, P = torch.linalg.eigh(Q.T @ (S @ Q))
        Q = Q @ P
        V = Q[:, :N]
        if old is not None and float((V - old * torch.sign((old * V).sum(0))).norm(dim=0).max()) < 1e-14 * math.sqrt(n):
            break
        old = V
    top = V.gather(0, V.abs().argmax(0)[None])[0]
    return w[:N], V * torch.sign(top)


def exact(case, seed):
    call = case["call"]
    if call == "bsolve" or case.get("level", 0) >= 1:
        return None  # on the decomposition's own matrices
    if call == "batch":
        out = [_lowest(_matrix(case, seed * 64 + b, n), case["n_eig"]) for b, n in enumerate(_batch_sizes(case))]
        return [(lam.cpu().numpy(), V.cpu().numpy()) for lam, V in out]
    A = _matrix(case, seed)
    n = A[0].numel() - 1
    if call == "spmv":
        return _csr(A) @ _randn(seed, n)
    if call == "op":
        return _solve(A, _randn(seed, n)[:, None])[:, 0]
    if call == "block":
        return _solve(A, _randn(seed, case["m"], n).T.contiguous()).T.contiguous()
    if call == "eig":
        lam, V = _lowest(A, case["n_eig"])
        return lam, V.T.contiguous()
    # the loss's gradient from all eigenpairs of the dense matrix
    N, t = case["n_eig"], _randn(seed, n)
    w, E = torch.linalg.eigh(_csr(A).to_dense())
    V = E[:, :N]
    V = V * torch.sign(V.gather(0, V.abs().argmax(0)[None])[0])
    v = V[:, 1]
    c = (E.T @ (t * v)) / (w[1] - w)
    c[1] = 0.0
    y = E @ c
    rows = torch.repeat_interleave(torch.arange(n, device=v.device), (A[0][1:] - A[0][:-1]).to(torch.int64))
    cols = A[1].to(torch.int64)
    grad = (V[rows] * V[cols]).sum(1) + y[rows] * v[cols]
    return w[:N], V, grad
