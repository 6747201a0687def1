"""FP64 CG on one right-hand side (mmd_level_op at level 0 without a decomposition) where its launch changes shape:
around a SELL slice and the cluster's sixteen blocks, at the change from the cluster to the grid, with rows much wider
than the others, with several components, and where the rows do not fit the shared memory of the SMs.

Well-conditioned matrices (Laplacian + I): the recurrence's residual and the true one then differ by rounding only, a few
hundred ulps of ||b|| against a tolerance of 1e-10, so the true residual is held to twice the tolerance, and the solution
(||A^{-1}|| <= 1) to twice the tolerance of ||b|| from the direct one."""
import numpy as np
import pytest
import scipy.sparse as sp
import scipy.sparse.linalg as spl

pytestmark = pytest.mark.gpu
TOL = 1e-10


def laplacian(n, i, j, seed):
    w = np.random.default_rng(seed).uniform(0.5, 2.0, len(i))
    W = sp.coo_matrix((w, (i, j)), shape=(n, n))
    W = (W + W.T).tocsr()
    W.setdiag(0)
    W.eliminate_zeros()
    return (sp.diags(np.asarray(W.sum(1)).ravel() + 1.0) - W).tocsr()


def matrix(kind, n):
    rng = np.random.default_rng(n)
    i = np.arange(n)
    if kind == "diag":
        return sp.diags(rng.uniform(1.0, 3.0, n)).tocsr()
    if kind == "path":  # numbered at random
        p = rng.permutation(n)
        return laplacian(n, p[:-1], p[1:], 1)
    if kind == "hub":  # a few rows as wide as the matrix
        return laplacian(n, np.concatenate([i, i]), np.concatenate([np.full(n, n // 2), (i * 7 + 3) % n]), 2)
    if kind == "parts":  # components of 50 rows, interleaved
        q = max(1, n // 50)
        return laplacian(n, i[:-q], i[q:], 3)
    return laplacian(n, np.repeat(i, 6), rng.integers(0, n, 6 * n), 4)  # random graph


def solve(A, b):
    import torch

    import paper_1804_03415_gb300 as G

    A = sp.csr_matrix(A)
    A.sort_indices()
    h = G.MMD(A.indptr.astype(np.int32), A.indices.astype(np.int32), A.data, k_max=0)
    x = torch.from_numpy(b).cuda()
    y = torch.zeros_like(x)
    h.level_op(0, x, y, TOL)
    first = y.cpu().numpy()
    y.zero_()
    h.level_op(0, x, y, TOL)
    assert np.array_equal(first, y.cpu().numpy())
    h.close()
    return first


@pytest.mark.parametrize("kind,n", [
    ("diag", 1), ("path", 2), ("path", 31), ("rand", 32), ("rand", 33), ("path", 511), ("rand", 513), ("parts", 1000),
    ("hub", 700), ("hub", 6000), ("rand", 3000), ("rand", 9000), ("path", 20000), ("diag", 40000), ("parts", 60001)])
def test_own_cg(kind, n):
    A = matrix(kind, n)
    b = np.random.default_rng(5).standard_normal(n)
    x = solve(A, b)
    nb = np.linalg.norm(b)
    assert np.linalg.norm(b - A @ x) <= 2 * TOL * nb
    if n <= 3000:
        assert np.linalg.norm(x - spl.spsolve(A.tocsc(), b)) <= 2 * TOL * nb


def test_own_cg_zero_rhs():
    assert not solve(matrix("rand", 100), np.zeros(100)).any()


def test_own_cg_beyond_shared_memory():
    """More rows than the SMs' shared memory holds: the general kernel, the same answer."""
    A = matrix("path", 1_200_000)
    b = np.random.default_rng(6).standard_normal(A.shape[0])
    assert np.linalg.norm(b - A @ solve(A, b)) <= 2 * TOL * np.linalg.norm(b)


@pytest.mark.parametrize("blocks", range(3, 17))
def test_own_cg_cluster_sizes(blocks):
    """Every cluster size from 3 to 16 blocks (a block per SELL slice of 32 rows), the last slice ragged; rows of one
    entry leave a block nothing to do before the sums that cross the cluster."""
    for kind in ("rand", "path", "diag"):
        n = 32 * blocks - 5
        A = matrix(kind, n)
        b = np.random.default_rng(blocks).standard_normal(n)
        x = solve(A, b)
        nb = np.linalg.norm(b)
        assert np.linalg.norm(b - A @ x) <= 2 * TOL * nb
        assert np.linalg.norm(x - spl.spsolve(A.tocsc(), b)) <= 2 * TOL * nb


def kernels_of(call):
    """Names of the kernels that a call launches; skips where the tracer gives none."""
    import torch
    from torch.profiler import ProfilerActivity, profile

    names = set()
    for _ in range(3):  # the first trace of a process may hold nothing
        with profile(activities=[ProfilerActivity.CUDA]) as p:
            call()
            torch.cuda.synchronize()
        names |= {e.key for e in p.key_averages()}
    if not any("kernel" in s for s in names):
        pytest.skip("no kernel records on this machine")
    return names


@pytest.mark.parametrize("kind,n,kernel", [
    ("path", 33, "own_cg_kernel<true>"), ("rand", 3000, "own_cg_kernel<true>"), ("rand", 9000, "own_cg_kernel<false>"),
    ("path", 200000, "own_cg_kernel<false>"), ("hub", 20000, "solve_kernel<1, double, 0>"),
    ("path", 600000, "solve_kernel<1, double, 0>")])
def test_which_kernel(kind, n, kernel):
    import torch

    import paper_1804_03415_gb300 as G

    A = sp.csr_matrix(matrix(kind, n))
    A.sort_indices()
    h = G.MMD(A.indptr.astype(np.int32), A.indices.astype(np.int32), A.data, k_max=0)
    x = torch.ones(n, dtype=torch.float64, device="cuda")
    y = torch.zeros_like(x)
    ran = kernels_of(lambda: h.level_op(0, x, y, TOL))
    assert any(kernel in s for s in ran), ran
    assert sum("own_cg" in s or "solve_kernel" in s for s in ran) == 1, ran
    h.close()


@pytest.mark.parametrize("n", [400, 6000])
def test_wait_runs_out_then_recovers(n):
    """Lanczos with plain CG on a handle without levels: its first device waits are those of the one-column launch, on a
    cluster and on a grid.  They give up after the limit, the call says so, and the handle solves on."""
    import workloads as W

    import paper_1804_03415_gb300 as G

    A = W.random_spd_mmatrix(n, 6, seed=9, shift=0.5)
    h = G.MMD(A.rowptr, A.col, A.val, k_max=0)
    for _ in range(2):
        with pytest.raises(G.MMDError) as ei:
            h.eig_leftmost(4, 1e-8, method=G.MMD_IRLM_CG, timeout_s=1e-9)
        assert ei.value.code == G._lib.MMD_ETIMEOUT
        lam, V, st = h.eig_leftmost(4, 1e-8, method=G.MMD_IRLM_CG)
        assert st["max_rel_residual"] <= 10 * 1e-8
    h.close()
