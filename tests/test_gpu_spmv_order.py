"""The one-column product (mmd_level_spmv) in the caller's order, in a permuted device order, and onto its own input.

Each entry is a sum of products of a row's length, so it is held to (length + 1) units of rounding of the sum of its
terms' magnitudes."""
import numpy as np
import pytest
import scipy.sparse as sp

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 33, 1500, 20001])
@pytest.mark.parametrize("scattered", [False, True])
def test_spmv_orders(n, scattered):
    import torch

    import paper_1804_03415_gb300 as G

    rng = np.random.default_rng(n)
    i = np.arange(n)
    far = rng.permutation(n) if scattered else np.minimum(i + 3, n - 1)
    W = sp.coo_matrix((rng.uniform(0.5, 2.0, n), (i, far)), shape=(n, n))
    W = (W + W.T).tocsr()
    A = (sp.diags(np.asarray(W.sum(1)).ravel() + 1.0) - W).tocsr()
    A.sort_indices()
    h = G.MMD(A.indptr.astype(np.int32), A.indices.astype(np.int32), A.data, k_max=0)
    xh = rng.standard_normal(n)
    x = torch.from_numpy(xh).cuda()
    y = torch.zeros_like(x)
    h.level_spmv(0, 0, x, y)
    bound = (np.diff(A.indptr) + 1) * np.finfo(float).eps * (abs(A) @ abs(xh))
    assert np.all(np.abs(y.cpu().numpy() - A @ xh) <= bound)
    h.level_spmv(0, 0, x, x)
    assert np.array_equal(x.cpu().numpy(), y.cpu().numpy())
    h.close()
