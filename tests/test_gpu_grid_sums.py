"""The fenced grid-wide sum of the persistent solver over small grids (tagged words) and large ones (arrival counter).

A block of three columns on a handle without levels runs one tile on ceil(n / 1024) blocks, at least 16.  Matrices are
Laplacians + I (||A^{-1}|| <= 1), as in the one-column tests: the true residual is held to twice the tolerance.  The sum
is also the barrier behind which blocks read each other's rows, so two runs have to agree in every bit."""
import numpy as np
import pytest
import scipy.sparse as sp

from test_gpu_own_cg import TOL, matrix

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("blocks", [16, 17, 21, 25, 26, 50, 101, 144, 145, 152])
def test_fenced_sums(blocks):
    import torch

    import paper_1804_03415_gb300 as G

    n = 1024 * blocks - 11
    A = sp.csr_matrix(matrix("path", n))
    A.sort_indices()
    h = G.MMD(A.indptr.astype(np.int32), A.indices.astype(np.int32), A.data, k_max=0)
    B = np.random.default_rng(blocks).standard_normal((3, n))
    X = torch.from_numpy(B).cuda()
    Y = torch.zeros_like(X)
    h.level_op_block(0, X, Y, TOL)
    first = Y.cpu().numpy()
    Y.zero_()
    h.level_op_block(0, X, Y, TOL)
    assert np.array_equal(first, Y.cpu().numpy())
    for b, x in zip(B, first):
        assert np.linalg.norm(b - A @ x) <= 2 * TOL * np.linalg.norm(b)
    h.close()
