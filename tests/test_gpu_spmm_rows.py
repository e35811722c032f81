"""s_spmm at the edges of its row kernel: a row long enough to be shared by a cluster of CTAs (more
than 256 blocks) next to short and empty rows, blocks of one and several panels and pieces,
vector counts around its ten at a time; and the norm estimate on such a pattern.

Tolerance 1e-13 relative: double sums of at most 12,000 products of [-1, 1] values in another order
(2^-53 times the square root of the length, times ten for cancellation)."""
import numpy as np
import pytest

import workloads as W
from tests.gpu_util import dev, host, rel_frob

pytestmark = pytest.mark.gpu


def arrow(nc, sizes, width):
    """Symmetric arrow-and-band pattern: a full first block row and column, `width` bands."""
    bsize = np.array([sizes[i % len(sizes)] for i in range(nc)])
    full = np.zeros((nc, nc), dtype=bool)
    for k in range(width + 1):
        i = np.arange(nc - k)
        full[i, i + k] = full[i + k, i] = True
    full[0, :] = full[:, 0] = True
    full[bsize == 0, :] = False
    full[:, bsize == 0] = False
    rowptr = np.concatenate([[0], np.cumsum(full.sum(1))])
    return bsize, rowptr, np.nonzero(full)[1], full


def dense_of(bsize, full, vals):
    off = np.concatenate([[0], np.cumsum(bsize)])
    M = np.zeros((off[-1], off[-1]))
    p = 0
    for i, j in zip(*np.nonzero(full)):
        m = bsize[i] * bsize[j]
        M[off[i]:off[i + 1], off[j]:off[j + 1]] = vals[p:p + m].reshape(bsize[i], bsize[j])
        p += m
    return M


@pytest.mark.parametrize("sizes", [[20, 3, 10, 0, 7], [41, 1, 12, 20], [1], [10]], ids=str)
@pytest.mark.parametrize("nc", [40, 600])
def test_spmm_rows_and_vectors(sizes, nc):
    import torch
    from paper_2211_11681_gb300 import sformat as sf
    bsize, rowptr, colidx, full = arrow(nc, sizes, 3)
    P = sf.Pattern(np.concatenate([[0], np.cumsum(bsize)]), np.zeros(nc, dtype=np.int32), rowptr, colidx)
    vals = W.random_values(P.nnz, 11)
    M = dense_of(bsize, full, vals)
    n = M.shape[0]
    for k in (1, 2, 9, 10, 11, 23):
        X = W.random_values(n * k, 12 + k).reshape(k, n)
        Y = dev(np.full((k, n), np.nan))
        sf.spmm(P, dev(vals), dev(X), Y)
        assert rel_frob(host(Y), X @ M.T) <= 1e-13, k
        Z = torch.zeros_like(Y)
        sf.spmm(P, dev(vals), dev(X), Z)
        np.testing.assert_array_equal(host(Z), host(Y))
    # power iteration on M M^T's symmetric part: a symmetric matrix on the symmetric pattern
    S = dense_of(bsize, full, vals)
    S = 0.5 * (S + S.T) + 40.0 * np.eye(n)
    off = np.concatenate([[0], np.cumsum(bsize)])
    sv = np.concatenate([S[off[i]:off[i + 1], off[j]:off[j + 1]].ravel() for i, j in zip(*np.nonzero(full))])
    x = np.full(n, 1.0 / np.sqrt(n))
    for _ in range(50):
        y = S @ x
        lam = x @ y
        x = y / np.linalg.norm(y)
    assert sf.norm_est(P, dev(sv), 50) == pytest.approx(lam, rel=1e-11)
