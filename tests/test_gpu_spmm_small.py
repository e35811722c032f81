"""s_spmm on matrices of few block rows, where rows of more than 32 blocks are shared by a cluster of CTAs:
around that length, and around the two rows per SM (304) up to which it holds; empty clusters and
rows of several panels among them.  Tolerance as in test_gpu_spmm_rows.py."""
import numpy as np
import pytest

import workloads as W
from tests.gpu_util import dev, host, rel_frob
from tests.test_gpu_spmm_rows import arrow, dense_of

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nc, width", [(32, 40), (33, 40), (34, 40), (100, 17), (304, 16), (305, 16), (304, 40), (305, 40)])
def test_rows_around_32_blocks(nc, width):
    import torch
    from paper_2211_11681_gb300 import sformat as sf
    bsize, rowptr, colidx, full = arrow(nc, [5, 20, 33, 1], min(width, nc - 1))
    bsize[7] = 0
    full[7, :] = full[:, 7] = False
    rowptr, colidx = np.concatenate([[0], np.cumsum(full.sum(1))]), np.nonzero(full)[1]
    P = sf.Pattern(np.concatenate([[0], np.cumsum(bsize)]), np.zeros(nc, dtype=np.int32), rowptr, colidx)
    vals = W.random_values(P.nnz, nc)
    M = dense_of(bsize, full, vals)
    n = M.shape[0]
    for k in (1, 3, 16):
        X = W.random_values(n * k, 5 + k).reshape(k, n)
        Y, Z = dev(np.full((k, n), np.nan)), dev(np.zeros((k, n)))
        sf.spmm(P, dev(vals), dev(X), Y)
        assert rel_frob(host(Y), X @ M.T) <= 1e-13, k
        sf.spmm(P, dev(vals), dev(X), Z)
        assert torch.equal(Y, Z)
