"""Selected inversion where its sums are split: a full pattern (a chain of levels, each with few
output blocks and long sums: several warps and CTAs to a sum, the diagonal sums shared by a
cluster of CTAs) and a band (many short sums: a warp per item), with blocks narrower than, equal
to and wider than one 20 x 20 tile.  Against numpy's inverse.

Tolerance 1e-12 relative (maximum entry): both are FP64 solves of diagonally dominant matrices
with condition numbers below 10, tens of units in the last place apart."""
import numpy as np
import pytest

from tests.gpu_util import dev, host, pattern_of

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sizes", [[10], [10, 6, 21, 1], [41, 20, 64, 3], [5, 0, 12]], ids=str)
@pytest.mark.parametrize("nc,band", [(3, 2), (90, 89), (200, 2)])
def test_split_sums(sizes, nc, band):
    from oracle.sformat import BlockCSR
    from paper_2211_11681_gb300.selinv import SelInv
    bsize = np.array([sizes[i % len(sizes)] for i in range(nc)])
    if bsize.sum() > 3000:
        bsize = bsize[:40]
        nc, band = 40, min(band, 39)
    i, j = np.meshgrid(np.arange(nc), np.arange(nc), indexing="ij")
    full = (np.abs(i - j) <= band) & (bsize[:, None] > 0) & (bsize[None, :] > 0)
    rowptr = np.concatenate([[0], np.cumsum(full.sum(1))])
    colidx = np.nonzero(full)[1]
    rng = np.random.Generator(np.random.PCG64(sum(sizes) + nc))
    n = int(bsize.sum())
    D = rng.uniform(-1, 1, size=(n, n))
    mask = np.repeat(np.repeat(full, bsize, axis=0), bsize, axis=1)
    D = 0.5 * (D + D.T) * mask
    D += np.diag(2.0 * np.abs(D).sum(axis=1) + 1.0)
    A = BlockCSR.from_dense(D, bsize, rowptr, colidx)
    inv = SelInv(pattern_of(A))
    Z = dev(np.full(len(A.val), np.nan))
    inv.factor(dev(A.val), 0.25)
    inv.invert(Z)
    inv.status()
    want = BlockCSR.from_dense(np.linalg.inv(D + 0.25 * np.eye(n)), bsize, rowptr, colidx).val
    assert np.abs(host(Z) - want).max() <= 1e-12 * np.abs(want).max()
    again = dev(np.zeros(len(A.val)))
    inv.factor(dev(A.val), 0.25)
    inv.invert(again)
    np.testing.assert_array_equal(host(again), host(Z))
