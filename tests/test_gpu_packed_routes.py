"""Routes of the packed float product that share one packed copy, read unaligned values or list range by
range: each does the same sums in the same order as the general route, so its results are
equal to the bit.  (That the general route is right is test_gpu_packed_float.py's.)"""
import numpy as np
import pytest

from oracle import product as oprod
from oracle.sformat import BlockCSR
from tests.gpu_util import dev, host, pattern_of, rel_frob
from tests.test_gpu_packed_float import SIZES
from tests.test_gpu_product import drop_empty
from tests.test_oracle_product import random_bcsr

pytestmark = pytest.mark.gpu


def symmetric(bsize, fill, seed):
    """A symmetric matrix on a symmetric random pattern."""
    X = drop_empty(random_bcsr(bsize, fill, seed))
    nc = len(bsize)
    M = np.zeros((nc, nc), dtype=bool)
    M[X.brow, X.colidx] = True
    M |= M.T
    Y = BlockCSR(bsize, np.concatenate([[0], np.cumsum(M.sum(axis=1))]), np.nonzero(M)[1])
    D = X.to_dense()
    D = D + D.T
    for k in range(Y.nblocks):
        i, j = Y.brow[k], Y.colidx[k]
        Y.val[Y.voff[k]:Y.voff[k + 1]] = D[Y.boff[i]:Y.boff[i + 1], Y.boff[j]:Y.boff[j + 1]].ravel()
    return Y


@pytest.mark.parametrize("sizes", SIZES, ids=lambda s: "-".join(map(str, s)))
@pytest.mark.parametrize("fill", [1.0, 0.4])
def test_one_copy_of_a_symmetric_matrix(sizes, fill):
    from paper_2211_11681_gb300 import sformat as sf
    A = symmetric(np.array(sizes * 6), fill, sum(sizes) + 7)
    P = pattern_of(A)
    a = dev(A.val, "float32")
    general, sym = sf.Plan(P, P, P, "fp32"), sf.Plan(P, P, P, "fp32")
    sym.set_symmetric_a(True)
    want, got, tiled = (dev(np.full(len(A.val), np.nan), "float32") for _ in range(3))
    general.mul(a, a, want)
    sym.mul(a, a, got)
    np.testing.assert_array_equal(host(got), host(want))
    ref = oprod.mul_masked(A, A, A, nthreads=8).val
    assert rel_frob(host(want), ref) <= 1e-5  # the bound of the other random-pattern float tests
    # another B: not read through A's rows; the tile kernel, whose sums run in another order
    sym.mul(a, a.clone(), tiled)
    assert rel_frob(host(tiled), ref) <= 1e-5
    assert not np.array_equal(host(tiled), host(want))
    sym.set_symmetric_a(False)
    got.fill_(float("nan"))
    sym.mul(a, a.clone(), got)
    np.testing.assert_array_equal(host(got), host(want))


def test_values_off_16_bytes():
    import torch
    from paper_2211_11681_gb300 import sformat as sf
    bsize = np.array(SIZES[2] * 6)
    A = drop_empty(random_bcsr(bsize, 0.5, 91))
    P = pattern_of(A)
    plan = sf.Plan(P, P, P, "fp32")
    n = len(A.val)
    a, b = dev(A.val, "float32"), dev(A.val[::-1], "float32")
    want = dev(np.full(n, np.nan), "float32")
    plan.mul(a, b, want)
    for off in (1, 2, 3):
        x, y, z = (torch.full((n + 4,), float("nan"), device="cuda") for _ in range(3))
        x[off:off + n], y[4 - off:4 - off + n] = a, b
        plan.mul(x[off:off + n], y[4 - off:4 - off + n], z[off:off + n])
        np.testing.assert_array_equal(host(z[off:off + n]), host(want))
        assert int(torch.isnan(z).sum()) == 4  # nothing written around it


def test_range_by_range():
    # 700 clusters of 1 and 2 rows, every block present: 3.4e8 block triples, 5.5 GB of lists, more than a
    # plan keeps.  Forward (general, symmetric, from a graph) and both adjoints against dense products.
    import torch
    from paper_2211_11681_gb300 import sformat as sf
    nc = 700
    bsize = 1 + np.arange(nc) % 2
    boff = np.concatenate([[0], np.cumsum(bsize)])
    P = sf.Pattern(boff, np.zeros(nc, dtype=np.int32), np.arange(nc + 1) * nc, np.tile(np.arange(nc), nc))
    n = int(boff[-1])
    row = np.repeat(np.arange(nc), bsize)
    order = np.lexsort((np.tile(np.arange(n), n), np.repeat(np.arange(n), n), np.tile(row, n), np.repeat(row, n)))
    rng = np.random.Generator(np.random.PCG64(4))
    M, G = (rng.uniform(-1, 1, size=(n, n)) for _ in range(2))
    M = (M + M.T).astype(np.float32).astype(np.float64)
    G = G.astype(np.float32).astype(np.float64)
    stored = lambda m: np.ascontiguousarray(m.ravel()[order])  # block-CSR values
    a, g = dev(stored(M), "float32"), dev(stored(G), "float32")
    new = lambda: dev(np.full(n * n, np.nan), "float32")
    free0 = torch.cuda.mem_get_info()[0]
    plan = sf.Plan(P, P, P, "fp32")
    assert 16 * plan.stats()[0] > 4 << 30
    assert free0 - torch.cuda.mem_get_info()[0] < 1 << 30  # a workspace, not the lists
    out = new()
    plan.mul(a, a, out)
    assert rel_frob(host(out), stored(M @ M)) <= 1e-5
    again = new()
    graph = plan.graph(a, a, again)
    graph.launch()
    graph.launch()
    torch.cuda.synchronize()
    np.testing.assert_array_equal(host(again), host(out))
    del graph
    dA, dB = new(), new()
    plan.adjoint(g, a, a, dA, dB)
    assert rel_frob(host(dA), stored(G @ M.T)) <= 1e-5
    assert rel_frob(host(dB), stored(M.T @ G)) <= 1e-5
    plan.set_symmetric_a(True)
    again.fill_(float("nan"))
    plan.mul(a, a, again)
    np.testing.assert_array_equal(host(again), host(out))


@pytest.mark.parametrize("nc", [120, 121, 139, 140])
def test_small_and_large_launches(nc):
    # around the lines where tiles are taken ahead (14592 tiles on 152 SMs) and where a block has a warp
    # of its own in the packing (19456 blocks): nc^2 blocks of 1 to 3 rows and columns
    from paper_2211_11681_gb300 import sformat as sf
    bsize = 1 + np.arange(nc) % 3
    A, B = random_bcsr(bsize, 1.0, nc), random_bcsr(bsize, 1.0, nc + 1)
    P = pattern_of(A)
    plan = sf.Plan(P, P, P, "fp32")
    out = dev(np.full(len(A.val), np.nan), "float32")
    plan.mul(dev(A.val, "float32"), dev(B.val, "float32"), out)
    assert rel_frob(host(out), oprod.mul_masked(A, B, A, nthreads=8).val) <= 1e-5
