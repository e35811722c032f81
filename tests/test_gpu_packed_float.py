"""The packed float product and the dealt double product at the sizes where its tiles, pieces and lists change: tile edges around
the micro-tile classes (6, 10, 12, 16, 20), blocks of several panels and several t pieces, odd
widths (padded t pairs), and a plan whose lists exceed what it keeps, so that every product goes
through ranges of blocks.  Against the FP64 oracle, forward and adjoint, general and symmetric.

Tolerance 1e-5 relative Frobenius on uniform [-1, 1] values (float rounding 6e-8 per operation,
about tenfold cancellation in these sums), the bound of the other random-pattern float tests; 1e-12 in
double."""
import numpy as np
import pytest

import workloads as W
from oracle import adjoint as oadj
from oracle import product as oprod
from tests.gpu_util import dev, host, pattern_of, rel_frob
from tests.test_gpu_product import drop_empty
from tests.test_oracle_product import random_bcsr

pytestmark = pytest.mark.gpu

SIZES = [
    [1, 2, 3, 4, 5, 6, 7],                    # micro-tile classes 6 and 10, one t pair and odd widths
    [9, 10, 11, 10, 12, 13, 10],              # around 10 and 12: 8, 4 and 2 blocks to a step
    [15, 16, 17, 19, 20, 21, 20],             # around 16 and 20: one and two panels
    [39, 40, 41, 1, 10, 20, 61],              # several panels and t pieces next to narrow blocks
    [0, 20, 0, 5, 33, 0, 10],                 # empty clusters
]


@pytest.mark.parametrize("sizes", SIZES, ids=lambda s: "-".join(map(str, s)))
@pytest.mark.parametrize("fill", [1.0, 0.4])
def test_tile_and_piece_edges(sizes, fill):
    from paper_2211_11681_gb300 import sformat as sf
    seed = sum(sizes)
    bsize = np.array(sizes * 6)
    A = drop_empty(random_bcsr(bsize, fill, seed))
    B = drop_empty(random_bcsr(bsize, fill, seed + 1, diag=False))
    C = drop_empty(random_bcsr(bsize, fill, seed + 2, diag=False))
    want = oprod.mul_masked(A, B, C, nthreads=8).val
    plan = sf.Plan(pattern_of(A), pattern_of(B), pattern_of(C), "fp32")
    out = dev(np.full(len(C.val), np.nan), "float32")
    plan.mul(dev(A.val, "float32"), dev(B.val, "float32"), out)
    assert rel_frob(host(out), want) <= 1e-5
    dC = C.like(W.random_values(len(C.val), seed + 3))
    wA, wB = oadj.mul_masked_adjoint(dC, A, B)
    gA, gB = dev(np.full(len(A.val), np.nan), "float32"), dev(np.full(len(B.val), np.nan), "float32")
    plan.adjoint(dev(dC.val, "float32"), dev(A.val, "float32"), dev(B.val, "float32"), gA, gB)
    assert rel_frob(host(gA), wA.val) <= 1e-5
    assert rel_frob(host(gB), wB.val) <= 1e-5


@pytest.mark.parametrize("sizes", SIZES, ids=lambda s: "-".join(map(str, s)))
@pytest.mark.parametrize("fill", [1.0, 0.4])
def test_double_product_deals(sizes, fill):
    # the double product deals 8, 4 or 2 lambda blocks (pieces of at most 10 or 20) to the lanes:
    # every tile class, both tile edges, forward and both transposes; 1e-12 as the other
    # double tests (another summation order of at most a few thousand products)
    from paper_2211_11681_gb300 import sformat as sf
    seed = sum(sizes) + 50
    bsize = np.array(sizes * 6)
    A = drop_empty(random_bcsr(bsize, fill, seed))
    B = drop_empty(random_bcsr(bsize, fill, seed + 1, diag=False))
    C = drop_empty(random_bcsr(bsize, fill, seed + 2, diag=False))
    want = oprod.mul_masked(A, B, C, nthreads=8).val
    plan = sf.Plan(pattern_of(A), pattern_of(B), pattern_of(C), "fp64")
    for v in range(plan.num_variants()):
        plan.set_variant(v)
        out = dev(np.full(len(C.val), np.nan))
        plan.mul(dev(A.val), dev(B.val), out)
        assert rel_frob(host(out), want) <= 1e-12, v
    dC = C.like(W.random_values(len(C.val), seed + 3))
    wA, wB = oadj.mul_masked_adjoint(dC, A, B)
    gA, gB = dev(np.full(len(A.val), np.nan)), dev(np.full(len(B.val), np.nan))
    plan.adjoint(dev(dC.val), dev(A.val), dev(B.val), gA, gB)
    assert rel_frob(host(gA), wA.val) <= 1e-12
    assert rel_frob(host(gB), wB.val) <= 1e-12


def test_lists_beyond_what_a_plan_keeps():
    # 700 clusters of 1 and 2 rows, every block present: 3.4e8 block triples, 5.5 GB of lists, so the
    # product runs range by range; the dense product is the reference
    from paper_2211_11681_gb300 import sformat as sf
    nc = 700
    bsize = 1 + np.arange(nc) % 2
    boff = np.concatenate([[0], np.cumsum(bsize)])
    rowptr = np.arange(nc + 1) * nc
    colidx = np.tile(np.arange(nc), nc)
    P = sf.Pattern(boff, np.zeros(nc, dtype=np.int32), rowptr, colidx)
    n = int(boff[-1])
    rng = np.random.Generator(np.random.PCG64(3))
    M = rng.uniform(-1, 1, size=(n, n)).astype(np.float32)
    row = np.repeat(np.arange(nc), bsize)

    def stored(m):  # dense -> block-CSR values: (block row, block column, row, column) order
        order = np.lexsort((np.tile(np.arange(n), n), np.repeat(np.arange(n), n), np.tile(row, n), np.repeat(row, n)))
        return np.ascontiguousarray(m.ravel()[order])

    plan = sf.Plan(P, P, P, "fp32")
    assert plan.stats()[0] == nc ** 3
    a = dev(stored(M), "float32")
    out = dev(np.full(n * n, np.nan), "float32")
    plan.mul(a, a, out)
    want = stored(M.astype(np.float64) @ M.astype(np.float64))
    assert rel_frob(host(out), want) <= 1e-5
    again = dev(np.zeros(n * n), "float32")
    plan.mul(a, a, again)
    np.testing.assert_array_equal(host(again), host(out))
