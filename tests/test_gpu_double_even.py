"""The double product on equally wide blocks, whose steps run several accumulators' chains side by side: every
tile class and count of live accumulators (blocks of 1 to 41 rows and columns, rectangular tiles from two widths),
even and odd numbers of lambda blocks, forward and both adjoints.  1e-12 relative as the other double
tests (another summation order of at most a few hundred products)."""
import numpy as np
import pytest

import workloads as W
from oracle import adjoint as oadj
from oracle import product as oprod
from tests.gpu_util import dev, host, pattern_of, rel_frob
from tests.test_oracle_product import random_bcsr

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("wide", [1, 2, 3, 5, 6, 7, 9, 10, 11, 13, 14, 15, 16, 19, 20, 21, 27, 40, 41])
@pytest.mark.parametrize("nc", [5, 17])
def test_equal_widths(wide, nc):
    # one cluster of another width makes tiles wide x 4 and 4 x wide, all steps but one stay even
    from paper_2211_11681_gb300 import sformat as sf
    bsize = np.full(nc, wide)
    bsize[nc // 2] = 4
    A, B = random_bcsr(bsize, 1.0, wide), random_bcsr(bsize, 1.0, wide + 1)
    P = pattern_of(A)
    plan = sf.Plan(P, P, P, "fp64")
    want = oprod.mul_masked(A, B, A, nthreads=8).val
    for v in range(plan.num_variants()):
        plan.set_variant(v)
        out = dev(np.full(len(A.val), np.nan))
        plan.mul(dev(A.val), dev(B.val), out)
        assert rel_frob(host(out), want) <= 1e-12, v
    dC = A.like(W.random_values(len(A.val), wide + 2))
    wA, wB = oadj.mul_masked_adjoint(dC, A, B)
    gA, gB = dev(np.full(len(A.val), np.nan)), dev(np.full(len(A.val), np.nan))
    plan.adjoint(dev(dC.val), dev(A.val), dev(B.val), gA, gB)
    assert rel_frob(host(gA), wA.val) <= 1e-12
    assert rel_frob(host(gB), wB.val) <= 1e-12
