"""Host logic of the packed float product (mul_nt.cu): what its plan does when memory runs out, and which
kernel a product takes.  The library's object files are linked with a CUDA runtime over host memory (fake_cuda_runtime.cpp), in which any
device or host allocation can be made to fail.  No GPU: the launches are only counted and their
operands checked against the live allocations."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


class Fake:
    """The library over host memory, with the few calls the tests make."""

    def __init__(self, path):
        self.lib = L = ctypes.CDLL(path, mode=ctypes.RTLD_LOCAL)
        for n in ("fake_used", "fake_bad", "fake_device_calls", "fake_host_calls", "fake_launches"):
            getattr(L, n).restype = ctypes.c_int64
        for n in ("fake_pool", "fake_fail_device", "fake_fail_host"):
            getattr(L, n).argtypes = [ctypes.c_int64]
        L.s_pattern_nnz.restype = ctypes.c_int64
        for n in ("s_pattern_nnz", "s_pattern_destroy", "s_plan_destroy"):
            getattr(L, n).argtypes = [ctypes.c_void_p]
        L.s_plan_set_symmetric_a.argtypes = [ctypes.c_void_p, ctypes.c_int]

    def pattern(self, sizes):
        nc = len(sizes)
        bo = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
        rp, ci = (np.arange(nc + 1) * nc).astype(np.int64), np.tile(np.arange(nc), nc).astype(np.int32)
        p = ctypes.c_void_p()
        assert self.lib.s_pattern_create(ctypes.c_int32(nc), bo.ctypes, np.zeros(nc, np.int32).ctypes, rp.ctypes, ci.ctypes,
                                         ctypes.byref(p)) == 0
        return p

    def plan(self, p, fp32):
        q = ctypes.c_void_p()
        return self.lib.s_plan_create(p, p, p, ctypes.c_int(fp32), ctypes.byref(q)), q

    def buffers(self, p, count):
        n, out = self.lib.s_pattern_nnz(p), []
        for _ in range(count):
            b = ctypes.c_void_p()
            assert self.lib.cudaMalloc(ctypes.byref(b), ctypes.c_size_t(4 * n)) == 0
            out.append(b)
        return out

    def launches_of(self, call):
        """Status of a call, and how often the packed and the tile kernel and the listing ran in it."""
        self.lib.fake_reset_launches()
        st = call()
        return st, [self.lib.fake_launches(k) for k in (b"mul_f32_nt_kernel", b"mul_f32_kernel", b"nt_list_kernelILb1E")]


@pytest.fixture(scope="module")
def fake(tmp_path_factory):
    from paper_2211_11681_gb300 import build
    build.build()
    d = tmp_path_factory.mktemp("fake")
    inc = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(build.nvcc()))), "include")
    obj, lib = str(d / "fake.o"), str(d / "libsformat_fake.so")
    subprocess.check_call(["g++", "-std=c++17", "-O1", "-fPIC", "-I", inc, "-c", os.path.join(HERE, "fake_cuda_runtime.cpp"),
                           "-o", obj])
    objs = [os.path.join(build.OBJ_DIR, os.path.basename(s) + ".o") for s in build.sources()]
    subprocess.check_call(["g++", "-shared", "-Wl,-Bsymbolic", "-Wl,--no-undefined", "-o", lib] + objs + [obj, "-lgomp", "-lpthread"])
    return Fake(lib)


@pytest.fixture
def calm(fake):
    """The library with nothing made to fail, before and after a test."""
    fake.lib.fake_pool(1 << 40)
    yield fake
    fake.lib.fake_fail_device(-1)
    fake.lib.fake_fail_host(-1)
    fake.lib.fake_pool(1 << 40)


SIZES = [3, 20, 7, 41, 10, 1]


@pytest.mark.parametrize("kind", ["device", "host"])
def test_symmetric_flag_survives_a_failed_allocation(calm, kind):
    # whichever allocation of s_plan_set_symmetric_a fails, the plan stays usable: the next product runs
    # on the packed kernel with everything it reads in live memory, or on the tile kernel
    from paper_2211_11681_gb300 import sformat as sf
    L = calm.lib
    fail = L.fake_fail_device if kind == "device" else L.fake_fail_host
    p = calm.pattern(SIZES)
    A, C = calm.buffers(p, 2)
    used0, i, packed = L.fake_used(), 0, []
    while True:
        st, q = calm.plan(p, sf.PREC["fp32"])
        assert st == 0
        fail(i)
        st = L.s_plan_set_symmetric_a(q, 1)
        reached = (L.fake_device_calls() if kind == "device" else L.fake_host_calls()) > i
        fail(-1)
        assert st in (0, sf.S_ERR_NOMEM)
        st, n = calm.launches_of(lambda: L.s_mul_masked(q, A, A, C, None))
        assert (st, L.fake_bad()) == (0, 0), i
        assert n[0] + n[1] == 1
        packed.append(n[0])
        assert L.s_plan_destroy(q) == 0
        assert L.fake_used() == used0 and L.fake_bad() == 0
        if not reached:
            break
        i += 1
    assert i > 3 and packed[-1] == 1  # nothing failed in the last turn


@pytest.mark.parametrize("call", ["create", "adjoint"])
def test_failed_allocations_of_a_plan(calm, call):
    # every device allocation of plan creation, and of the first adjoint, in turn: S_ERR_NOMEM, or a
    # call that ran with all it reads in live memory; nothing stays allocated behind either
    from paper_2211_11681_gb300 import sformat as sf
    L = calm.lib
    p = calm.pattern(SIZES)
    A, B, C, dA, dB = calm.buffers(p, 5)
    used0, i, refused = L.fake_used(), 0, 0
    while True:
        if call == "create":
            L.fake_fail_device(i)
        st, q = calm.plan(p, sf.PREC["fp32"])
        if call == "adjoint":
            assert st == 0
            L.fake_fail_device(i)
            st = L.s_mul_masked_adjoint(q, C, A, B, dA, dB, None)
        reached = L.fake_device_calls() > i
        L.fake_fail_device(-1)
        assert st in (0, sf.S_ERR_NOMEM), (i, st)
        refused += st != 0
        if q:
            st, n = calm.launches_of(lambda: L.s_mul_masked(q, A, B, C, None))
            assert (st, n[0] + n[1]) == (0, 1), i
            st, n = calm.launches_of(lambda: L.s_mul_masked_adjoint(q, C, A, B, dA, dB, None))
            assert (st, n[0] + n[1]) == (0, 2), i
            assert L.s_plan_destroy(q) == 0
        assert (L.fake_used(), L.fake_bad()) == (used0, 0), i
        if not reached:
            break
        i += 1
    assert 0 < refused < i


def footprint(fake, p):
    """Device bytes a float plan on p takes when it lists in one piece, and the lists' share."""
    from paper_2211_11681_gb300 import sformat as sf
    L = fake.lib
    used = L.fake_used()
    st, q = fake.plan(p, sf.PREC["fp32"])
    assert st == 0
    all_bytes = L.fake_used() - used
    assert L.s_plan_destroy(q) == 0
    return all_bytes


def test_lists_leave_room(calm):
    # 120 one-wide clusters, every block present: 1.73e6 triples, 27.6 MB of lists beside a matrix of 58 KB
    from paper_2211_11681_gb300 import sformat as sf
    L, lists = calm.lib, 16 * 120 ** 3
    p = calm.pattern([1] * 120)
    A, C = calm.buffers(p, 2)
    rest = footprint(calm, p) - lists  # packed copies, tiles
    assert 0 < rest < 3 << 20
    used0 = L.fake_used()
    # (pool, ranges of a product): kept while half of the pool stays free, else range by range in 1 MiB
    # (1/512 of what is free is less) of 16-byte entries, rows of 120 entries a block
    per_range = ((1 << 20) // 16) // 120 * 120
    many = -(-120 ** 3 // per_range)
    for pool, want in [(1 << 30, 0), (2 * (used0 + rest + lists) + 4096, 0), (2 * (used0 + rest + lists) - 65536, many),
                       (used0 + rest + (2 << 20), many)]:
        L.fake_pool(pool)
        st, q = calm.plan(p, sf.PREC["fp32"])
        assert st == 0, pool
        if want:
            assert L.fake_used() - used0 <= rest + (1 << 20) + 4096
        st, n = calm.launches_of(lambda: L.s_mul_masked(q, A, A, C, None))
        assert (st, n, L.fake_bad()) == (0, [max(want, 1), 0, want], 0), pool
        assert L.s_plan_destroy(q) == 0 and L.fake_used() == used0
    # not even a workspace: the tile kernel, and no packed copies kept for nothing
    L.fake_pool(used0 + rest + (1 << 19))
    st, q = calm.plan(p, sf.PREC["fp32"])
    assert st == 0
    assert L.fake_used() - used0 < rest // 2
    st, n = calm.launches_of(lambda: L.s_mul_masked(q, A, A, C, None))
    assert (st, n, L.fake_bad()) == (0, [0, 1, 0], 0)
    assert L.s_plan_destroy(q) == 0


def test_many_plans_share_a_pool(calm):
    # as many plans as fit without lists (and a workspace of 1 MiB each) can be held together, all on
    # the packed kernel, whatever their lists would take (32 times the pool)
    from paper_2211_11681_gb300 import sformat as sf
    L = calm.lib
    p = calm.pattern([1] * 120)
    A, C = calm.buffers(p, 2)
    count = 64
    pool = 256 << 20
    assert count * 16 * 120 ** 3 > 6 * pool
    L.fake_pool(pool)
    plans = []
    for _ in range(count):
        st, q = calm.plan(p, sf.PREC["fp32"])
        assert st == 0, len(plans)
        assert L.s_plan_set_symmetric_a(q, 1) == 0
        plans.append(q)
    for q in plans:
        st, n = calm.launches_of(lambda: L.s_mul_masked(q, A, A, C, None))
        assert (st, n[0] > 0, n[1], L.fake_bad()) == (0, True, 0, 0)
        assert L.s_plan_destroy(q) == 0


@pytest.mark.parametrize("nc, ahead", [(3, False), (120, False), (121, True), (160, True)])
def test_tiles_taken_ahead(calm, nc, ahead):
    # nc^2 tiles; the runtime has 152 SMs and 4 resident CTAs of 4 warps: the line is at 6 x 2432 = 14592
    from paper_2211_11681_gb300 import sformat as sf
    L = calm.lib
    p = calm.pattern([2] * nc)
    A, C = calm.buffers(p, 2)
    st, q = calm.plan(p, sf.PREC["fp32"])
    assert st == 0
    L.fake_reset_launches()
    assert L.s_mul_masked(q, A, A, C, None) == 0
    assert [L.fake_launches(b"mul_f32_nt_kernelILb%d" % v) for v in (0, 1)] == [not ahead, ahead]
    assert L.s_plan_destroy(q) == 0


@pytest.mark.parametrize("nc, lanes", [(3, 32), (139, 32), (140, 8)])
def test_packing_lanes(calm, nc, lanes):
    # a warp a block while all are resident: 152 SMs of 8 CTAs of 8 warps, twice over: 19456 blocks
    from paper_2211_11681_gb300 import sformat as sf
    L = calm.lib
    p = calm.pattern([2] * nc)
    A, B, C = calm.buffers(p, 3)
    st, q = calm.plan(p, sf.PREC["fp32"])
    assert st == 0
    L.fake_reset_launches()
    assert L.s_mul_masked(q, A, B, C, None) == 0
    assert [L.fake_launches(b"nt_prepare_kernelILi%d" % v) for v in (8, 32)] == [lanes == 8, lanes == 32]
    assert (L.s_plan_destroy(q), L.fake_bad()) == (0, 0)


@pytest.mark.parametrize("ms, products", [(10.0, (1, 0)), (0.5, (4, 0)), (0.03, (4, 9))])
def test_autotuner_stops_at_the_packed_kernel(calm, ms, products):
    # (time of a measurement, products of the packed and of the other kernels): a first launch of 10 ms ends
    # it, so do three of 0.17 ms each; at 0.01 ms each the 9 other shapes are tried (equal times: one
    # launch each, the packed kernel is kept)
    from paper_2211_11681_gb300 import sformat as sf
    L = calm.lib
    p = calm.pattern([2] * 5)
    A, C = calm.buffers(p, 2)
    st, q = calm.plan(p, sf.PREC["fp32"])
    assert st == 0
    L.fake_event_ms(ctypes.c_float(ms))
    chosen = ctypes.c_int(-1)
    L.fake_reset_launches()
    assert L.s_plan_autotune(q, A, A, C, None, ctypes.byref(chosen)) == 0
    n = [L.fake_launches(k) for k in (b"mul_f32_nt_kernel", b"mul_f32_kernel", b"mul_f32_panel_kernel")]
    assert (chosen.value, n[0], n[1] + n[2]) == (0,) + products
    assert (L.s_plan_destroy(q), L.fake_bad()) == (0, 0)
