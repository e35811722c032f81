"""Performance cases: the calls a user of the S-format library makes, at the sizes of its
workloads, with the inputs such a program holds and the result in 64 bits to compare with.

    listed()             the named cases
    draw(rng)            one more case of the same ranges
    prepare(case, seed)  inputs on the GPU, patterns and plans (what a program keeps)
    run(state)           one pass through the public entry points, its outputs
    work(case)           bytes and operations one pass cannot do without
    exact(case, seed)    the outputs of run() as torch gives them in 64 bits

Every matrix is a samplet-compressed Matern kernel matrix, built by the library's own builder
on the points of one of the families below (the workloads of the paper's experiments and of
the tests).  The points, and with them the pattern, are fixed by family and size; the seed
draws a standard deviation per samplet coordinate (the symmetric scaling D A D, which keeps
the pattern, the symmetry and the positive definiteness) and the right-hand sides, second
factors, incoming gradients and the length scale of a matrix that is built.
"""
import math

import numpy as np
import torch

from paper_2211_11681_gb300 import autograd as ag
from paper_2211_11681_gb300 import sformat as sf
from paper_2211_11681_gb300.builder import Builder
from paper_2211_11681_gb300.selinv import SelInv

# Kernel, tree and pattern parameters of the workloads; tau is the a-posteriori threshold,
# relative to 1/N where "tau_over_n" is set (as the kernel itself, which is scaled by 1/N).
FAMILIES = {
    # FP64 parity and batch workload: small 2D matrices, 6- to 10-wide blocks
    "matern32_2d": dict(d=2, nu=1.5, ell=0.2, nugget=1e-3, q=2, leaf=16, eta=1.25, tau=1e-10),
    # the multiplication benchmark of Sec. 5.1 in the plane (10-wide blocks) and in space (20-wide)
    "paper_2d": dict(d=2, nu=0.5, ell=1.0, nugget=0.0, q=3, leaf=20, eta=1.25, tau=1e-5, tau_over_n=True),
    "paper_3d": dict(d=3, nu=0.5, ell=1.0, nugget=0.0, q=3, leaf=40, eta=1.25, tau=1e-5, tau_over_n=True),
    # the headline product: 20-wide blocks, symmetric
    "matern12_3d": dict(d=3, nu=0.5, ell=0.1, nugget=0.0, q=3, leaf=32, eta=1.0, tau=1e-8),
    # matrix functions on a closed surface and differentiation in space: no threshold
    "matern52_sphere": dict(d=3, sphere=True, nu=2.5, ell=0.3, nugget=1e-2, q=2, leaf=16, eta=1.25, tau=0.0),
    "matern32_3d": dict(d=3, nu=1.5, ell=0.15, nugget=1e-2, q=2, leaf=16, eta=1.25, tau=0.0),
}
RIDGE = 1e-2  # shift of the selected inversion (the largest of the paper's ridge parameters)
NS_STEPS = 10  # Newton-Schulz steps of the differentiated square root
TAYLOR = 8     # Taylor degree of the exponential


def listed():
    return [
        # the smallest product: one matrix of the batch workload, A A with A symmetric; launches and
        # the longest sum of a single output block decide
        dict(name="mul_fp32_2d_1000", op="mul", family="matern32_2d", n=1000, prec="fp32", second="same"),
        # the FP64 parity workload, the default arithmetic on a small matrix
        dict(name="mul_fp64_2d_4096", op="mul", family="matern32_2d", n=4096, prec="fp64", second="same"),
        # Sec. 5.1 in the plane: K times a perturbed, no longer symmetric K, float and double
        dict(name="mul_fp32_2d_50000", op="mul", family="paper_2d", n=50000, prec="fp32", second="perturbed"),
        dict(name="mul_fp64_2d_20000", op="mul", family="paper_2d", n=20000, prec="fp64", second="perturbed"),
        # the headline product (20-wide blocks, symmetric, float) at the size one pass of which takes tens of ms
        dict(name="mul_fp32_3d_65536", op="mul", family="matern12_3d", n=65536, prec="fp32", second="same"),
        # Sec. 5.1 in space, double, leaves that do not divide evenly
        dict(name="mul_fp64_3d_5000", op="mul", family="paper_3d", n=5000, prec="fp64", second="perturbed"),
        # a training step through one float product: forward and both gradients
        dict(name="mul_grad_fp32_3d_6000", op="mul_grad", family="matern32_3d", n=6000, prec="fp32"),
        # the error estimator's application of a matrix to ten vectors
        dict(name="spmm_2d_60000_x10", op="spmm", family="paper_2d", n=60000, k=10),
        # whole calls: the differentiated float square root with its quadratic-form loss, and exp(-A) in double
        dict(name="sqrt_grad_fp32_3d_2000", op="sqrt_grad", family="matern32_3d", n=2000),
        dict(name="exp_neg_fp64_sphere_3000", op="exp_neg", family="matern52_sphere", n=3000),
        # (K + mu I)^{-1} on the pattern: one factorization and one selected inversion (Sec. 5.2)
        dict(name="selinv_2d_8192", op="selinv", family="paper_2d", n=8192),
        # compressing the kernel matrix itself, once per length scale: what every program does before
        # anything else
        dict(name="build_sphere_40000", op="build", family="matern52_sphere", n=40000),
    ]


# Sizes of the drawn cases per operation, family and arithmetic.
RANGES = [
    ("mul", "matern32_2d", "fp32", 500, 20000), ("mul", "paper_2d", "fp32", 500, 50000),
    ("mul", "matern12_3d", "fp32", 500, 65536), ("mul", "paper_3d", "fp32", 500, 8000),
    ("mul", "matern32_2d", "fp64", 500, 12000), ("mul", "paper_2d", "fp64", 500, 20000),
    ("mul", "matern12_3d", "fp64", 500, 6000), ("mul", "paper_3d", "fp64", 500, 5000),
    ("mul", "matern32_2d", "fp64_df", 500, 8000), ("mul", "matern12_3d", "fp64_df", 500, 6000),
    ("mul_grad", "matern32_3d", "fp32", 500, 6000), ("mul_grad", "paper_2d", "fp32", 500, 20000),
    ("mul_grad", "paper_2d", "fp64", 500, 6000),
    ("spmm", "paper_2d", None, 1000, 60000), ("spmm", "matern12_3d", None, 1000, 30000),
    ("sqrt_grad", "matern32_3d", None, 300, 2000), ("sqrt_grad", "matern52_sphere", None, 300, 2000),
    ("exp_neg", "matern52_sphere", None, 500, 3000), ("exp_neg", "matern32_2d", None, 500, 3000),
    ("selinv", "paper_2d", None, 500, 8192), ("selinv", "matern52_sphere", None, 500, 2000),
    ("build", "matern52_sphere", None, 1000, 40000), ("build", "matern32_2d", None, 1000, 40000),
]


def draw(rng):
    op, family, prec, lo, hi = rng.choice(RANGES)
    case = dict(op=op, family=family, n=int(round(math.exp(rng.uniform(math.log(lo), math.log(hi))))))
    if prec is not None:
        case["prec"] = prec
    if op == "mul":
        case["second"] = rng.choice(["same", "perturbed"])
    if op == "spmm":
        case["k"] = rng.randint(1, 16)
    return case


# ---- inputs ------------------------------------------------------------------------------


def _points(case):
    f = FAMILIES[case["family"]]
    g = np.random.Generator(np.random.PCG64(case["n"]))
    if f.get("sphere"):
        x = g.standard_normal((case["n"], f["d"]))
        return x / np.linalg.norm(x, axis=1, keepdims=True)
    return g.random((case["n"], f["d"]))


def _builder(case):
    f = FAMILIES[case["family"]]
    return Builder(_points(case), f["leaf"], f["q"], f["eta"])


def _kernel_args(case, seed=None):
    f, n = FAMILIES[case["family"]], case["n"]
    args = dict(nu=f["nu"], ell=f["ell"], kscale=1.0 / n, nugget=f["nugget"],
                tau=f["tau"] / n if f.get("tau_over_n") else f["tau"])
    if case["op"] == "build":  # another length scale on the whole eta pattern
        args.update(ell=f["ell"] * float(np.random.Generator(np.random.PCG64(seed)).uniform(0.8, 1.25)), tau=0.0)
    return args


def _rng(seed, salt):
    return torch.Generator(device="cuda").manual_seed(1000003 * salt + seed)


def _inputs(case, seed):
    """The tensors and pattern of a case (no plan): shared by prepare() and exact()."""
    b = _builder(case)
    if case["op"] == "build":
        return dict(op="build", builder=b, args=_kernel_args(case, seed))
    pat, a = b.values(**_kernel_args(case))
    sd = 0.8 + 0.4 * torch.rand(case["n"], generator=_rng(seed, 5), device="cuda", dtype=torch.float64)
    r, c = _Layout(pat).coordinates()
    a = a * (sd[r] * sd[c])  # one product first: both triangles get the same rounding
    del r, c
    s = dict(op=case["op"], pat=pat, A=a)
    dt = torch.float32 if case.get("prec") == "fp32" else torch.float64
    if case["op"] in ("mul", "mul_grad"):
        s["A"] = a.to(dt)
        s["B"] = s["A"]
        if case.get("second") != "same":  # every stored entry times 1 + 0.1 u
            s["B"] = (a * (1.0 + 0.1 * torch.rand(a.shape, generator=_rng(seed, 1), device="cuda",
                                                  dtype=torch.float64))).to(dt)
    if case["op"] == "mul_grad":
        # the gradient that comes back has the matrix's own decay
        s["dC"] = (a * torch.randn(a.shape, generator=_rng(seed, 2), device="cuda", dtype=torch.float64)).to(dt)
    if case["op"] == "spmm":
        s["X"] = torch.rand((case["k"], case["n"]), generator=_rng(seed, 3), device="cuda", dtype=torch.float64)
    if case["op"] == "sqrt_grad":
        s["z"] = torch.randn(case["n"], generator=_rng(seed, 4), device="cuda", dtype=torch.float64)
    return s


def prepare(case, seed):
    s = _inputs(case, seed)
    op = s["op"]
    if op in ("mul", "mul_grad"):
        p = s["pat"]
        s["plan"] = sf.Plan(p, p, p, case["prec"])
        if case.get("second") == "same" and case["prec"] == "fp32":
            s["plan"].set_symmetric_a(True)  # B = A, a symmetric matrix
    if op == "mul":
        s["C"] = torch.empty_like(s["A"])
    if op == "mul_grad":
        s["A"] = s["A"].requires_grad_(True)
        s["B"] = s["B"].requires_grad_(True)
    if op == "spmm":
        s["Y"] = torch.empty_like(s["X"])
    if op == "sqrt_grad":
        s["A"] = s["A"].requires_grad_(True)
    if op == "exp_neg":
        s["F"] = torch.empty_like(s["A"])
    if op == "selinv":
        s["inv"] = SelInv(s["pat"])
        s["Z"] = torch.empty_like(s["A"])
    return s


# ---- one pass ----------------------------------------------------------------------------


def run(s):
    op = s["op"]
    if op == "mul":
        return s["plan"].mul(s["A"], s["B"], s["C"])
    if op == "mul_grad":
        c = ag.MaskedMul.apply(s["A"], s["B"], s["plan"])
        da, db = torch.autograd.grad(c, (s["A"], s["B"]), s["dC"])
        return c.detach(), da, db
    if op == "spmm":
        return sf.spmm(s["pat"], s["A"], s["X"], s["Y"])
    if op == "sqrt_grad":
        # the float iteration: its square root and gradient are good to float accuracy and are
        # kept in float
        f = ag.SqrtmNS.apply(s["A"], s["pat"], NS_STEPS, None, "fp32", 0)
        loss = ag.QuadForm.apply(f, s["pat"], s["z"])
        (da,) = torch.autograd.grad(loss, (s["A"],))
        return f.detach().float(), da.float()
    if op == "exp_neg":
        sf.funm(s["pat"], "exp_neg", s["A"], s["F"], taylor_degree=TAYLOR)
        return s["F"]
    if op == "selinv":
        s["inv"].factor(s["A"], RIDGE)
        s["inv"].invert(s["Z"])
        s["inv"].status()
        return s["Z"]
    if op == "build":
        pat, vals = s["builder"].values(**s["args"])
        return vals, pat.nblocks
    raise ValueError(op)


# ---- what a pass cannot do without ---------------------------------------------------------

_WORK = {}


def work(case):
    key = tuple(sorted((k, v) for k, v in case.items() if k != "name"))
    if key not in _WORK:
        _WORK[key] = _work(case)
    return _WORK[key]


def _work(case):
    """Counted on the case's own pattern."""
    op, n = case["op"], case["n"]
    if op == "build":
        # every kernel entry of the upper triangle once (a distance, a root, an exponential and the
        # polynomial: about 20 operations); points in, kept values out
        pat, vals = _builder(case).values(**_kernel_args(case, 0))
        return dict(bytes=8.0 * vals.numel() + 8.0 * 3 * n, flops=20.0 * n * (n + 1) / 2)
    s = _inputs(case, 0)
    nnz, nblk = s["A"].numel(), s["pat"].nblocks
    if op == "spmm":
        return dict(bytes=8.0 * nnz + 4.0 * nblk + 16.0 * n * case["k"], flops=2.0 * nnz * case["k"])
    if op == "selinv":
        st = SelInv(s["pat"]).stats()
        return dict(bytes=16.0 * nnz, flops=st["flops_factor"] + st["flops_invert"])
    prec = case.get("prec", "fp64")
    p = s["pat"]
    _, flops = sf.Plan(p, p, p, prec).stats()
    w = s["A"].element_size()
    if op == "mul":
        return dict(bytes=float(w * nnz * (2 if case["second"] == "same" else 3)), flops=flops)
    if op == "mul_grad":  # A, B, dC in, C, dA, dB out
        return dict(bytes=float(w * nnz * 6), flops=3.0 * flops)
    if op == "exp_neg":
        return dict(bytes=16.0 * nnz, flops=(TAYLOR - 1) * flops)
    if op == "sqrt_grad":  # 3 products forward and 7 back per step
        return dict(bytes=16.0 * nnz, flops=10.0 * NS_STEPS * flops)
    raise ValueError(op)


# ---- the same in 64 bits --------------------------------------------------------------------

DENSE_MUL = 10000    # largest matrix multiplied as a dense one
DENSE_BUILD = 6000   # largest kernel matrix transformed as a dense one


class _Layout:
    """Block layout of a pattern: sizes, rows and columns of the blocks and of their entries."""

    def __init__(self, pat):
        bo, rp, ci = (torch.from_numpy(np.asarray(v).astype(np.int64)).cuda() for v in pat.arrays())
        self.bo, self.bs, self.nc, self.n = bo, bo[1:] - bo[:-1], len(bo) - 1, int(bo[-1])
        self.row = torch.repeat_interleave(torch.arange(self.nc, device="cuda"), rp[1:] - rp[:-1])
        self.col = ci
        size = self.bs[self.row] * self.bs[self.col]
        self.voff = torch.cumsum(size, 0) - size

    def coordinates(self):
        """Row and column of every stored entry."""
        nr, ncol = self.bs[self.row], self.bs[self.col]
        blk = torch.repeat_interleave(torch.arange(len(nr), device="cuda"), nr * ncol)
        e = torch.arange(len(blk), device="cuda") - self.voff[blk]
        w = ncol[blk]
        r = torch.div(e, w, rounding_mode="floor")
        return self.bo[self.row[blk]] + r, self.bo[self.col[blk]] + e - r * w

    def gather(self, dense):
        r, c = self.coordinates()
        return dense[r, c]

    def dense(self, vals):
        d = torch.zeros((self.n, self.n), device="cuda", dtype=torch.float64)
        r, c = self.coordinates()
        d[r, c] = vals.double()
        return d

    def by_size(self):
        """{(rows, cols): block ids} of the distinct block shapes."""
        key = self.bs[self.row] * 4096 + self.bs[self.col]
        return {(int(k) // 4096, int(k) % 4096): torch.nonzero(key == k).flatten() for k in torch.unique(key)}


def _masked_product(lay, a, b):
    """sum over lambda of A(nu, lambda) B(lambda, nu') on the blocks of the pattern, by batches of
    equally shaped block triples in 64 bits."""
    groups = lay.by_size()
    group_of = torch.empty(len(lay.row), dtype=torch.int64, device="cuda")
    place = torch.empty_like(group_of)
    shapes, am, bm, cm = [], [], [], []
    for g, (shape, ids) in enumerate(groups.items()):
        group_of[ids] = g
        place[ids] = torch.arange(len(ids), device="cuda")
        at = lay.voff[ids][:, None] + torch.arange(shape[0] * shape[1], device="cuda")
        shapes.append(shape)
        am.append(a[at].double())
        bm.append(b[at].double())
        cm.append(torch.zeros(am[-1].shape, dtype=torch.float64, device="cuda"))
    key = lay.row * lay.nc + lay.col  # ascending: blocks are stored row by row
    first = torch.searchsorted(lay.row, torch.arange(lay.nc + 1, device="cuda"))
    fan = (first[1:] - first[:-1])[lay.col]  # B blocks each A block meets
    ends = torch.cumsum(fan, 0)
    k0, nb, ng = 0, len(lay.row), len(shapes)
    while k0 < nb:
        base = int(ends[k0 - 1]) if k0 else 0
        k1 = max(k0 + 1, int(torch.searchsorted(ends, torch.tensor(base + 20_000_000, device="cuda"))))
        f = fan[k0:k1]
        ka = torch.repeat_interleave(torch.arange(k0, k1, device="cuda"), f)
        kb = first[lay.col[ka]] + torch.arange(len(ka), device="cuda") - torch.repeat_interleave(
            ends[k0:k1] - f - base, f)
        want = lay.row[ka] * lay.nc + lay.col[kb]
        kc = torch.searchsorted(key, want).clamp_(max=nb - 1)
        hit = key[kc] == want
        ka, kb, kc = ka[hit], kb[hit], kc[hit]
        combo = group_of[ka] * ng + group_of[kb]
        for c in torch.unique(combo).tolist():
            ga, gb = c // ng, c % ng
            sel = torch.nonzero(combo == c).flatten()
            ni, nl, nj = shapes[ga][0], shapes[ga][1], shapes[gb][1]
            gc = shapes.index((ni, nj))
            step = max(1, 200_000_000 // max(ni * nl, nl * nj, ni * nj))
            for t in range(0, len(sel), step):
                q = sel[t:t + step]
                prod = torch.bmm(am[ga][place[ka[q]]].view(-1, ni, nl), bm[gb][place[kb[q]]].view(-1, nl, nj))
                cm[gc].index_add_(0, place[kc[q]], prod.view(len(q), -1))
        k0 = k1
    out = torch.zeros(len(a), dtype=torch.float64, device="cuda")
    for g, (shape, ids) in enumerate(groups.items()):
        out[lay.voff[ids][:, None] + torch.arange(shape[0] * shape[1], device="cuda")] = cm[g]
    return out


def _exact_sqrt_grad(lay, a, z):
    """The masked Newton-Schulz iteration and the gradient of z^T F z with the scaling frozen."""
    r, c = lay.coordinates()
    mask = torch.zeros((lay.n, lay.n), device="cuda", dtype=torch.float64)
    mask[r, c] = 1.0
    A = lay.dense(a)
    eye = torch.eye(lay.n, device="cuda", dtype=torch.float64)
    x = torch.full((lay.n,), 1.0 / math.sqrt(lay.n), device="cuda", dtype=torch.float64)
    lam = 0.0
    for _ in range(50):  # power iteration with Rayleigh quotients
        y = A @ x
        lam = float(x @ y)
        x = y / torch.linalg.norm(y)
    scale = 1.01 * lam
    Y, Z, keep = A / scale, eye, []
    for _ in range(NS_STEPS):
        keep.append((Y, Z))
        T = 0.5 * (3.0 * eye - (Z @ Y) * mask)
        Y, Z = (Y @ T) * mask, (T @ Z) * mask
    F = math.sqrt(scale) * Y
    dY, dZ = math.sqrt(scale) * torch.outer(z, z) * mask, torch.zeros_like(Y)
    for Y, Z in reversed(keep):
        T = 0.5 * (3.0 * eye - (Z @ Y) * mask)
        dT = (Y.T @ dY) * mask + (dZ @ Z.T) * mask
        dP = -0.5 * dT
        dY, dZ = (dY @ T.T) * mask + (Z.T @ dP) * mask, (T.T @ dZ) * mask + (dP @ Y.T) * mask
    return F[r, c], (dY / scale)[r, c]


def exact(case, seed):
    op = case["op"]
    s = _inputs(case, seed)
    if op == "build":
        if case["n"] > DENSE_BUILD:
            return None
        return _exact_build(case, s)
    lay = _Layout(s["pat"])
    if op == "mul":
        if case["n"] <= DENSE_MUL:
            return lay.gather(lay.dense(s["A"]) @ lay.dense(s["B"]))
        return _masked_product(lay, s["A"], s["B"])
    if op == "mul_grad":
        if case["n"] > DENSE_MUL:
            return None
        A, B, dC = (lay.dense(s[k]) for k in ("A", "B", "dC"))
        return lay.gather(A @ B), lay.gather(dC @ B.T), lay.gather(A.T @ dC)
    if op == "spmm":
        return (lay.dense(s["A"]) @ s["X"].T).T.contiguous()
    if op == "sqrt_grad":
        return _exact_sqrt_grad(lay, s["A"], s["z"])
    if op == "exp_neg":
        r, c = lay.coordinates()
        mask = torch.zeros((lay.n, lay.n), device="cuda", dtype=torch.float64)
        mask[r, c] = 1.0
        X = -lay.dense(s["A"])  # norm below 0.5: no squarings
        eye = torch.eye(lay.n, device="cuda", dtype=torch.float64)
        E = eye + X / TAYLOR
        for k in range(TAYLOR - 1, 0, -1):
            E = eye + (X @ E) * mask / k
        return E[r, c]
    if op == "selinv":
        A = lay.dense(s["A"])
        A.diagonal().add_(RIDGE)
        return lay.gather(torch.linalg.inv(A))
    raise ValueError(op)


def _exact_build(case, s):
    """P_S(T K T^T) with the tree's dense transform T, in 64 bits."""
    f, n = FAMILIES[case["family"]], case["n"]
    x = torch.from_numpy(_points(case)).cuda()
    dist = torch.cdist(x, x, compute_mode="donot_use_mm_for_euclid_dist")
    t = math.sqrt(2.0 * f["nu"]) * dist / s["args"]["ell"]
    poly = {0.5: torch.ones_like(t), 1.5: 1.0 + t, 2.5: 1.0 + t + t * t / 3.0}[f["nu"]]
    T = torch.from_numpy(s["builder"].dense_transform()).cuda()
    full = T @ (poly * torch.exp(-t) / n) @ T.T
    full.diagonal().add_(f["nugget"])
    pat, _ = s["builder"].values(**s["args"])
    return _Layout(pat).gather(full), pat.nblocks
