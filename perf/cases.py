"""The measured workloads of the library: products, batched products and solves, through the public entry points.

A case is a dict of plain values.  ``op`` says what a user does:

* ``mm``     Y <- A X, and Y <- Aᵀ X with ``trans``, of one H² matrix, in one of the product's precisions (``dtype``);
* ``cmm``    the complex product (Helmholtz kernel, complex128 blocks);
* ``batch``  the FP32 product of several independent systems of different sizes in one call;
* ``solve``  A X = B by block CG to a relative residual, FP64 or mixed precision.

``prepare`` makes what a user's program holds before the call (the built matrix or batch, the blocks on the GPU), ``run``
is one pass, ``exact`` the same result by plain torch in 64 bits, written from the definitions of the method: cluster
tree, block tree, tensor Chebyshev interpolation, and the product over them.
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

import paper_2509_17257_gb300 as P

LEAF, ETA, LENGTH, SIGMA = 64, 2.0, 0.5, 1e-2
KAPPA, DELTA = 1.0, 0.05
#: relative residual of the solves: the default of the differentiable solve
TOL = 1e-10
ELT = {"f64": 8, "f32": 4, "bf16": 2, "f32mf": 4}


def listed():
    return [
        # one right-hand side on a small cloud: the matrix-vector product inside someone's own iteration, all latency
        dict(name="mm f32 n2048 q3 m1", op="mm", dtype="f32", n=2048, q=3, m=1, axes="sphere", trans=False),
        # the small FP64 workload of the repository
        dict(name="mm f64 n4096 q3 m8", op="mm", dtype="f64", n=4096, q=3, m=8, axes="sphere", trans=False),
        # an ordinary FP32 product with a column count that no tile divides, on an ellipsoid
        dict(name="mm f32 n20011 q4 m13", op="mm", dtype="f32", n=20011, q=4, m=13, axes="ellipsoid", trans=False),
        # the benchmark's product
        dict(name="mm f32 n65536 q4 m32", op="mm", dtype="f32", n=65536, q=4, m=32, axes="sphere", trans=False),
        # the same in BF16, where the caller accepts its error
        dict(name="mm bf16 n65536 q4 m32", op="mm", dtype="bf16", n=65536, q=4, m=32, axes="sphere", trans=False),
        # the same with the coupling matrices evaluated instead of stored: for matrices that would not fit
        dict(name="mm f32mf n65536 q4 m32", op="mm", dtype="f32mf", n=65536, q=4, m=32, axes="sphere", trans=False),
        # the product of the differentiation workload: the largest matrix, few columns
        dict(name="mm f32 n262144 q4 m16", op="mm", dtype="f32", n=262144, q=4, m=16, axes="sphere", trans=False),
        # the adjoint direction, as the gradient of a loss through the product or the solve needs it
        dict(name="mmT f32 n65536 q4 m16", op="mm", dtype="f32", n=65536, q=4, m=16, axes="sphere", trans=True),
        # FP64: the true residuals of every mixed solve, and the FP64 solves
        dict(name="mm f64 n32768 q4 m16", op="mm", dtype="f64", n=32768, q=4, m=16, axes="sphere", trans=False),
        # the Helmholtz kernel
        dict(name="cmm f32 n32768 q4 m16", op="cmm", dtype="f32", n=32768, q=4, m=16, axes="sphere"),
        # many systems of uneven sizes at once
        dict(name="batch f32 16 systems", op="batch", dtype="f32", count=16, n_lo=2048, n_hi=32768, m_hi=64, shape=7),
        # the mixed-precision solve that the documentation recommends
        dict(name="solve f32 n8192 q4 m32", op="solve", dtype="f32", n=8192, q=4, m=32, axes="sphere", variant="gram",
             precond="block_jacobi"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["mm", "mm", "mm", "mm", "mm", "cmm", "batch", "solve"])
    axes = rng.choice(["sphere", "ellipsoid"])
    if op == "mm":
        dtype = rng.choice(["f32", "f32", "f32", "bf16", "f64", "f32mf"])
        n = _log_int(rng, 2048, {"f64": 32768, "f32mf": 65536}.get(dtype, 262144))
        most = {"f64": 32768 * 16, "f32mf": 65536 * 32}.get(dtype, 262144 * 16)
        return dict(op=op, dtype=dtype, n=n, q=rng.choice([3, 4]), m=_log_int(rng, 1, min(64, most // n)), axes=axes,
                    trans=dtype != "f32mf" and rng.random() < 0.25)
    if op == "cmm":
        n = _log_int(rng, 2048, 32768)
        return dict(op=op, dtype="f32", n=n, q=rng.choice([3, 4]), m=_log_int(rng, 1, min(32, 32768 * 16 // n)), axes=axes)
    if op == "batch":
        return dict(op=op, dtype="f32", count=rng.randint(2, 16), n_lo=2048, n_hi=_log_int(rng, 4096, 32768),
                    m_hi=_log_int(rng, 4, 64), shape=rng.randint(100, 1 << 20))
    if rng.random() < 0.5:
        return dict(op=op, dtype="f32", n=_log_int(rng, 2048, 8192), q=4, m=_log_int(rng, 16, 32), axes=axes,
                    variant="gram", precond="block_jacobi")
    return dict(op=op, dtype="f32", n=_log_int(rng, 2048, 5000), q=4, m=_log_int(rng, 1, 32), axes=axes,
                variant="columnwise", precond="block_jacobi")


# ---- inputs -------------------------------------------------------------------------------------------------------
def _points(n, axes, seed):
    rng = np.random.default_rng([seed, 1])
    g = rng.standard_normal((n, 3))
    p = g / np.sqrt((g * g).sum(axis=1, keepdims=True))
    if axes == "ellipsoid":
        p = p * rng.uniform(0.5, 2.0, size=3)[None, :]
    return np.ascontiguousarray(p)


def _block(n, m, seed, device, cplx=False):
    g = torch.Generator(device=device).manual_seed(1000003 * int(seed) + 17)
    return torch.randn(n, m, generator=g, device=device, dtype=torch.complex128 if cplx else torch.float64)


def _systems(case, seed):
    """(n, m, q, points) of a batch's systems: sizes by the case, coordinates by the seed."""
    rng = np.random.default_rng(case["shape"])
    out = []
    for i in range(case["count"]):
        n = int(round(math.exp(rng.uniform(math.log(case["n_lo"]), math.log(case["n_hi"])))))
        out.append((n, int(rng.integers(1, case["m_hi"] + 1)), int(rng.integers(3, 5)),
                    _points(n, "ellipsoid", 1009 * seed + i)))
    return out


def _matrix(pts, q, dtype, **kernel):
    extra = ("f32",) if dtype in ("f32", "f32mf") else (("bf16",) if dtype == "bf16" else ())
    return P.H2Matrix(pts, q=q, leaf_size=LEAF, eta=ETA, length=LENGTH, sigma=SIGMA, precisions=extra, **kernel)


def prepare(case, seed):
    op = case["op"]
    if op == "batch":
        systems = _systems(case, seed)
        mats = [_matrix(pts, q, case["dtype"]) for _, _, q, pts in systems]
        Xs = [_block(n, m, 1009 * seed + i, "cuda") for i, (n, m, _, _) in enumerate(systems)]
        return dict(case=case, A=P.H2Batch(mats), X=Xs, Y=[torch.zeros_like(x) for x in Xs])
    kernel = dict(kernel="helmholtz", kappa=KAPPA, delta=DELTA) if op == "cmm" else {}
    A = _matrix(_points(case["n"], case["axes"], seed), case["q"], case["dtype"], **kernel)
    X = _block(case["n"], case["m"], seed, "cuda", op == "cmm")
    return dict(case=case, A=A, X=X, Y=torch.zeros_like(X))


def run(state):
    case, A, X, Y = state["case"], state["A"], state["X"], state["Y"]
    op = case["op"]
    if op == "batch":
        torch._foreach_zero_(Y)
        return A.matmul(X, Y, dtype=case["dtype"])
    Y.zero_()
    if op == "cmm":
        return A.matmul_complex(X, Y, dtype=case["dtype"])
    if op == "mm":
        return (A.matmul_transposed if case["trans"] else A.matmul)(X, Y, dtype=case["dtype"])
    A.block_cg(X, Y, tol=TOL, dtype=case["dtype"], refine=2, inner_tol=0.1, variant=case["variant"],
               precond=case["precond"])
    return Y


# ---- what a pass cannot do without --------------------------------------------------------------------------------
def _sizes(pts):
    """(clusters, admissible blocks, entries of the nearfield)."""
    T = _tree(pts)
    adm, near = _blocks(T)
    return len(T["off"]), len(adm), int((T["size"][near[:, 0]] * T["size"][near[:, 1]]).sum())


@functools.lru_cache(maxsize=64)
def _counts(n, axes):
    return _sizes(_points(n, axes, 0))


def _product_work(n, q, m, dtype, cplx, counts):
    """One product: the couplings and the nearfield once (none of the couplings if they are evaluated), the bases and
    transfer matrices by their one-dimensional factors, X once, Y read and written."""
    nc, n_adm, nnz = counts
    k, elt, z = q ** 3, ELT[dtype], 2 if cplx else 1
    stored = (0 if dtype == "f32mf" else n_adm * k * k) + nnz
    data = elt * (z * stored + 3 * q * n + 3 * q * q * nc)
    flops = m * z * (4.0 * n * k + 4.0 * (nc - 1) * k * k) + m * (8.0 if cplx else 2.0) * (n_adm * k * k + nnz) + 2.0 * z * n * m
    return data + 8 * z * 3 * n * m, flops


def _iterations(case):
    """Iterations of the preconditioned solves to TOL, as measured (n = 2048, 4111, 8192 and m = 1, 5, 32; within a third
    of it): 228, 368, 568 column by column, and fewer with m columns searched together."""
    steps = 1.54 * case["n"] ** 0.655
    return steps * case["m"] ** -0.3 if case["variant"] == "gram" else steps


def work(case):
    if case["op"] == "batch":
        parts = [_product_work(n, q, m, case["dtype"], False, _sizes(pts)) for n, m, q, pts in _systems(case, 0)]
        return {"bytes": float(sum(p[0] for p in parts)), "flops": float(sum(p[1] for p in parts))}
    b, f = _product_work(case["n"], case["q"], case["m"], case["dtype"], case["op"] == "cmm",
                         _counts(case["n"], case["axes"]))
    passes = _iterations(case) if case["op"] == "solve" else 1.0  # one product an iteration
    return {"bytes": float(passes * b), "flops": float(passes * f)}


def tolerance(case):
    """Four times the largest error against ``exact`` that was seen over the ranges of ``draw``: 1.5e-15 in FP64, 3.0e-6
    in FP32 (it grows with n; 1e-6 at n = 65536 and m = 32), 1.9e-3 in BF16 (largest difference 1.8e-2), 1.6e-11 for
    the solves to TOL."""
    if case["op"] == "solve":
        return {"rel": 7e-11}
    return {"f64": {"rel": 6e-15}, "f32": {"rel": 1.2e-5}, "f32mf": {"rel": 1.2e-5},
            "bf16": {"rel": 8e-3, "max": 0.08}}[case["dtype"]]


# ---- the same results by plain torch in 64 bits -------------------------------------------------------------------
def _tree(pts):
    """The cluster tree in pre-order: a cluster of more than LEAF points is cut at the midpoint of the longest side of
    its tight box, points at or below the cut first; halves by index where a side would stay empty."""
    off, size, sons, lo, hi, order = [], [], [], [], [], []
    stack = [(np.arange(len(pts)), -1, 0)]
    at = 0
    while stack:
        idx, father, which = stack.pop()
        p = pts[idx]
        c = len(off)
        a, b = p.min(axis=0), p.max(axis=0)
        off.append(at)
        size.append(len(idx))
        sons.append([-1, -1])
        lo.append(a)
        hi.append(b)
        if father >= 0:
            sons[father][which] = c
        if len(idx) <= LEAF:
            order.append(idx)
            at += len(idx)
            continue
        d = int(np.argmax(b - a))
        low = p[:, d] <= (a[d] + b[d]) * 0.5
        first, second = idx[low], idx[~low]
        if len(first) == 0 or len(second) == 0:
            first, second = idx[: len(idx) // 2], idx[len(idx) // 2:]
        stack += [(second, c, 1), (first, c, 0)]
    return dict(off=np.array(off), size=np.array(size), sons=np.array(sons), lo=np.array(lo), hi=np.array(hi),
                perm=np.concatenate(order))


def _blocks(T):
    """The admissible pairs of clusters and the pairs of leaves left over, level of the block tree by level."""
    lo, hi, sons = T["lo"], T["hi"], T["sons"]
    w = hi - lo
    diam = np.sqrt((w[:, 0] * w[:, 0] + w[:, 1] * w[:, 1]) + w[:, 2] * w[:, 2])
    pairs, adm, near = np.zeros((1, 2), dtype=np.int64), [], []
    while len(pairs):
        t, s = pairs[:, 0], pairs[:, 1]
        g = np.maximum(np.maximum(lo[s] - hi[t], lo[t] - hi[s]), 0.0)
        dist = np.sqrt((g[:, 0] * g[:, 0] + g[:, 1] * g[:, 1]) + g[:, 2] * g[:, 2])
        ok = (dist > 0) & (np.maximum(diam[t], diam[s]) <= ETA * dist)
        tl, sl = sons[t, 0] < 0, sons[s, 0] < 0
        adm.append(pairs[ok])
        near.append(pairs[~ok & tl & sl])
        nxt = []
        for a in (0, 1):
            for b in (0, 1):
                # a leaf stands for both of its sons' places: its pair is listed once
                keep = ~ok & ~(tl & sl) & ~(tl & (a == 1)) & ~(sl & (b == 1))
                nxt.append(np.stack([np.where(tl, t, sons[t, a]), np.where(sl, s, sons[s, b])], axis=1)[keep])
        pairs = np.concatenate(nxt)
    return np.concatenate(adm), np.concatenate(near)


def _lagrange(nodes, x):
    """L_i(x) of the nodes [..., q] at x [..., p]: [..., p, q]."""
    q = nodes.shape[-1]
    out = []
    for i in range(q):
        v = torch.ones_like(x)
        for j in range(q):
            if j != i:
                v = v * (x - nodes[..., j, None]) / (nodes[..., i, None] - nodes[..., j, None])
        out.append(v)
    return torch.stack(out, dim=-1)


def _tensor(fx, fy, fz):
    """Products of the axes' polynomials [..., q], first axis fastest."""
    return (fz[..., :, None, None] * fy[..., None, :, None] * fx[..., None, None, :]).flatten(-3)


class _Plain:
    """The H² matrix of a point cloud in 64 bits, and its product with a block."""

    def __init__(self, pts, q, cplx=False):
        self.dev = dev = torch.device("cuda" if torch.cuda.is_available() else "cpu")
        self.q, self.k, self.cplx = q, q ** 3, cplx
        self.T = T = _tree(pts)
        adm, near = _blocks(T)
        self.adm, self.near = (torch.from_numpy(v).to(dev) for v in (adm, near))
        lo, hi = (torch.from_numpy(T[v]).to(dev) for v in ("lo", "hi"))
        half = (hi - lo) * 0.5
        most = half.amax(dim=1, keepdim=True)
        half = torch.maximum(half, torch.where(most > 0, 1e-8 * most, torch.full_like(most, 1e-8)))
        ref = torch.cos((2.0 * torch.arange(q, dtype=torch.float64, device=dev) + 1.0) * math.pi / (2.0 * q))
        self.axis = (lo + hi)[:, :, None] * 0.5 + half[:, :, None] * ref  # [cluster, axis, q]
        one = torch.ones(len(lo), q, q, q, dtype=torch.float64, device=dev)
        ax = self.axis
        self.nodes = torch.stack([ax[:, 0, None, None, :] * one, ax[:, 1, None, :, None] * one,
                                  ax[:, 2, :, None, None] * one], dim=-1).reshape(len(lo), self.k, 3)
        self.off, self.size = (torch.from_numpy(T[v]).to(dev) for v in ("off", "size"))
        self.perm = torch.from_numpy(T["perm"]).to(dev)
        self.pts = torch.from_numpy(pts).to(dev)[self.perm]
        self.leaf = torch.from_numpy(np.flatnonzero(T["sons"][:, 0] < 0)).to(dev)
        self.rows, self.mask = self._rows(self.leaf)
        self.V = self._basis(self.leaf, self.pts[self.rows]) * self.mask[..., None]
        level, depth, sons = np.zeros(len(lo), dtype=np.int64), 0, T["sons"]
        for c in range(len(lo)):
            for s in sons[c]:
                if s >= 0:
                    level[s] = level[c] + 1
        self.levels = [torch.from_numpy(np.flatnonzero((level == l) & (sons[:, 0] >= 0))).to(dev)
                       for l in range(level.max() + 1)]
        self.sons = torch.from_numpy(sons).to(dev)

    def _rows(self, c):
        """Positions of the clusters' points in cluster order, padded to LEAF, and which are points."""
        i = torch.arange(LEAF, device=self.dev)
        mask = i[None, :] < self.size[c][:, None]
        return torch.where(mask, self.off[c][:, None] + i[None, :], 0), mask

    def _basis(self, c, x):
        a = self.axis[c]
        return _tensor(*(_lagrange(a[:, d, :], x[..., d]) for d in range(3)))

    def _g(self, x, y):
        d = x[:, :, None, :] - y[:, None, :, :]
        r = torch.sqrt((d * d).sum(dim=-1))
        if not self.cplx:
            return torch.exp(-r / LENGTH)
        return torch.polar(1.0 / (4.0 * math.pi * torch.sqrt(r * r + DELTA * DELTA)), KAPPA * r)

    def matmul(self, X, trans=False):
        """A X; the matrix is symmetric, and the transposed product runs over the transposed lists all the same."""
        kind = torch.complex128 if self.cplx else torch.float64
        X = X.to(device=self.dev, dtype=kind)[self.perm]
        m, nc = X.shape[1], len(self.off)
        step = max(1, (1 << 28) // (8 * 4 * max(self.k, LEAF) ** 2))
        xh = torch.zeros(nc, self.k, m, dtype=kind, device=self.dev)
        yh = torch.zeros_like(xh)
        xh[self.leaf] = self.V.to(kind).transpose(1, 2) @ X[self.rows]
        for c in reversed(self.levels):
            for s in (0, 1):
                son = self.sons[c, s]
                E = self._basis(c, self.nodes[son]).to(kind)  # the father's polynomials at the son's nodes
                xh[c] += E.transpose(1, 2) @ xh[son]
        for j in range(0, len(self.adm), step):
            t, s = self.adm[j: j + step].unbind(1)
            S = self._g(self.nodes[t], self.nodes[s])
            yh.index_add_(0, s if trans else t, S.transpose(1, 2) @ xh[t] if trans else S @ xh[s])
        for c in self.levels:
            for s in (0, 1):
                son = self.sons[c, s]
                yh[son] += self._basis(c, self.nodes[son]).to(kind) @ yh[c]
        Y = SIGMA * X
        part = self.V.to(kind) @ yh[self.leaf]
        Y.index_add_(0, self.rows[self.mask], part[self.mask])
        for j in range(0, len(self.near), step):
            t, s = self.near[j: j + step].unbind(1)
            (rt, mt), (rs, ms) = self._rows(t), self._rows(s)
            G = self._g(self.pts[rt], self.pts[rs]) * (mt[:, :, None] & ms[:, None, :])
            out, keep, to = (G.transpose(1, 2) @ X[rt], ms, rs) if trans else (G @ X[rs], mt, rt)
            Y.index_add_(0, to[keep], out[keep])
        R = torch.empty_like(Y)
        R[self.perm] = Y
        return R


def exact(case, seed):
    op = case["op"]
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    if op == "batch":
        return [_Plain(pts, q).matmul(_block(n, m, 1009 * seed + i, dev))
                for i, (n, m, q, pts) in enumerate(_systems(case, seed))]
    A = _Plain(_points(case["n"], case["axes"], seed), case["q"], op == "cmm")
    X = _block(case["n"], case["m"], seed, dev, op == "cmm")
    if op != "solve":
        return A.matmul(X, case.get("trans", False))
    n = case["n"]
    dense = torch.empty(n, n, dtype=torch.float64, device=A.dev)
    eye = torch.zeros(n, 512, dtype=torch.float64, device=A.dev)
    for j in range(0, n, 512):
        w = min(512, n - j)
        eye.zero_()
        eye[torch.arange(j, j + w), torch.arange(w)] = 1.0
        dense[:, j: j + w] = A.matmul(eye[:, :w])
    return torch.linalg.solve(dense, X)
