"""Short work lists with their long items in two halves: against the same products with whole items (H2_TC_HALVES=0)
and against FP64, bit for bit from run to run."""
import numpy as np
import pytest

from _helpers import rel_fro, require_cuda
from workloads import ellipsoid_points, gaussian_rhs

pytestmark = pytest.mark.gpu

# a sum in another order and the FP32 roundings of the two halves: a few 2^-24 of a result whose terms cancel little;
# the split operands of BF16 carry 2^-16 each, but both sides round them alike
TOL = {"f32": 2e-6, "f32mf": 2e-6, "bf16": 2e-6}


def build(P, n, q, **kw):
    return P.H2Matrix(ellipsoid_points(n, (1.0, 0.8, 0.6), 9), q=q, leaf_size=64, eta=2.0, sigma=1e-2,
                      precisions=("f32", "bf16"), **kw)


@pytest.mark.parametrize("n,q", [(500, 2), (2048, 3), (9000, 4)])
def test_halves_match_whole_items(n, q, monkeypatch):
    torch = require_cuda()
    import paper_2509_17257_gb300.build as bld
    bld.build()
    import paper_2509_17257_gb300 as P
    halves = build(P, n, q)
    monkeypatch.setenv("H2_TC_HALVES", "0")
    whole = build(P, n, q)
    for m in (1, 7, 32, 50, 70):
        X = torch.from_numpy(gaussian_rhs(n, m, m)).cuda()
        exact = torch.zeros_like(X)
        whole.matmul(X, exact, dtype="f64")
        for dtype, trans in (("f32", False), ("f32", True), ("f32mf", False), ("bf16", False), ("bf16", True)):
            ys = []
            for A in (halves, halves, whole):
                Y = torch.zeros_like(X)
                (A.matmul_transposed if trans else A.matmul)(X, Y, dtype=dtype)
                ys.append(Y)
            assert torch.equal(ys[0], ys[1])
            assert rel_fro(ys[0].cpu().numpy(), ys[2].cpu().numpy()) <= TOL[dtype]
            if dtype != "bf16" and not trans:
                assert rel_fro(ys[0].cpu().numpy(), exact.cpu().numpy()) <= 3e-6


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("n,q", [(500, 2), (2048, 3)])
def test_halves_keep_subnormal_results(n, q, dtype, monkeypatch):
    """Results around the smallest normal FP32 number, 1.2e-38, where each rounding is off by half of 2^-149 whatever the
    result's size.  Where a whole item rounds a sum once, two halves round one each, so a column may be twice as far off
    as with whole items, and 2e-6 more where the format's own error shows.  A sum that takes subnormals for zero is off
    by up to 1.2e-38 instead, 20 to 200 times as far here.  Unit columns: one half of most items is zero; a column of
    ordinary size and one with a NaN among the small ones."""
    torch = require_cuda()
    import paper_2509_17257_gb300.build as bld
    bld.build()
    import paper_2509_17257_gb300 as P
    A = build(P, n, q)
    monkeypatch.setenv("H2_TC_HALVES", "0")
    whole = build(P, n, q)
    for M in (A, whole):
        P.h2_shift_set(M.handle, 0.0)
    for m in (6, 32, 41):
        for scale in (1e-36, 1e-38, 1e-39):
            x = gaussian_rhs(n, m, m) * scale
            x[:, 1] = 0.0
            x[7, 1] = scale
            x[:, 2] /= scale
            x[n // 2, 3] = np.nan
            X = torch.from_numpy(x).cuda()
            exact, Y, W = torch.zeros_like(X), torch.zeros_like(X), torch.zeros_like(X)
            whole.matmul(X, exact, dtype="f64")
            whole.matmul(X, W, dtype=dtype)
            A.matmul(X, Y, dtype=dtype)
            exact, Y, W = (v.cpu().numpy() / scale for v in (exact, Y, W))
            assert (np.isnan(Y[:, 3]) == np.isnan(W[:, 3])).all() and np.isnan(Y[:, 3]).any()
            for c in [c for c in range(m) if c != 3]:
                assert rel_fro(Y[:, c], exact[:, c]) <= 2 * rel_fro(W[:, c], exact[:, c]) + 2e-6, (m, scale, c)
