"""The transfer passes as lists of pairs (h2_transfer.cu) on trees of every shape: a single leaf,
few levels, flat and linear point sets (boxes without extent), clusters of very uneven depth (66
levels), and column counts around the lane groups."""
import numpy as np
import pytest

from _helpers import rel_fro, require_cuda
from oracle import h2_oracle as O
from workloads import gaussian_rhs, sphere_points

pytestmark = pytest.mark.gpu

# FP32 against the oracle: sums of at most 1e4 terms stay below 1e-5.  BF16 against the BF16
# product with the level-by-level passes (H2_KRON=0): the matrices are the same, so what is left
# is the split of the activations to 16 bits (2^-17 = 7.6e-6 each) and the FP32 passes (1e-5
# each), in sums whose terms cancel by less than a factor of 5 here: 2e-4, as for the hybrid pass.
# (Against the oracle BF16 has no bound of its own on a line: entries along it round alike, and
# the errors add up with them.)
F32_TOL, BF16_TOL = 1e-5, 2e-4


def _plane(n):
    p = np.random.default_rng(2).uniform(-1, 1, (n, 3))
    p[:, 2] = 0.25
    return p


def _line(n):
    p = np.zeros((n, 3))
    p[:, 1] = np.random.default_rng(3).uniform(0, 3, n)
    return p


def _uneven(n, octaves):
    # distances from the origin halve and halve again: one side of every cut is nearly empty
    g = np.random.default_rng(4).standard_normal((n, 3))
    return g / np.linalg.norm(g, axis=1)[:, None] * 2.0 ** -np.random.default_rng(5).uniform(0, octaves, n)[:, None]


CASES = {
    "one point": (lambda: sphere_points(1, 0), 64), "one leaf": (lambda: sphere_points(50, 0), 64),
    "two levels": (lambda: sphere_points(110, 1), 64), "sphere": (lambda: sphere_points(3000, 2), 24),
    "plane": (lambda: _plane(2000), 32), "line": (lambda: _line(1500), 16), "uneven": (lambda: _uneven(2500, 24), 20),

}


@pytest.mark.parametrize("q", [2, 3, 4])
@pytest.mark.parametrize("name", CASES)
def test_pairs_on_every_tree(monkeypatch, name, q):
    torch = require_cuda()
    import paper_2509_17257_gb300 as P

    make, leaf = CASES[name]
    pts = make()
    n = pts.shape[0]
    H = O.H2Matrix(pts, q=q, leaf_size=leaf, eta=2.0, sigma=1e-2)
    build = dict(q=q, leaf_size=leaf, eta=2.0, sigma=1e-2, precisions=("f32", "bf16"))
    A = P.H2Matrix(pts, **build)
    monkeypatch.setenv("H2_KRON", "0")
    A0 = P.H2Matrix(pts, **build)
    X = gaussian_rhs(n, 64, 5)
    want = O.h2mm(H, 1.0, X)
    for m in (1, 4, 5, 8, 12, 16, 20, 32, 40, 64):
        Xd = torch.from_numpy(X[:, :m].copy()).cuda()
        for trans in (False, True):
            def run(M, dtype):
                product = M.matmul_transposed if trans else M.matmul
                return product(Xd, torch.zeros_like(Xd), dtype=dtype).cpu().numpy()

            assert rel_fro(run(A, "f32"), want[:, :m]) <= F32_TOL, m
            assert rel_fro(run(A, "bf16"), run(A0, "bf16")) <= BF16_TOL, m
    A.close()
    A0.close()
