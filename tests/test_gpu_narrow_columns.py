"""The tensor-core products on both sides of the line between the two-CTAs-per-SM instances
(at most 64 activation rows, i.e. 32 columns of a chunk) and the wide ones, in every mode:
coupling and leaf launches, hybrid upward pass, tensor-core transfer passes, matrix-free, Aᵀ."""
import numpy as np
import pytest

from _helpers import rel_fro, require_cuda
from oracle import h2_oracle as O
from workloads import ellipsoid_points, gaussian_rhs

pytestmark = pytest.mark.gpu

# the products' error bounds: FP32 sums of at most 1e4 terms stay below 1e-5, BF16 operands
# (unit roundoff 2^-8) below 3e-3
TOL = {"f32": 1e-5, "bf16": 3e-3, "f32mf": 1e-5}
PATHS = {"default": {}, "hybrid": {"H2_TC_HYBRID": "1"}, "flow": {"H2_TC_TRANSFER": "1"}}


@pytest.mark.parametrize("path", PATHS)
@pytest.mark.parametrize("q", [2, 3, 4])
def test_columns_around_the_line(monkeypatch, q, path):
    torch = require_cuda()
    import paper_2509_17257_gb300 as P

    for key, value in PATHS[path].items():
        monkeypatch.setenv(key, value)
    n = 6000
    pts = ellipsoid_points(n, (0.6, 1.1, 1.9), 3)
    H = O.H2Matrix(pts, q=q, leaf_size=40, eta=2.0, sigma=1e-2)
    A = P.H2Matrix(pts, q=q, leaf_size=40, eta=2.0, sigma=1e-2, precisions=("f32", "bf16"))
    X = gaussian_rhs(n, 33, 5)
    want = O.h2mm(H, 1.0, X)
    for m in (1, 8, 9, 16, 20, 31, 32, 33):
        Xd = torch.from_numpy(X[:, :m].copy()).cuda()
        for dtype in ("f32", "bf16", "f32mf"):
            for product in (A.matmul,) if dtype == "f32mf" else (A.matmul, A.matmul_transposed):
                out = [product(Xd, torch.zeros_like(Xd), dtype=dtype).cpu().numpy() for _ in range(2)]
                assert rel_fro(out[0], want[:, :m]) <= TOL[dtype], (m, dtype)
                assert np.array_equal(out[0], out[1]), (m, dtype)
    A.close()
