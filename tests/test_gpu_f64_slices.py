"""The FP64 phases (h2_mm64.cu) at the edges of their cuts: output pairs (odd k and odd leaf
sizes), chunks of 32 pairs (ceil(rows / 2) times the columns, at most 32, of a tile), column
tiles of 32, slices of 1, 2 and 4 columns, 64-column tiles."""
import numpy as np
import pytest

from _helpers import rel_fro, require_cuda
from oracle import h2_oracle as O
from workloads import ellipsoid_points, gaussian_rhs

pytestmark = pytest.mark.gpu

# a sum of p products of FP64 numbers rounds to p·2^-53 of its absolute terms; p is at most
# the points of the near lists and k per level, below 2000 here, and the terms do not cancel
# by more than the oracle's own rounding shows
TOL = 2000 * 2.0 ** -53


@pytest.mark.parametrize("q,leaf", [(1, 24), (2, 7), (3, 64), (4, 33), (5, 64)])
@pytest.mark.parametrize("m", [1, 2, 3, 16, 17, 32, 33, 64, 65, 130])
def test_f64_product_at_the_cuts(q, leaf, m):
    torch = require_cuda()
    import paper_2509_17257_gb300 as P

    n = 1501
    pts = ellipsoid_points(n, (0.6, 1.1, 1.9), 3)
    H = O.H2Matrix(pts, q=q, leaf_size=leaf, eta=2.0, sigma=1e-2)
    A = P.H2Matrix(pts, q=q, leaf_size=leaf, eta=2.0, sigma=1e-2, precisions=())
    X, Y0 = gaussian_rhs(n, m, 5), gaussian_rhs(n, m, 6)
    want = O.h2mm(H, 0.5, X, Y0)
    for ld in (m, m + 3):
        Xd = torch.zeros(n, ld, dtype=torch.float64, device="cuda")[:, :m]
        Yd = torch.zeros(n, ld, dtype=torch.float64, device="cuda")[:, :m]
        for product in (A.matmul, A.matmul_transposed):  # the kernel is symmetric
            Xd.copy_(torch.from_numpy(X))
            Yd.copy_(torch.from_numpy(Y0))
            product(Xd, Yd, alpha=0.5, dtype="f64")
            first = Yd.cpu().numpy()
            assert rel_fro(first, want) <= TOL
            Yd.copy_(torch.from_numpy(Y0))
            product(Xd, Yd, alpha=0.5, dtype="f64")
            assert np.array_equal(first, Yd.cpu().numpy())
    A.close()


# groups of `size` points at the corners of a cube, a leaf each: 31, 32 and 33 pairs of a leaf's
# row pairs and columns, and twice 31 and 32; k = 27 has 14 row pairs: 28 pairs with 2 columns,
# 42 with 3
@pytest.mark.parametrize("size,m", [(62, 1), (63, 1), (64, 1), (6, 11), (62, 2), (64, 2), (22, 3), (21, 3)])
def test_f64_product_at_the_chunks(size, m):
    torch = require_cuda()
    import paper_2509_17257_gb300 as P

    corners = np.array([[i & 1, i >> 1 & 1, i >> 2] for i in range(8)], dtype=np.float64)
    pts = np.repeat(corners, size, axis=0) + 0.1 * ellipsoid_points(8 * size, (0.6, 1.1, 1.9), 3)
    n = len(pts)
    H = O.H2Matrix(pts, q=3, leaf_size=size, eta=2.0, sigma=1e-2)
    A = P.H2Matrix(pts, q=3, leaf_size=size, eta=2.0, sigma=1e-2, precisions=())
    assert P.h2_info(A.handle)["n_leaves"] == 8  # of exactly `size` points then
    X, Y0 = gaussian_rhs(n, m, 5), gaussian_rhs(n, m, 6)
    want = O.h2mm(H, 0.5, X, Y0)
    for product in (A.matmul, A.matmul_transposed):  # the kernel is symmetric
        Yd = torch.from_numpy(Y0).cuda()
        product(torch.from_numpy(X).cuda(), Yd, alpha=0.5, dtype="f64")
        assert rel_fro(Yd.cpu().numpy(), want) <= TOL
    A.close()
