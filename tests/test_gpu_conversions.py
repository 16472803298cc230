"""FP64 columns through the FP32 product's conversions: exponents at both ends of the FP32 range, zeros, subnormals,
overflow, infinities and NaN, each in a column of its own."""
import numpy as np
import pytest

from _helpers import require_cuda
from workloads import ellipsoid_points, gaussian_rhs

pytestmark = pytest.mark.gpu

SCALES = [1.0, 1e-30, 1e30, 2.0 ** -100, 0.0, 1e-320, 1e-42]


@pytest.mark.parametrize("q,extra", [(3, 0), (4, 20)])
def test_scaled_columns_and_nonfinite_values_stay_apart(q, extra):
    torch = require_cuda()
    import paper_2509_17257_gb300.build as bld
    bld.build()
    import paper_2509_17257_gb300 as P
    n = 1500
    A = P.H2Matrix(ellipsoid_points(n, (1.0, 0.8, 0.6), 3), q=q, leaf_size=64, eta=2.0, sigma=1e-2, precisions=("f32",))
    x = gaussian_rhs(n, 1, 5)
    cols = [x * s for s in SCALES]
    for bad in (np.inf, np.nan, 1e300):
        y = x.copy()
        y[7] = bad
        cols.append(y)
    cols += [gaussian_rhs(n, 1, 20 + i) for i in range(extra)]
    X = torch.from_numpy(np.ascontiguousarray(np.concatenate(cols, axis=1))).cuda()
    Y, R = torch.zeros_like(X), torch.zeros_like(X)
    A.matmul(X, Y, dtype="f32")
    A.matmul(X, R, dtype="f64")
    Y, R = Y.cpu().numpy(), R.cpu().numpy()
    for c in [0, 1, 2, 3] + list(range(len(SCALES) + 3, Y.shape[1])):
        assert np.linalg.norm(Y[:, c] - R[:, c]) <= 3e-6 * np.linalg.norm(R[:, c]), c
    assert not Y[:, 4].any()
    assert np.abs(Y[:, 5]).max() <= 1e-318  # zero in FP32; σX is added in FP64
    # subnormal in FP32, where a sum may count as zero: off by its own size at most
    assert np.abs(Y[:, 6] - R[:, 6]).max() <= 1e-38
    for c in range(len(SCALES), len(SCALES) + 3):
        assert not np.isfinite(Y[:, c]).all()
