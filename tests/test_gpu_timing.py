"""Per-phase times (h2_timing_enable / h2_timing_query): each phase's work is counted under its own slot."""
import pytest

from _helpers import require_cuda
from workloads import gaussian_rhs, sphere_points

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", ["f32", "bf16", "f32mf"])
def test_phases_of_a_product_on_lists_of_pairs(dtype):
    """The leaves' launch gathers X, so the gather's slot holds two event records and nothing else; the leaves and the
    upward pass are several launches, tens of times as long."""
    torch = require_cuda()
    import paper_2509_17257_gb300.build as bld
    bld.build()
    import paper_2509_17257_gb300 as P
    n, m = 20000, 32
    A = P.H2Matrix(sphere_points(n, 1), q=4, leaf_size=64, eta=2.0, sigma=1e-2, precisions=("f32", "bf16"))
    X = torch.from_numpy(gaussian_rhs(n, m, 1)).cuda()
    Y = torch.zeros_like(X)
    A.matmul(X, Y, dtype=dtype)
    P.h2_timing_enable(A.handle, True)
    P.h2_timing_query(A.handle, reset=True)
    for _ in range(5):
        A.matmul(X, Y, dtype=dtype)
    ms, calls = P.h2_timing_query(A.handle, reset=True)
    P.h2_timing_enable(A.handle, False)
    assert calls == 5
    assert ms["leaf_fwd"] > 2 * ms["gather"] and ms["leaf_fwd"] > 2 * ms["up"]
    assert min(ms["coupling"], ms["down"], ms["leaf_bwd_near"]) > 2 * ms["up"]
    assert ms["coupling_kernel"] <= ms["coupling"]
    A.close()
