"""The two routes of an FP32 batch: a graph branch per system where every system has lists of transfer pairs, the
multi-system launches where one has not (H2_KRON=0 leaves it without), and both kinds in one batch."""
import pytest

from _helpers import rel_fro, require_cuda
from workloads import ellipsoid_points, gaussian_rhs

pytestmark = pytest.mark.gpu

SIZES = [(700, 3, 1), (1531, 4, 33), (900, 2, 64), (3001, 4, 16)]  # n, q, m


@pytest.mark.parametrize("no_pairs", [(), (0, 1, 2, 3), (2,)], ids=["branches", "multi", "mixed"])
def test_batch_routes_equal_single_fp64_products(no_pairs, monkeypatch):
    torch = require_cuda()
    import paper_2509_17257_gb300.build as bld
    bld.build()
    import paper_2509_17257_gb300 as P
    mats = []
    for i, (n, q, _) in enumerate(SIZES):
        if i in no_pairs:
            monkeypatch.setenv("H2_KRON", "0")
        else:
            monkeypatch.delenv("H2_KRON", raising=False)
        mats.append(P.H2Matrix(ellipsoid_points(n, (1.0, 0.7, 0.5), 40 + i), q=q, leaf_size=64, eta=2.0, sigma=1e-2,
                               precisions=("f32",)))
    B = P.H2Batch(mats)
    for seed in (1, 2):  # new buffers each time
        X = [torch.from_numpy(gaussian_rhs(n, m, 10 * seed + i)).cuda() for i, (n, _, m) in enumerate(SIZES)]
        Y = [torch.from_numpy(gaussian_rhs(n, m, 50 * seed + i)).cuda() for i, (n, _, m) in enumerate(SIZES)]
        ref = [y.clone() for y in Y]
        for A, x, y in zip(mats, X, ref):
            A.matmul(x, y, alpha=0.5, dtype="f64")
        B.matmul(X, Y, alpha=0.5, dtype="f32")
        torch.cuda.synchronize()
        for y, r in zip(Y, ref):
            # a few FP32 roundings, as for the single products of the other batches' tests
            assert rel_fro(y.cpu().numpy(), r.cpu().numpy()) <= 3e-6
    B.close()


def test_cached_graph_follows_workspaces_and_lists():
    """A batch's graph is replayed for the same buffers: not after a wider product outside the batch has grown a
    workspace, nor after the autotuner has rebuilt a matrix's lists."""
    torch = require_cuda()
    import paper_2509_17257_gb300.build as bld
    bld.build()
    import paper_2509_17257_gb300 as P
    n, m = 3001, 5
    mats = [P.H2Matrix(ellipsoid_points(n, (1.0, 0.7, 0.5), s), q=3, leaf_size=64, eta=2.0, sigma=1e-2,
                       precisions=("f32",)) for s in (1, 2)]
    B = P.H2Batch(mats)
    X = [torch.from_numpy(gaussian_rhs(n, m, 60 + i)).cuda() for i in range(2)]
    Y = [torch.zeros_like(x) for x in X]

    def check():
        for y in Y:
            y.zero_()
        B.matmul(X, Y, dtype="f32")
        for A, x, y in zip(mats, X, Y):
            ref = torch.zeros_like(x)
            A.matmul(x, ref, dtype="f64")
            assert rel_fro(y.cpu().numpy(), ref.cpu().numpy()) <= 3e-6

    check()
    wide = torch.from_numpy(gaussian_rhs(n, 64, 7)).cuda()
    mats[0].matmul(wide, torch.zeros_like(wide), dtype="f32")
    check()
    P.h2_autotune_ex(mats[1].handle, m, "f32")
    check()
    B.close()


def test_cached_multi_system_graph_follows_the_bookkeeping(monkeypatch):
    """The multi-system route's graph holds the addresses of the ready flags too: a product of more than 64 columns
    outside the batch lays the bookkeeping out anew, while the workspace is large enough already and stays."""
    torch = require_cuda()
    import paper_2509_17257_gb300.build as bld
    bld.build()
    import paper_2509_17257_gb300 as P
    monkeypatch.setenv("H2_KRON", "0")
    n, m = 3001, 64
    mats = [P.H2Matrix(ellipsoid_points(n, (1.0, 0.7, 0.5), s), q=3, leaf_size=64, eta=2.0, sigma=1e-2,
                       precisions=("f32",)) for s in (1, 2)]
    B = P.H2Batch(mats)
    X = [torch.from_numpy(gaussian_rhs(n, m, 80 + i)).cuda() for i in range(2)]
    Y = [torch.zeros_like(x) for x in X]
    ref = [torch.zeros_like(x) for x in X]
    for A, x, r in zip(mats, X, ref):
        A.matmul(x, r, dtype="f64")
    for wide in (0, 65, 200):
        if wide:
            w = torch.from_numpy(gaussian_rhs(n, wide, 7)).cuda()
            mats[0].matmul(w, torch.zeros_like(w), dtype="f32")
        for y in Y:
            y.zero_()
        B.matmul(X, Y, dtype="f32")
        torch.cuda.synchronize()
        for y, r in zip(Y, ref):
            assert rel_fro(y.cpu().numpy(), r.cpu().numpy()) <= 3e-6
    B.close()


@pytest.mark.parametrize("dtype", ["f32", "bf16", "f64"])
def test_first_batched_product_of_many_columns(dtype):
    """Everything a captured product needs is allocated before the capture, at several chunks of 64 columns too."""
    torch = require_cuda()
    import paper_2509_17257_gb300.build as bld
    bld.build()
    import paper_2509_17257_gb300 as P
    n, m = 900, 300
    mats = [P.H2Matrix(ellipsoid_points(n, (1.0, 0.7, 0.5), s), q=4, leaf_size=64, eta=2.0, sigma=1e-2,
                       precisions=("f32", "bf16")) for s in (1, 2)]
    B = P.H2Batch(mats)
    X = [torch.from_numpy(gaussian_rhs(n, m, 95 + i)).cuda() for i in range(2)]
    Y = [torch.zeros_like(x) for x in X]
    B.matmul(X, Y, dtype=dtype)
    for A, x, y in zip(mats, X, Y):
        ref = torch.zeros_like(x)
        A.matmul(x, ref, dtype="f64")
        torch.cuda.synchronize()
        assert rel_fro(y.cpu().numpy(), ref.cpu().numpy()) <= {"f32": 3e-6, "bf16": 3e-3, "f64": 1e-13}[dtype]
    B.close()


@pytest.mark.parametrize("kron,dtype", [("1", "f32"), ("0", "f32"), ("1", "f64")], ids=["branches", "multi", "f64"])
def test_cached_graph_follows_the_shift(kron, dtype, monkeypatch):
    """A changed shift counts at the next batched product, also for the same blocks."""
    torch = require_cuda()
    import paper_2509_17257_gb300.build as bld
    bld.build()
    import paper_2509_17257_gb300 as P
    monkeypatch.setenv("H2_KRON", kron)
    n, m = 1200, 6
    mats = [P.H2Matrix(ellipsoid_points(n, (1.0, 0.7, 0.5), s), q=3, leaf_size=64, eta=2.0, sigma=1e-2,
                       precisions=("f32",)) for s in (1, 2)]
    B = P.H2Batch(mats)
    X = [torch.from_numpy(gaussian_rhs(n, m, 90 + i)).cuda() for i in range(2)]
    Y = [torch.zeros_like(x) for x in X]
    for sigma in (1e-2, 1e3):
        P.h2_shift_set(mats[1].handle, sigma)
        for y in Y:
            y.zero_()
        B.matmul(X, Y, dtype=dtype)
        for A, x, y in zip(mats, X, Y):
            ref = torch.zeros_like(x)
            A.matmul(x, ref, dtype="f64")
            torch.cuda.synchronize()
            assert rel_fro(y.cpu().numpy(), ref.cpu().numpy()) <= 3e-6
    B.close()


@pytest.mark.parametrize("dtype", ["f64", "f32", "bf16"])
def test_branches_equal_single_products_of_whole_items_bit_for_bit(dtype, monkeypatch):
    """A captured branch runs whole items and no hybrid upward pass; with both switched off a single product runs the
    same lists, so the bits agree.  (By default a single FP32 product may sum in another order.)"""
    torch = require_cuda()
    import paper_2509_17257_gb300.build as bld
    bld.build()
    import paper_2509_17257_gb300 as P
    monkeypatch.setenv("H2_TC_HALVES", "0")
    monkeypatch.setenv("H2_TC_HYBRID", "0")
    mats = [P.H2Matrix(ellipsoid_points(n, (1.0, 0.7, 0.5), 40 + i), q=q, leaf_size=64, eta=2.0, sigma=1e-2,
                       precisions=("f32", "bf16")) for i, (n, q, _) in enumerate(SIZES)]
    B = P.H2Batch(mats)
    X = [torch.from_numpy(gaussian_rhs(n, m, 10 + i)).cuda() for i, (n, _, m) in enumerate(SIZES)]
    Y = [torch.from_numpy(gaussian_rhs(n, m, 50 + i)).cuda() for i, (n, _, m) in enumerate(SIZES)]
    ref = [y.clone() for y in Y]
    for A, x, y in zip(mats, X, ref):
        A.matmul(x, y, alpha=0.5, dtype=dtype)
    B.matmul(X, Y, alpha=0.5, dtype=dtype)
    torch.cuda.synchronize()
    for y, r in zip(Y, ref):
        assert torch.equal(y, r)
    B.close()
