"""The FP32 edge list where it is sized from a sample (above 1.4 million points), where
there are many work items of few edges each, and where there is no memory for
it: the list is used (the emit pass decides its entries alone) or the block
masks are, and the graph is the same."""
import numpy as np
import pytest

import oracle
from paper_2510_14147_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2510_14147_gb300 import build
    build.build()
    oracle.build()


def _tree(x):
    import torch
    from paper_2510_14147_gb300 import ctgraph as cg
    return cg.ct_build(points=torch.from_numpy(x).cuda())


def _eps(x, degree):
    d = oracle.brute_rows(oracle.Space(points=x), 1e30, np.arange(6))["dist"]
    return float(np.float32(np.quantile(d, degree / x.shape[0])))


def _both(t, eps, **kw):
    """The graph through the list and through the masks: (entries, the emit pass's decisions)."""
    import torch
    from paper_2510_14147_gb300 import ctgraph as cg
    got = cg.eps_graph_query(t, eps, **kw)
    try:
        cg.ct_debug_capacity_budget(64)
        ref = cg.eps_graph_query(t, eps, **kw)
    finally:
        cg.ct_debug_capacity_budget(0)
    for k in ("row_ptr", "col", "dist"):
        assert torch.equal(getattr(got, k), getattr(ref, k)), k
    assert ref.stats()["emit_pairs"] > got.nnz
    return got.nnz, got.stats()["emit_pairs"]


@pytest.mark.parametrize("n,dim,degree", [(1420001, 3, 20), (1410001, 61, 8), (1405001, 66, 6)])
@pytest.mark.parametrize("upper", [False, True])
def test_list_sized_from_a_sample(n, dim, degree, upper):
    x = I.gmm_embedded(n, dim=dim, intrinsic=min(dim, 5), n_centres=60, seed=n)
    x[100:180] = x[7]  # pairs that only FP64 decides, a large leaf block
    t, eps = _tree(x), _eps(x, degree)
    for own in (False, True):
        nnz, emitted = _both(t, eps, upper_triangle=upper, include_self=own)
        assert emitted <= nnz and (upper or emitted == nnz)


def test_list_of_a_dense_graph():
    # more than 192 edges a point (as a sample sees, or as the count pass finds): masks
    for n in (60001, 1420001):
        x = I.uniform_cube(n, 3, seed=n)
        nnz, emitted = _both(_tree(x), float((270 / n / 4.18879) ** (1 / 3)))
        assert nnz > 200 * n and emitted > nnz


@pytest.mark.parametrize("dim", [16, 68])
def test_many_items_with_few_edges(dim):
    x = np.zeros((100001, dim), np.float32)  # 16 coordinates: the same items for both kernels
    x[:, :16] = I.uniform_cube(100001, 16, seed=3)
    nnz, emitted = _both(_tree(x), 0.75)
    assert emitted == nnz


@pytest.mark.parametrize("n", [3000, 1420001])
def test_without_memory_for_the_list(n):
    """Each allocation of the call fails in turn: the call either fails with
    CT_ENOMEM or, when the list's failed, gives the graph without it."""
    from paper_2510_14147_gb300 import ctgraph as cg
    x = I.gmm_embedded(n, dim=4, intrinsic=4, n_centres=60, seed=4)
    t, eps = _tree(x), _eps(x, 8)
    ref = cg.eps_graph_query(t, eps).to_numpy()
    plan_ref = cg.ct_plan_create([t], [eps])
    cg.ct_plan_launch(plan_ref)
    assert np.array_equal(cg.ct_plan_result(plan_ref)[0].to_numpy()["col"], ref["col"])
    plan_ref.free()
    for plan in (False, True):
        failed, without_list, whole = 0, 0, 0
        for k in range(1, 400):
            before = cg.ct_debug_pool_used()
            cg.ct_debug_fail_alloc(k)
            p = None
            try:
                if plan:
                    p = cg.ct_plan_create([t], [eps])
                    cg.ct_debug_fail_alloc(0)
                    cg.ct_plan_launch(p)
                    c = cg.ct_plan_result(p)[0]
                else:
                    c = cg.eps_graph_query(t, eps)
                got, emitted = c.to_numpy(), c.stats()["emit_pairs"]
                c.free()
            except cg.CtError as e:
                assert e.status == cg.CT_ENOMEM
                failed += 1
                continue
            finally:
                cg.ct_debug_fail_alloc(0)
                if p is not None:
                    p.free()
                assert cg.ct_debug_pool_used() == before
            for name in ("row_ptr", "col", "dist"):
                assert np.array_equal(got[name], ref[name]), name
            without_list += emitted > len(got["col"])
            whole += emitted == len(got["col"])
            if whole >= 3 + plan:  # (a plan's sizing query has a list of its own)
                break
        assert failed > 20 and whole >= 3 and without_list >= 1
