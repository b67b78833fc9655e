"""The FP32 edge list where there are many work items of few edges each: the list
is used (the emit pass decides its entries alone), and the graph is that of the
block masks."""
import pytest

from paper_2510_14147_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2510_14147_gb300 import build
    build.build()


def _tree(x):
    import torch
    from paper_2510_14147_gb300 import ctgraph as cg
    return cg.ct_build(points=torch.from_numpy(x).cuda())


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


def test_many_items_with_few_edges():
    x = I.uniform_cube(100001, 16, seed=3)
    nnz, emitted = _both(_tree(x), 0.75)
    assert emitted == nnz
