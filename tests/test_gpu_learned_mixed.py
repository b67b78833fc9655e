"""The one-pass emit of a batch that mixes tensor-core and FP32 clouds, one of
them empty: the entries placed for the tensor-core clouds are compared with the
edges found for them alone, and every graph is the two-pass form's."""
import numpy as np
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


@pytest.mark.parametrize("dims", [(64,), (3, 64), (64, 3, 16, 128, 3), (32, 31)])
@pytest.mark.parametrize("upper", [False, True])
def test_mixed_batch(dims, upper):
    import torch
    from paper_2510_14147_gb300 import ctgraph as cg
    cg.ct_autotune_reset()  # tensor-core tiles from 32 floats per row up
    xs = [I.gmm_embedded(900 + 101 * i, dim=d, intrinsic=min(d, 4), n_centres=3, seed=i) for i, d in enumerate(dims)]
    xs.insert(1, np.zeros((0, 40), np.float32))
    trees = [cg.ct_build(points=torch.from_numpy(x).cuda()) for x in xs]
    eps = [1.5] * len(trees)
    p = cg.ct_predictor_create(seed=1)
    cg.ct_predictor_fit(p, trees[0], 1.5, steps=50, seed=2)
    want = cg.eps_graph_query_batched(trees, eps)
    got = cg.eps_graph_query_batched(trees, eps, precision=2, use_predictor=True, predictor=p, upper_triangle=upper)
    assert sum(c.nnz for c in want) > 1000
    for a, b in zip(got, want):
        for k in ("row_ptr", "col", "dist"):
            assert torch.equal(getattr(a, k), getattr(b, k)), k
    p.free()
