"""Pair lists of the tensor-core filter that run out: a list grown once the need
is known, waves of all items, of the sample and of the rest cut in parts, and an
emit pass that filters again.  The kept pairs that a query counts show that its
first list cannot have held them, its launches that a budget cut the waves."""
import numpy as np
import pytest

from paper_2510_14147_gb300 import inputs as I

pytestmark = pytest.mark.gpu

CHUNK = 1024  # entries a warp of the filter reserves at a time; 12 such warps per SM


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2510_14147_gb300 import build
    build.build()


def _first_list(n, nbytes):
    """Entries of a query's first list: 512 per point, 16 M at most, within the budget."""
    import torch
    slack = torch.cuda.get_device_properties(0).multi_processor_count * 12 * CHUNK
    return slack + min(512 * n, 16 << 20, nbytes // 8 if nbytes else 1 << 62)


def _same(a, b):
    import torch
    for k in ("row_ptr", "col", "dist"):
        assert torch.equal(getattr(a, k), getattr(b, k)), k


@pytest.mark.parametrize("n,dim,degree,nbytes,sampled", [
    (3100, 16, 3100, 0, 0),            # grown
    (30000, 32, 300, 1 << 20, 0),      # all items, cut
    (30000, 32, 300, 24 << 20, 0),     # cut once or twice
    (170000, 3, 700, 1 << 20, 32),     # the sample cut, the rest in a thousand parts
])
def test_lists_shorter_than_the_kept_pairs(n, dim, degree, nbytes, sampled):
    import torch
    from paper_2510_14147_gb300 import ctgraph as cg
    x = torch.from_numpy(I.gmm_embedded(n, dim=dim, intrinsic=min(dim, 4), n_centres=8, seed=n)).cuda()
    d = torch.cdist(x[:6], x).reshape(-1)
    eps = float(np.float32(torch.quantile(d, min(1.0, degree / n)).item()))
    t = cg.ct_build(points=x)
    p = cg.ct_predictor_create(seed=1)
    cg.ct_predictor_fit(p, t, eps, steps=100, seed=2)
    ref = cg.eps_graph_query(t, eps)
    launches = cg.eps_graph_query(t, eps, precision=1).stats()["kernel_launches"]
    try:
        cg.ct_debug_capacity_budget(nbytes)
        for kw in ({}, {"upper_triangle": True}, {"use_predictor": True, "predictor": p},
                   {"upper_triangle": True, "use_predictor": True, "predictor": p}):
            got = cg.eps_graph_query(t, eps, precision=1, **kw)
            _same(got, ref)
            if not kw:
                s, first = got.stats(), _first_list(n, nbytes)
                assert s["recheck_fp32"] / max(1, sampled) > first
                if nbytes:  # a wave is a filter and a decision launch, and the first list takes one such wave
                    assert s["kernel_launches"] >= launches + 2 * (s["recheck_fp32"] // first)
    finally:
        cg.ct_debug_capacity_budget(0)
    p.free()
