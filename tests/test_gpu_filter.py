"""The tensor-core filter and its pair lists: row lengths at which the MMA's K
blocks, the lanes per pair or the load width change, tiles with few rows, and
lists that run out -- waves cut in two, and an emit pass that filters again.
Every form gives the FP32 form's graph, bit for bit."""
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


def _cg():
    from paper_2510_14147_gb300 import ctgraph as cg
    return cg


def _tree(x):
    import torch
    return _cg().ct_build(points=torch.from_numpy(x).cuda())


def _eps(x, degree):
    if x.shape[0] == 1:
        return 1.0
    d = oracle.brute_rows(oracle.Space(points=x), 1e30, np.arange(6))["dist"]
    return float(np.float32(np.quantile(d, degree / x.shape[0])))


def _same(a, b):
    for k in ("row_ptr", "col", "dist"):
        assert np.array_equal(a[k], b[k]), k


def _query(t, eps, **kw):
    c = _cg().eps_graph_query(t, eps, **kw)
    out = c.to_numpy()
    out["stats"] = c.stats()
    return out


@pytest.mark.parametrize("n", [1, 33, 700, 5000])
@pytest.mark.parametrize("dim", [1, 3, 4, 16, 17, 20, 24, 60, 64, 65, 68, 72, 100, 124, 126, 128])
def test_row_lengths(dim, n):
    x = I.gmm_embedded(n, dim=dim, intrinsic=min(dim, 6), n_centres=4, seed=dim)
    t = _tree(x)
    eps = _eps(x, min(40, n / 2))
    ref = _query(t, eps)
    for up in (False, True):
        for own in (False, True):
            got = _query(t, eps, precision=1, upper_triangle=up, include_self=own)
            _same(got, _query(t, eps, include_self=own) if own else ref)


@pytest.mark.parametrize("n,dim,degree", [(30000, 32, 300), (170000, 3, 40)])
def test_lists_that_run_out(n, dim, degree):
    cg = _cg()
    x = I.gmm_embedded(n, dim=dim, intrinsic=min(dim, 4), n_centres=8, seed=n)
    t = _tree(x)
    eps = _eps(x, degree)
    p = cg.ct_predictor_create(seed=1)
    cg.ct_predictor_fit(p, t, eps, steps=200, seed=2)
    ref = _query(t, eps)
    learned = {"use_predictor": True, "predictor": p}
    try:
        for nbytes in (0, 1 << 20, 16 << 20):
            cg.ct_debug_capacity_budget(nbytes)
            for up in (False, True):
                _same(_query(t, eps, precision=1, upper_triangle=up), ref)
                _same(_query(t, eps, precision=1, upper_triangle=up, **learned), ref)
    finally:
        cg.ct_debug_capacity_budget(0)
    p.free()
