"""The FP32 form's edge list: the emit pass of the count pass's list and of the
block masks (a list that runs out) give the same graph, which is the
oracle's, in single queries, batches and plans."""
import numpy as np
import pytest

import oracle
from paper_2510_14147_gb300 import inputs as I
from helpers import assert_csr_matches

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2510_14147_gb300 import build
    build.build()
    oracle.build()


@pytest.mark.parametrize("dim", [1, 3, 16, 17, 61, 64, 65, 128, 130])
@pytest.mark.parametrize("upper", [False, True])
def test_list_and_masks_agree(dim, upper):
    import torch
    from paper_2510_14147_gb300 import ctgraph as cg
    n = 2300
    x = I.gmm_embedded(n, dim=dim, intrinsic=min(dim, 5), n_centres=3, seed=dim)
    x[5:60] = x[4]  # pairs that only FP64 decides (distance 0) and a large leaf block
    sp = oracle.Space(points=x)
    eps = float(np.float32(np.quantile(oracle.brute_rows(sp, 1e30, np.arange(8))["dist"], 0.1)))
    t = cg.ct_build(points=torch.from_numpy(x).cuda())
    for e in (0.0, eps):
        ref = oracle.brute_force(sp, e)
        for own in (False, True):
            try:
                got = []
                for nbytes in (0, 64):  # the default list; one of eight entries
                    cg.ct_debug_capacity_budget(nbytes)
                    got.append(cg.eps_graph_query(t, e, upper_triangle=upper, include_self=own).to_numpy())
                    got.append(cg.eps_graph_query_batched([t, t], [e, e], upper_triangle=upper,
                                                          include_self=own)[1].to_numpy())
            finally:
                cg.ct_debug_capacity_budget(0)
            if e > 0.0:
                plan = cg.ct_plan_create([t, t], [e, e], upper_triangle=upper, include_self=own)
                cg.ct_plan_launch(plan)
                got.append(cg.ct_plan_result(plan)[1].to_numpy())
                plan.free()
            for g in got[1:]:
                for k in ("row_ptr", "col", "dist"):
                    assert np.array_equal(g[k], got[0][k]), k
            if not own:
                assert_csr_matches(got[0], ref)
