"""Walks whose candidates exceed the first candidate pool (256 entries per
point): they stop, the pool grows and they go on.  Rows are compared with the
oracle's brute force; the candidate count shows that the pool ran out."""
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


@pytest.mark.parametrize("metric", ["l2", "l2-upper-tc", "hamming", "strings"])
def test_rows_after_the_pool_grew(metric):
    import torch
    from paper_2510_14147_gb300 import ctgraph as cg
    opts = {}
    if metric.startswith("l2"):
        # (an upper-triangle walk leaves out what lies before a group: half the candidates)
        n = 100001 if metric == "l2-upper-tc" else 40001
        x = I.uniform_cube(n, 16, seed=3)
        sp, args, eps = oracle.Space(points=x), {"points": torch.from_numpy(x).cuda()}, 0.75
        if metric == "l2-upper-tc":
            opts = {"precision": 1, "upper_triangle": True}
    elif metric == "hamming":
        n = 40001
        rows = I.binary_codes(n, 64, n_centres=n, flip=0.5, seed=4)
        sp, args, eps = oracle.Space(bits=(rows, 64)), {"bits": (torch.from_numpy(rows).cuda(), 64)}, 18
    else:
        n = 30001
        data, off = I.random_strings(n, 20, 24, seed=5)
        sp = oracle.Space(strings=(data, off))
        args, eps = {"strings": (torch.from_numpy(data).cuda(), torch.from_numpy(off).cuda())}, 8
    csr = cg.eps_graph_query(cg.ct_build(**args), eps, **opts)
    assert csr.stats()["candidates"] > 256 * n
    got = csr.to_numpy()
    ids = np.sort(np.random.default_rng(1).choice(n, 200, replace=False))
    ref = oracle.brute_rows(sp, eps, ids)
    rp = got["row_ptr"]
    assert np.array_equal(np.diff(rp)[ids], np.diff(ref["row_ptr"]))
    assert np.array_equal(np.concatenate([got["col"][rp[i]:rp[i + 1]] for i in ids]), ref["col"])
