"""The Hamming leaf stage at the row lengths where its register blocking
changes (one, two and four 128-bit pieces, several chunks), with ragged
groups and tiles, in the forms that share it: integer parity with the
oracle's brute force."""
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


@pytest.mark.parametrize("dim", [128, 129, 256, 257, 512, 513, 1024, 1025])
@pytest.mark.parametrize("zeta", [5, 32])
def test_rows_of_every_register_form(dim, zeta):
    import torch
    from paper_2510_14147_gb300 import ctgraph as cg
    rows = I.binary_codes(1371, dim, n_centres=9, flip=0.08, seed=dim)
    eps = dim // 7
    sp = oracle.Space(bits=(rows, dim))
    t = cg.ct_build(bits=(torch.from_numpy(rows).cuda(), dim), leaf_size=zeta)
    pred = cg.ct_predictor_create(seed=1)
    cg.ct_predictor_fit(pred, t, eps, steps=50, seed=2)
    for inc in (False, True):
        ref = oracle.brute_force(sp, eps, include_self=inc)
        for opts in ({}, {"upper_triangle": True},
                     {"use_predictor": True, "predictor": pred, "upper_triangle": True}):
            got = cg.eps_graph_query(t, eps, include_self=inc, **opts).to_numpy()
            assert_csr_matches(got, ref, integer_dist=True)
