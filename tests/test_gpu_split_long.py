"""Splits of long rows and strings: rows that the selection does not stage
(above 256 floats), batches of a few centres (3 at 4096 floats, 6 of long
strings of many symbols), fewer candidates than lanes, duplicates.  The tree is checked by the oracle's invariant checker, the
graph by its brute force."""
import numpy as np
import pytest

import oracle
from paper_2510_14147_gb300 import inputs as I
from helpers import assert_csr_matches, gpu_graph, tree_from_export

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2510_14147_gb300 import build
    build.build()
    oracle.build()


@pytest.mark.parametrize("dim", [257, 260, 300, 1025, 2052, 4093, 4096])
@pytest.mark.parametrize("kind,n", [("gmm", 40), ("gmm", 1500), ("uniform", 700)])
def test_l2_long_rows(dim, kind, n):
    x = I.gmm_embedded(n, dim=dim, intrinsic=5, n_centres=4, seed=dim) if kind == "gmm" else I.uniform_cube(n, dim, seed=dim)
    x[n // 2:n // 2 + 15] = x[1]
    sp = oracle.Space(points=x)
    eps = float(np.float32(np.quantile(oracle.brute_rows(sp, 1e30, np.arange(6))["dist"], 0.05)))
    out = gpu_graph(points=x, eps=eps, leaf_size=4, export=True)
    assert_csr_matches(out, oracle.brute_force(sp, eps))
    # fp32 splits and the radius rounded up: 2^-16 + 2^-17 (as in the parity tests)
    code, msg = oracle.check_tree(sp, tree_from_export(out["tree"]), 2.5e-5)
    assert code == 0, msg


@pytest.mark.parametrize("symbols,length", [(256, 512), (256, 1024), (81, 1024), (79, 1000), (161, 512)])
@pytest.mark.parametrize("n", [43, 130])
def test_strings_of_many_symbols(symbols, length, n):
    alphabet = bytes((np.arange(symbols) + 20 & 255).astype(np.uint8))
    data, off = I.random_strings(n, length - 90, length, alphabet=alphabet, seed=n)
    sp = oracle.Space(strings=(data, off))
    out = gpu_graph(strings=(data, off), eps=0.9 * length, leaf_size=4, export=True)
    assert_csr_matches(out, oracle.brute_force(sp, 0.9 * length), integer_dist=True)
    code, msg = oracle.check_tree(sp, tree_from_export(out["tree"]), 0.0)
    assert code == 0, msg
