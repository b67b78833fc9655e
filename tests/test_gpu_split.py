"""The batched split passes at the edges of their tiles: row lengths at which
the lanes per row or the registers per lane change (and rows too long for
registers), hubs at and past the single-block limit, chunk remainders,
alphabets and string lengths at which the match masks change size.  The tree
is checked by the oracle's invariant checker, the graph by its brute force."""
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


@pytest.mark.parametrize("dim", [4, 8, 9, 16, 17, 28, 29, 32, 63, 64, 100, 125, 128, 129, 256, 500, 512, 1024, 1028])
@pytest.mark.parametrize("n", [513, 1100])
def test_l2_row_lengths(dim, n):
    x = np.concatenate([I.gmm_embedded(n - 40, dim=dim, intrinsic=min(dim, 5), n_centres=4, seed=dim),
                        np.zeros((40, dim), np.float32)])  # duplicates above the leaf size
    sp = oracle.Space(points=x)
    eps = float(np.float32(np.quantile(oracle.brute_rows(sp, 1e30, np.arange(6))["dist"], 0.05)))
    out = gpu_graph(points=x, eps=eps, leaf_size=8, export=True)
    assert_csr_matches(out, oracle.brute_force(sp, eps))
    # fp32 splits and the radius rounded up: 2^-16 + 2^-17 (as in the parity tests)
    code, msg = oracle.check_tree(sp, tree_from_export(out["tree"]), 2.5e-5)
    assert code == 0, msg


@pytest.mark.parametrize("n", [63, 64, 65, 129, 1000])
@pytest.mark.parametrize("alphabet,lo,hi", [(b"A", 0, 70), (b"ACGT", 60, 66), (b"ACGT", 120, 140),
                                            (bytes(range(256)), 100, 300), (bytes(range(256)), 600, 1000)])
def test_strings(n, alphabet, lo, hi):
    if hi >= 300:
        n = min(n, 129)
    data, off = I.random_strings(n, lo, hi, alphabet=alphabet, seed=n)
    data, off = np.concatenate([np.zeros(3, np.uint8), data]), off + 3  # strings that do not start the buffer
    sp = oracle.Space(strings=(data, off))
    out = gpu_graph(strings=(data, off), eps=0.5 * hi, leaf_size=4, export=True)
    assert_csr_matches(out, oracle.brute_force(sp, 0.5 * hi), integer_dist=True)
    code, msg = oracle.check_tree(sp, tree_from_export(out["tree"]), 0.0)
    assert code == 0, msg


@pytest.mark.parametrize("bits", [1, 128, 129, 256, 384, 512, 513, 4000])
@pytest.mark.parametrize("n", [255, 257, 1500])
def test_codes(bits, n):
    import torch
    from paper_2510_14147_gb300 import ctgraph as cg
    rows = I.binary_codes(n, bits, n_centres=9, flip=0.08, seed=bits)
    t = cg.ct_build(bits=(torch.from_numpy(rows).cuda(), bits), leaf_size=6)
    tree = cg.ct_tree_export(t)
    csr = cg.eps_graph_query(t, bits // 8)
    sp = oracle.Space(bits=(rows, bits))
    assert_csr_matches(csr.to_numpy(), oracle.brute_force(sp, bits // 8), integer_dist=True)
    code, msg = oracle.check_tree(sp, tree_from_export(tree), 0.0)
    assert code == 0, msg


@pytest.mark.parametrize("metric", ["l2-dim7", "l2-dim16", "bits"])
@pytest.mark.parametrize("centres", [[5], [0, 0, 1], [3, 700, 3, 12, 12, 900, 5]])
def test_forest_with_empty_and_small_cells(metric, centres):
    """The landmark form's trees are split together: repeated centres leave
    cells without points, and some cells hold fewer points than a leaf."""
    import torch
    from paper_2510_14147_gb300 import ctgraph as cg
    n = 1400
    if metric == "bits":
        rows = I.binary_codes(n, 96, n_centres=7, flip=0.06, seed=2)
        args, eps, sp = {"bits": (torch.from_numpy(rows).cuda(), 96)}, 9, oracle.Space(bits=(rows, 96))
    else:
        x = I.gmm_embedded(n, dim=int(metric[6:]), intrinsic=4, n_centres=7, seed=3)
        args, eps, sp = {"points": torch.from_numpy(x).cuda()}, 1.25, oracle.Space(points=x)
    for kw in ({}, {"upper_triangle": True}):
        csr, info = cg.eps_graph_query_landmark(centres, eps, **args, **kw)
        assert info["cells"] == len(centres)
        assert_csr_matches(csr.to_numpy(), oracle.brute_force(sp, eps), integer_dist=metric == "bits")
