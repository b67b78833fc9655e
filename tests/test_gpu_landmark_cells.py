"""The landmark form's cell and ghost passes at the edges of their tiles (64
points, 64 centres, 32 words of a row): the CSR equals the oracle's brute
force and every point is a member of one cell of its own."""
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


@pytest.mark.parametrize("metric", ["l2", "hamming"])
@pytest.mark.parametrize("n,m,dim", [(1, 1, 1), (63, 63, 31), (64, 64, 32), (65, 65, 33), (300, 129, 70)])
def test_cells_at_tile_edges(metric, n, m, dim):
    import torch
    from paper_2510_14147_gb300 import ctgraph as cg
    centres = np.random.default_rng(n).permutation(n)[:m]
    if metric == "l2":
        x = I.gmm_embedded(n, dim=dim, intrinsic=min(dim, 4), n_centres=min(n, 5), seed=n)
        sp, args = oracle.Space(points=x), {"points": torch.from_numpy(x).cuda()}
        eps = float(np.float32(np.quantile(oracle.brute_rows(sp, 1e30, [0])["dist"], 0.1))) if n > 1 else 1.0
    else:
        rows = I.binary_codes(n, dim, n_centres=min(n, 5), flip=0.1, seed=n)
        sp, args, eps = oracle.Space(bits=(rows, dim)), {"bits": (torch.from_numpy(rows).cuda(), dim)}, dim // 6
    got, info = cg.eps_graph_query_landmark(centres, eps, **args)
    assert info["cells"] == m and info["members"] == n + info["ghosts"]
    assert_csr_matches(got.to_numpy(), oracle.brute_force(sp, eps), integer_dist=metric == "hamming")
