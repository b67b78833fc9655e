"""Edit distance within a band of one 32-bit or 64-bit word: string lengths
around the words' ends, bounds on both sides of the two word lengths, in the
walk, the leaf stage and the build; integer parity with the oracle's brute
force."""
import numpy as np
import pytest

import oracle
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


def _mutants(n, length, symbols, seed):
    rng = np.random.default_rng(seed)
    seeds = [rng.integers(0, symbols, length).astype(np.uint8) + 65 for _ in range(7)]
    out = []
    for i in range(n):
        s = list(seeds[i % 7])
        for _ in range(int(rng.integers(0, length // 2))):
            at, kind = int(rng.integers(0, len(s))), int(rng.integers(0, 3))
            if kind == 0 and len(s) > 1:
                del s[at]
            elif kind == 1 and len(s) < length + 6:
                s.insert(at, np.uint8(rng.integers(0, symbols) + 65))
            else:
                s[at] = np.uint8(rng.integers(0, symbols) + 65)
        out.append(np.array(s, dtype=np.uint8))
    off = np.concatenate([[0], np.cumsum([len(s) for s in out])]).astype(np.int64)
    return np.concatenate(out), off


@pytest.mark.parametrize("length,symbols", [(62, 4), (65, 2), (96, 4), (127, 20), (260, 4)])
def test_band_words(length, symbols):
    import torch
    from paper_2510_14147_gb300 import ctgraph as cg
    data, off = _mutants(400, length, symbols, seed=length)
    sp = oracle.Space(strings=(data, off))
    t = cg.ct_build(strings=(torch.from_numpy(data).cuda(), torch.from_numpy(off).cuda()))
    for eps in (0, 1, 13, 31, 32, 63, 64):
        ref = oracle.brute_force(sp, eps)
        for opts in ({}, {"upper_triangle": True}):
            assert_csr_matches(cg.eps_graph_query(t, eps, **opts).to_numpy(), ref, integer_dist=True)
