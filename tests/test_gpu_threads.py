"""Calls from several host threads, each on its own stream, whose kernels need
different amounts of shared memory: one call's limit never holds for another's
launch.  Trees and graphs are those of the same calls made one after another."""
import threading

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


def _kinds(metric):
    """(arguments of ct_build, radius) of inputs that share kernels."""
    import torch
    if metric == "points":
        return [({"points": torch.from_numpy(I.gmm_embedded(900, dim=d, intrinsic=5, n_centres=6, seed=d)).cuda()}, 1.0)
                for d in (128, 252, 3400, 4096)]
    if metric == "bits":
        return [({"bits": (torch.from_numpy(I.binary_codes(900, b, n_centres=6, flip=0.1, seed=b)).cuda(), b)}, b // 6)
                for b in (512, 2048, 4096)]
    out = []
    for a in (20, 60, 256):  # match masks of 64 to 128 symbols: two words
        data, off = I.random_strings(300, 70, 120, alphabet=bytes(range(a)), seed=a)
        out.append(({"strings": (torch.from_numpy(data).cuda(), torch.from_numpy(off).cuda())}, 80))
    return out


@pytest.mark.parametrize("metric", ["points", "bits", "strings"])
def test_builds_and_queries_at_the_same_time(metric):
    import torch
    from paper_2510_14147_gb300 import ctgraph as cg
    kinds = _kinds(metric)
    refs = [cg.eps_graph_query(cg.ct_build(**a), e).to_numpy() for a, e in kinds]
    torch.cuda.synchronize()
    failed = []

    def work(a, e, ref):
        try:
            s = torch.cuda.Stream()
            for _ in range(30):
                t = cg.ct_build(**a, stream=s)
                got = cg.eps_graph_query(t, e, stream=s).to_numpy()
                t.free()
                for k in ("row_ptr", "col", "dist"):
                    assert np.array_equal(got[k], ref[k]), k
        except Exception as x:  # reported by the main thread
            failed.append(repr(x))

    threads = [threading.Thread(target=work, args=(a, e, r)) for (a, e), r in zip(kinds, refs)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not failed, failed
