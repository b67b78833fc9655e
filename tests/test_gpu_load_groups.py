"""A tree file whose query groups hold more points than a group may: the
Hamming leaf stage keeps a group's queries in arrays of 32, so such a Hamming
file is refused when it is read (no query runs); the L2 stages take larger
groups in chunks."""
import struct

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


def _checksum(raw):
    h = 1469598103934665603
    for b in raw:
        h = ((h ^ b) * 1099511628211) & 0xffffffffffffffff
    return struct.pack("<Q", h)


def _with_group_count(raw, hamming, count):
    """The file with the first group's point count replaced."""
    version, metric, dim, dp, leaf, max_len, n, sbytes = struct.unpack_from("<I5i2q", raw, 8)
    nodes, leaves, depth, max_leaf, groups, max_group = struct.unpack_from("<6i", raw, 48)
    assert len(raw) == 72 + 4 * (n * dp + 2 * n + 7 * nodes + (0 if hamming else nodes * dp) + leaves + 4 * groups) + 8
    at = len(raw) - 8 - 3 * 4 * groups  # group counts, radii, order
    body = raw[:at] + struct.pack("<i", count) + raw[at + 4:-8]
    return body + _checksum(body)


@pytest.mark.parametrize("metric", ["bits", "points"])
def test_group_sizes_of_a_file(metric, tmp_path):
    import torch
    from paper_2510_14147_gb300 import ctgraph as cg
    if metric == "bits":
        rows = I.binary_codes(200, 64, n_centres=5, flip=0.1, seed=3)
        tree = cg.ct_build(bits=(torch.from_numpy(rows).cuda(), 64))
    else:
        tree = cg.ct_build(points=torch.from_numpy(I.uniform_cube(200, 3, seed=3)).cuda())
    path = str(tmp_path / "t.cttree")
    cg.ct_tree_save(tree, path)
    tree.free()
    raw = open(path, "rb").read()
    for count, taken in ((1, True), (32, True), (33, metric == "points"), (0, False), (201, False)):
        with open(path, "wb") as f:
            f.write(_with_group_count(raw, metric == "bits", count))
        if taken:
            cg.ct_tree_load(path).free()
        else:
            with pytest.raises(cg.CtError) as e:
                cg.ct_tree_load(path)
            assert e.value.status == cg.CT_EINVAL
