"""Scratch memory per point of builds and queries: what the library's memory
pool grows by over one call, in a process of its own (the pool keeps the most
that was in use).  The bounds are sums of the arrays' sizes."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

COMMON = """
import torch
from paper_2510_14147_gb300 import ctgraph as cg
g = torch.Generator(device="cuda").manual_seed(1)
def strings(seeds, children, leaves, length):
    # seeds far apart, children 6 to 8 edits away, two more for the leaves
    s = torch.randint(4, (seeds, length), generator=g, device="cuda")
    for k, edits in ((children, 7), (leaves, 2)):
        s = s.repeat_interleave(k, 0)
        rows = torch.arange(s.shape[0], device="cuda")
        for _ in range(edits):
            s[rows, torch.randint(length, rows.shape, generator=g, device="cuda")] = torch.randint(4, rows.shape, generator=g, device="cuda")
    data = (s + 65).to(torch.uint8).reshape(-1)
    return data, torch.arange(s.shape[0] + 1, dtype=torch.int64, device="cuda") * length
def free():
    torch.cuda.synchronize()
    return torch.cuda.mem_get_info()[0]
"""


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2510_14147_gb300 import build
    build.build()


def _numbers(program):
    out = subprocess.run([sys.executable, "-c", COMMON + program], cwd=ROOT, stdout=subprocess.PIPE, check=True)
    return [float(v) for v in out.stdout.split()]


def test_build_of_rows_that_are_pruned():
    # zero columns leave the distances and the tree as they are: the difference is the rows (two
    # copies and the vertices' centres, of which there is at most one per point) and the distances
    # to a batch, 8 floats a point; 33 MB for the pool's granularity
    n = 2000000
    pruned, plain = [_numbers("""
cg.ct_build(points=torch.rand(5000, %d, generator=g, device="cuda")).free()
x = torch.zeros(%d, %d, device="cuda")
x[:, :3] = torch.rand(%d, 3, generator=g, device="cuda")
torch.cuda.empty_cache()
before = free()
t = cg.ct_build(points=x)
print(before - free())
""" % (dim, n, dim, n))[0] for dim in (20, 16)]
    assert pruned - plain <= n * (3 * 16 + 8 * 4) + (33 << 20)


def test_build_of_many_small_string_hubs():
    # 100 bytes of strings twice, vertices (2 n, 28 bytes), hubs (n, 88), labels and distances
    # (16), candidates and their pairs (28), distances to a batch (32), positions (8), the
    # partition (28) and at most as much again per child, chunks (at most one per two points,
    # 64): about 500; 8 KB per hub with two strings or more would be over 2000
    n, grown = _numbers("""
cg.ct_build(strings=strings(3, 5, 3, 60), leaf_size=1).free()
a = strings(60, 1000, 3, 60)
torch.cuda.empty_cache()
before = free()
t = cg.ct_build(strings=a, leaf_size=1)
print(a[1].numel() - 1, before - free())
""")
    assert grown <= 800 * n + (33 << 20)


def test_query_of_low_degree():
    # the candidate pool (256 entries of 4 bytes a point), a copy of the candidates in use (at
    # most a quarter of it), the walk's lists and the CSR's arrays (under 200): 1500; a list of
    # 192 edges a point whatever the degree would add 1536
    n, grown = _numbers("""
cg.eps_graph_query(cg.ct_build(points=torch.rand(5000, 3, generator=g, device="cuda")), 0.01).free()
t = cg.ct_build(points=torch.rand(2000000, 3, generator=g, device="cuda"))
torch.cuda.empty_cache()
before = free()
c = cg.eps_graph_query(t, 0.008)
assert c.stats()["emit_pairs"] == c.nnz and 2 < c.nnz / 2e6 < 8
print(2000000, before - free())
""")
    assert grown <= 1500 * n + (200 << 20)
