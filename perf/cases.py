"""The calls that users of the ε-graph library make, as measurable cases.

A case is one call pattern (``call``) on one kind of input (``data``):

  step      ct_build + eps_graph_query: a new point set, its graph, once
  query     eps_graph_query on a tree that the program keeps
  sweep     eps_graph_query_sweep: three radii over one kept tree
  batch     eps_graph_query_batched over the kept trees of many clouds
  plan      ct_plan_launch + ct_plan_result: a batch with kept buffers, replayed
  landmark  eps_graph_query_landmark: Voronoi cells of random centres

Inputs follow the recipes of ``paper_2510_14147_gb300/inputs.py`` (embedded
Gaussian mixtures, uniform cubes, mutated DNA strings, clustered bit codes),
drawn on the GPU.  The radius is calibrated on a sample of the input for the
case's mean degree, as the workloads of this repository are.
"""
import math

import torch

from paper_2510_14147_gb300 import ctgraph as cg


def _case(call, data, n, dim, degree, precision=0, learned=False, upper=False, include_self=False, clouds=1, cells=0):
    return {"call": call, "data": data, "n": n, "dim": dim, "degree": degree, "precision": precision,
            "learned": learned, "upper": upper, "include_self": include_self, "clouds": clouds, "cells": cells}


def listed():
    tuned = {"precision": 1, "learned": True, "upper": True}
    cases = {
        # the smallest call in use: a 3-D scan of 2000 points with a handful of neighbours, default options
        "scan_2k_3d": _case("step", "uniform", 2000, 3, 4),
        # an ordinary point cloud (odd size) with default options
        "cloud_32k_3d": _case("step", "uniform", 32300, 3, 22),
        # feature vectors of a mid-size data set, default options, self pairs kept (DBSCAN-style core counts)
        "features_174k_64d": _case("step", "gmm", 173645, 64, 87, include_self=True),
        # data in which a cover tree prunes little, through the tensor-core filter
        "uniform_121k_16d": _case("step", "uniform", 120831, 16, 21, precision=1, upper=True),
        # the main workload: a million 128-D descriptors, 70 neighbours, the fastest form
        "gmm_1m_k70": _case("step", "gmm", 1000000, 128, 70, **tuned),
        # a kept tree queried at a large radius: the largest output (about 500 M entries)
        "gmm_1m_k500_query": _case("query", "gmm", 1000000, 128, 500, **tuned),
        # sequence clustering: DNA reads under edit distance
        "dna_50k": _case("step", "dna", 50000, 96, 99, learned=True, upper=True),
        # binary descriptors under the Hamming distance
        "ham_1m_256": _case("step", "bits", 1000000, 256, 70, learned=True, upper=True),
        # three radii over one kept tree, as a parameter study runs them
        "sweep_300k_128d": _case("sweep", "gmm", 300007, 128, 300, precision=1, upper=True),
        # many clouds of mixed sizes, dimensions and densities in one call
        "batch_20_clouds": _case("batch", "mixed", 65536, 64, 90, precision=1, upper=True, clouds=20),
        # small clouds of fixed shape queried again and again (a serving loop): graph replay
        "plan_16_clouds": _case("plan", "mixed", 16261, 64, 60, clouds=16),
        # the landmark form at the paper's 60 centres
        "landmark_100k_64d": _case("landmark", "gmm", 96820, 64, 34, precision=1, cells=60),
    }
    return [dict(c, name=name) for name, c in cases.items()]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    call = rng.choice(["step", "step", "step", "query", "query", "strings", "codes", "sweep", "batch", "plan", "landmark"])
    form = rng.choice([{}, {}, {"precision": 1}, {"precision": 1, "upper": True}, {"upper": True},
                       {"precision": 1, "learned": True, "upper": True}, {"learned": True}])
    own = rng.random() < 0.25
    if call in ("step", "query"):
        data = rng.choice(["gmm", "gmm", "uniform"])
        dim = rng.choice([2, 3, 5, 16, 30, 64, 100, 128, 150]) if data == "gmm" else rng.choice([2, 3, 3, 7, 16])
        most = 60000 if data == "uniform" and dim > 3 else 1000000 if form.get("precision") and form.get("upper") else 250000
        n = _log(rng, 2000, most) | rng.randint(0, 1)
        return _case(call, data, n, dim, _log(rng, 4, 300 if n < 300000 else 100), include_self=own, **form)
    if call == "strings":
        return _case("step", "dna", _log(rng, 2000, 50000), rng.choice([60, 90, 96, 100, 130]), 99, include_self=own,
                     learned=form.get("learned", False), upper=form.get("upper", False))
    if call == "codes":
        return _case("step", "bits", _log(rng, 10000, 600000), rng.choice([64, 100, 128, 256, 300, 512]),
                     _log(rng, 10, 150), include_self=own, learned=form.get("learned", False), upper=True)
    if call == "sweep":
        return _case("sweep", "gmm", _log(rng, 10000, 300000), rng.choice([3, 16, 50, 128]), _log(rng, 40, 300),
                     include_self=own, **form)
    if call == "batch":
        return _case("batch", "mixed", _log(rng, 8000, 60000), 64, _log(rng, 20, 120), include_self=own,
                     precision=form.get("precision", 0), upper=form.get("upper", False), clouds=rng.randint(3, 20))
    if call == "plan":
        return _case("plan", "mixed", _log(rng, 4000, 25000), 64, _log(rng, 10, 80), include_self=own,
                     upper=form.get("upper", False), clouds=rng.randint(2, 16))
    return _case("landmark", "gmm", _log(rng, 10000, 60000), rng.choice([3, 16, 33, 64]), _log(rng, 10, 60),
                 precision=form.get("precision", 0), upper=form.get("upper", False), cells=rng.choice([10, 60]))


# ------------------------------------------------------------------ inputs

def _clouds(case):
    """The clouds of a case: (kind, n, dim, degree) each, by the case alone."""
    if case["data"] != "mixed":
        return [(case["data"], case["n"], case["dim"], case["degree"])]
    out = []
    for c in range(case["clouds"]):
        f = (c + 0.5) / case["clouds"]
        n = int(case["n"] * math.exp(1.4 * (f - 0.6))) + c          # sizes over a factor of four, some odd
        dim = (3, 16, case["dim"])[c % 3]
        kind = "uniform" if dim == 3 and c % 2 else "gmm"
        out.append((kind, n, dim, case["degree"] * math.exp(1.6 * (((7 * c) % case["clouds"]) / case["clouds"] - 0.5))))
    return out


def _points(g, kind, n, dim):
    if kind == "uniform":
        return torch.rand(n, dim, generator=g, device="cuda")
    k = min(8, dim)
    m = 100 if dim == 128 else max(1, n // 10000)
    centres = 5.0 * torch.randn(m, k, generator=g, device="cuda")
    q = torch.linalg.qr(torch.randn(dim, k, generator=g, device="cuda").double().cpu())[0].float().cuda()
    label = torch.randint(m, (n,), generator=g, device="cuda")
    z = centres[label] + torch.randn(n, k, generator=g, device="cuda")
    x = 0.01 * torch.randn(n, dim, generator=g, device="cuda")
    for j in range(k):
        x.addcmul_(z[:, j:j + 1], q[:, j][None, :])
    return x


def _strings(g, n, length):
    """Reads of about `length` bases: 100 mutants of each random seed string."""
    rnd = lambda *s: torch.rand(*s, generator=g, device="cuda")  # noqa: E731
    code = lambda hi, *s: torch.randint(hi, s, generator=g, device="cuda")  # noqa: E731
    seeds = code(4, (n + 99) // 100, length)
    seq = seeds.repeat_interleave(100, 0)[:n]
    u = rnd(n, length)
    sub = (u >= 0.005) & (u < 0.045)
    seq = torch.where(sub, (seq + 1 + code(3, n, length)) % 4, seq)
    pieces = torch.stack([code(4, n, length), seq], 2).reshape(n, -1)
    keep = torch.stack([rnd(n, length) < 0.005, u >= 0.005], 2).reshape(n, -1)
    offsets = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    offsets[1:] = keep.sum(1).cumsum(0)
    return torch.tensor(list(b"ACGT"), dtype=torch.uint8, device="cuda")[pieces[keep]], offsets


def _unpack(rows, bits):
    x = (rows[:, :, None] >> torch.arange(8, device="cuda", dtype=torch.uint8)) & 1
    return x.reshape(rows.shape[0], -1)[:, :bits].bool()


def _pack(x, bits):
    x = torch.nn.functional.pad(x.to(torch.uint8), (0, -bits % 8)).reshape(x.shape[0], -1, 8)
    return (x << torch.arange(8, device="cuda", dtype=torch.uint8)).sum(2, dtype=torch.uint8)


def _codes(g, n, bits):
    m = max(1, n // 1000)
    centres = torch.rand(m, bits, generator=g, device="cuda") < 0.5
    label = torch.randint(m, (n,), generator=g, device="cuda")
    return _pack(centres[label] ^ (torch.rand(n, bits, generator=g, device="cuda") < 0.05), bits)


def _signs(rows, bits):
    """Bit rows as +1 / -1: the distance of two is (bits - dot) / 2."""
    return 1.0 - 2.0 * _unpack(rows, bits).float()


def _radius(g, kind, x, dim, degree):
    """The radius at which a point has about `degree` neighbours, from 1024
    points against a sample of the others."""
    n = x.shape[0]
    m = min(n, 65536)
    ask = x[torch.randint(n, (1024,), generator=g, device="cuda")]
    rest = x if m == n else x[torch.randint(n, (m,), generator=g, device="cuda")]
    if kind == "bits":
        d = (dim - _signs(ask, dim) @ _signs(rest, dim).T) / 2
    else:
        c = rest.mean(0)
        d = torch.cdist(ask - c, rest - c)
    k = min(1024 * m, max(1, int(round(1024 * (degree + 1) * m / n))))
    r = float(d.reshape(-1).sort().values[k - 1])
    return float(int(r)) if kind == "bits" else float("%.4g" % r)


def _input(kind, n, dim, degree, draw_seed, seed):
    """(arguments of ct_build, radius).  The point set is drawn by `draw_seed`;
    `seed` gives another input of the same geometry -- the points in another
    order, the coordinates permuted and reflected (bits permuted and flipped,
    letters renamed) -- so that every input of a case has a graph of the same
    size."""
    g = torch.Generator(device="cuda").manual_seed(draw_seed)
    h = torch.Generator(device="cuda").manual_seed(seed)
    perm = lambda m: torch.randperm(m, generator=h, device="cuda")  # noqa: E731
    if kind == "dna":
        data, off = _strings(g, n, dim)
        p = perm(n)
        new = torch.zeros_like(off)
        new[1:] = (off[1:] - off[:-1])[p].cumsum(0)
        at = torch.arange(data.numel(), device="cuda")
        at += (off[:-1][p] - new[:-1]).repeat_interleave(new[1:] - new[:-1])
        letters = torch.zeros(256, dtype=torch.uint8, device="cuda")
        acgt = torch.tensor(list(b"ACGT"), device="cuda")
        letters[acgt] = acgt[perm(4)].to(torch.uint8)
        return {"strings": (letters[data[at].long()], new)}, 8.0
    if kind == "bits":
        rows = _codes(g, n, dim)
        eps = _radius(g, kind, rows, dim, degree)
        order, flip = perm(dim), torch.rand(dim, generator=h, device="cuda") < 0.5
        return {"bits": (_pack(_unpack(rows, dim)[:, order] ^ flip, dim)[perm(n)], dim)}, eps
    x = _points(g, kind, n, dim)
    eps = _radius(g, kind, x, dim, degree)
    sign = (torch.rand(dim, generator=h, device="cuda") < 0.5).float() * 2 - 1
    return {"points": (x[:, perm(dim)] * sign)[perm(n)]}, eps


def _inputs(case, seed, draw_seed=0):
    """[(build arguments, radius)] of the case's clouds."""
    return [_input(*cloud, draw_seed + 101 * c, 1000 * seed + c) for c, cloud in enumerate(_clouds(case))]


def _sweep(case):
    """Mean degrees of the three radii (sift's three in the paper: 10, 70 and 500 to one)."""
    return [max(2.0, case["degree"] / 30), max(3.0, case["degree"] / 5), case["degree"]]


def _sweep_radii(case):
    g = torch.Generator(device="cuda").manual_seed(7)
    x = _points(torch.Generator(device="cuda").manual_seed(0), case["data"], case["n"], case["dim"])
    return [_radius(g, case["data"], x, case["dim"], d) for d in _sweep(case)]


def prepare(case, seed):
    made = _inputs(case, seed)
    s = {"call": case["call"], "args": made[0][0], "eps": made[0][1], "radii": [e for _, e in made]}
    s["opts"] = {"precision": case["precision"], "upper_triangle": case["upper"], "include_self": case["include_self"]}
    if case["learned"]:
        # fitted once by the program, on another draw of the same recipe
        fit_args, fit_eps = _inputs(case, seed, draw_seed=50)[0]
        s["opts"].update(use_predictor=True, predictor=cg.ct_predictor_create(seed=1))
        tree = cg.ct_build(**fit_args)
        cg.ct_predictor_fit(s["opts"]["predictor"], tree, fit_eps, include_self=case["include_self"], seed=2)
        tree.free()
    if case["call"] in ("query", "sweep", "batch", "plan"):
        s["trees"] = [cg.ct_build(**args) for args, _ in made]
    if case["call"] == "sweep":
        s["radii"] = _sweep_radii(case)
    if case["call"] == "plan":
        s["plan"] = cg.ct_plan_create(s["trees"], s["radii"], **s["opts"])
    if case["call"] == "landmark":
        g = torch.Generator().manual_seed(seed)
        s["centres"] = torch.randperm(case["n"], generator=g)[:case["cells"]].numpy()
    return s


def _graph(csr):
    return {"row_ptr": csr.row_ptr, "col": csr.col, "dist": csr.dist}


def run(state):
    call, opts = state["call"], state["opts"]
    if call == "step":
        return _graph(cg.eps_graph_query(cg.ct_build(**state["args"]), state["eps"], **opts))
    if call == "query":
        return _graph(cg.eps_graph_query(state["trees"][0], state["eps"], **opts))
    if call == "sweep":
        return [_graph(c) for c in cg.eps_graph_query_sweep(state["trees"][0], state["radii"], **opts)]
    if call == "batch":
        return [_graph(c) for c in cg.eps_graph_query_batched(state["trees"], state["radii"], **opts)]
    if call == "plan":
        cg.ct_plan_launch(state["plan"])
        out = [_graph(c) for c in cg.ct_plan_result(state["plan"])]
        for graph in out:   # the graphs are views into the plan's buffers: they keep it
            for t in graph.values():
                t.plan = state["plan"]
        return out
    return _graph(cg.eps_graph_query_landmark(state["centres"], state["eps"], **state["args"], **opts)[0])


def work(case):
    """Each input read once, each graph written once (row_ptr 8 B per row, col and
    dist 8 B per entry); the distance of every pair of neighbours once."""
    nbytes = flops = 0.0
    for kind, n, dim, degree in _clouds(case):
        row = {"dna": dim, "bits": dim / 8}.get(kind, 4.0 * dim)
        pair = {"dna": 17.0 * dim * math.ceil(dim / 64), "bits": 3 * dim / 32}.get(kind, 3.0 * dim)
        degrees = _sweep(case) if case["call"] == "sweep" else [degree]
        edges = n * sum(degrees)
        nbytes += n * row + 8.0 * (n + 1) * len(degrees) + 8.0 * edges
        flops += pair * n * max(degrees) / 2
    return {"bytes": nbytes, "flops": flops}


# ------------------------------------------------------------------- exact

def _exact_graph(kind, args, eps, include_self):
    """Brute force: every pair whose distance, in 64 bits, is at most eps.  An
    fp32 product of the centred rows (signs for bits) first drops the
    pairs that are far outside it."""
    x, dim = args["bits"] if kind == "bits" else (args["points"], args["points"].shape[1])
    n = x.shape[0]
    if kind == "bits":
        a = _signs(x, dim)
    else:
        a = (x.double() - x.double().mean(0)).float()
        sq = (a * a).sum(1)
        top = float(sq.max())
    rows, cols, dist = [], [], []
    step = max(1, (1 << 28) // n)
    for at in range(0, n, step):
        p = a[at:at + step] @ a.T
        if kind == "bits":
            keep = (dim - p) / 2 <= eps + 0.25
        else:
            keep = p.mul_(-2).add_(sq[at:at + step, None]).add_(sq[None, :]) <= eps * eps * 1.001 + 1e-5 * top
        i, j = keep.nonzero(as_tuple=True)
        del p, keep
        for b in range(0, i.numel(), 1 << 24):
            u, v = i[b:b + (1 << 24)] + at, j[b:b + (1 << 24)]
            d2 = torch.zeros(u.numel(), dtype=torch.float64, device="cuda")
            for k in range(0, a.shape[1], 16):   # 16 coordinates at a time: less memory
                if kind == "bits":
                    d2 += (a[u, k:k + 16] != a[v, k:k + 16]).sum(1)
                else:
                    d2 += (x[u, k:k + 16].double() - x[v, k:k + 16].double()).square().sum(1)
            near = d2 <= (eps if kind == "bits" else eps * eps)
            if not include_self:
                near &= u != v
            rows.append(u[near])
            cols.append(v[near])
            dist.append(d2[near] if kind == "bits" else d2[near].sqrt())
    ptr = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    ptr[1:] = torch.bincount(torch.cat(rows), minlength=n).cumsum(0)
    return {"row_ptr": ptr, "col": torch.cat(cols).to(torch.int32), "dist": torch.cat(dist)}


def exact(case, seed):
    clouds = _clouds(case)
    # edit distance is in whole numbers, which are compared as they are; larger inputs would take too long
    if case["data"] == "dna" or sum(n * n for _, n, _, _ in clouds) > 6e10:
        return None
    made = _inputs(case, seed)
    if case["call"] == "sweep":
        made = [(made[0][0], eps) for eps in _sweep_radii(case)]
        clouds = clouds * len(made)
    out = [_exact_graph(c[0], args, eps, case["include_self"]) for c, (args, eps) in zip(clouds, made)]
    return out if case["call"] in ("sweep", "batch", "plan") else out[0]
