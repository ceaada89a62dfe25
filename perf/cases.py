"""The work that users of this library have it do, as measurable cases.

An index of this library is a set of vectors resident on the GPU with a base
graph over them.  A program tunes the base to one or several (alpha, R)
targets and stores or searches the results (``tune``, ``search``), answers
mixed requests against several tuned graphs at once (``mixed``), builds a base
(``vamana``), computes exact neighbours (``knn``) and loads stored indexes
(``load``).  Data come in the four shapes of ``datagen``: 128-d uint8
descriptors (sift), 96-d unit float embeddings (deep), 960-d float descriptors
(gist) and small 32-d float sets (tiny); their distributions are drawn here on
the GPU by the same recipes.  Sizes are those of the benchmark, its targets
and its query batches, with n cut so that an index is built in about a second.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2602_08097_gb300 as rp

# (alpha, R) sweeps of the benchmark's workloads, as text so that a case stays a dict of plain values
SIFT_SWEEP = "1.1:64 1.05:48 1.0:32"
DEEP_SWEEP = "1.15:64 1.15:48 1.1:64 1.1:48 1.05:64 1.05:48 1.0:64 1.0:48"
GIST_SWEEP = "1.175:64 1.15:64 1.125:64 1.1:64 1.075:64 1.05:64 1.025:64 1.0:64 1.0:32"


def listed():
    return [
        # one target on a small index, the smallest call a tuning loop makes: launches and host work count
        dict(name="tune tiny one", kind="tune", data="tiny", n=2000, d=32, targets="1.1:32", variant="sorted"),
        # the uint8 sweep: three targets in one launch
        dict(name="tune sift sweep", kind="tune", data="sift", n=400000, d=128, targets=SIFT_SWEEP, variant="sorted"),
        # the float sweep of the default benchmark: eight targets over a Vamana base
        dict(name="tune deep sweep", kind="tune", data="deep", n=400000, d=96, targets=DEEP_SWEEP, variant="sorted"),
        # the same on wide rows, nine targets
        dict(name="tune gist sweep", kind="tune", data="gist", n=30000, d=960, targets=GIST_SWEEP, variant="sorted"),
        # one query from host memory: the latency of an interactive search
        dict(name="search deep one", kind="search", data="deep", n=400000, d=96, targets="1.1:64", nq=1, L=100, k=100,
             host=True),
        # offline batches on the three shapes, the benchmark's query counts and list sizes
        dict(name="search sift batch", kind="search", data="sift", n=400000, d=128, targets="1.1:64", nq=10000, L=128,
             k=100, host=False),
        dict(name="search deep batch", kind="search", data="deep", n=400000, d=96, targets="1.1:64", nq=10000, L=100,
             k=100, host=False),
        dict(name="search gist batch", kind="search", data="gist", n=30000, d=960, targets="1.1:64", nq=1000, L=200,
             k=100, host=False),
        # one round of a server: ragged requests on the base and three tuned graphs, host buffers
        dict(name="mixed sift round", kind="mixed", data="sift", n=200000, d=128, targets=SIFT_SWEEP, nq=333, Lmin=100,
             Lmax=256, k=100),
        # building a base index, two passes
        dict(name="vamana deep build", kind="vamana", data="deep", n=30000, d=96, R=64, L=75),
        # ground truth of a query set
        dict(name="knn deep truth", kind="knn", data="deep", n=400000, d=96, nq=10000, k=100),
        # a stored index from host memory, its start vertex not stored with it
        dict(name="load deep index", kind="load", data="deep", n=200000, d=96, host=True, start=False),
    ]


def _log(rng, lo, hi):
    """A whole number between lo and hi, spread over the logarithm."""
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _shape(rng, most):
    """A data shape, its width and an n of up to ``most`` rows (fewer of the wide ones)."""
    data = rng.choice(["sift", "deep", "deep", "gist", "tiny"])
    d = {"sift": rng.choice([96, 100, 128, 128, 200]), "deep": rng.choice([64, 96, 96, 100, 200]),
         "gist": rng.choice([384, 777, 960]), "tiny": rng.choice([17, 32, 50])}[data]
    top = {"sift": most, "deep": most, "gist": min(most, 25000), "tiny": min(most, 20000)}[data]
    return dict(data=data, n=_log(rng, 2000, top), d=d)


def _targets(rng, count):
    return " ".join("%s:%d" % (round(rng.randrange(1000, 1191, 5) / 1000, 3), rng.choice([24, 32, 48, 64]))
                    for _ in range(count))


def draw(rng):
    kind = rng.choice(["tune", "tune", "tune", "search", "search", "search", "search", "mixed", "vamana", "knn", "load"])
    if kind == "tune":
        c = dict(kind=kind, **_shape(rng, 300000), targets=_targets(rng, rng.choice([1, 1, 2, 3, 5, 8])),
                 variant=rng.choice(["sorted", "sorted", "unsorted"]))
    elif kind == "search":
        k = rng.choice([1, 10, 100])
        c = dict(kind=kind, **_shape(rng, 300000), targets=_targets(rng, 1), nq=_log(rng, 1, 9000),
                 L=_log(rng, max(k, 32), 256), k=k, host=rng.random() < 0.4)
        if c["d"] > 256:
            c["nq"] = min(c["nq"], 900)
    elif kind == "mixed":
        Lmin = _log(rng, 100, 160)
        c = dict(kind=kind, **_shape(rng, 200000), targets=_targets(rng, rng.choice([2, 3, 4])), nq=_log(rng, 16, 2000),
                 Lmin=Lmin, Lmax=Lmin + _log(rng, 1, 96), k=rng.choice([10, 100]))
        if c["d"] > 256:
            c["nq"] = min(c["nq"], 500)
    elif kind == "vamana":
        c = dict(kind=kind, **_shape(rng, 25000), R=rng.choice([32, 48, 64]), L=rng.choice([50, 64, 75]))
        if c["d"] > 256:
            c["n"] = min(c["n"], 5000)
    elif kind == "knn":
        c = dict(kind=kind, **_shape(rng, 300000), nq=_log(rng, 10, 8000), k=rng.choice([10, 64, 100, 128]))
        if c["d"] > 128:
            c["nq"] = min(c["nq"], 1500)
    else:
        c = dict(kind=kind, **_shape(rng, 180000), host=rng.random() < 0.6, start=rng.random() < 0.5)
    return c


# ---- inputs -------------------------------------------------------------------------------------------------------
def _vectors(case, seed, nq):
    """The base vectors and nq queries of the same distribution, on the GPU."""
    n, d, data = case["n"], case["d"], case["data"]
    torch.manual_seed(seed)
    rows, dev = n + nq, "cuda"
    if data == "sift":
        g = torch.distributions.Gamma(torch.tensor(0.6, device=dev), torch.tensor(1 / 40.0, device=dev))
        X = g.sample((rows, d)).clamp_(max=255.0).round_().to(torch.uint8)
    elif data == "gist":
        X = torch.randn(rows, d, device=dev).abs_().mul_(0.05)
        X = X / X.norm(dim=1, keepdim=True)
    else:
        ncent, sigma = (16, 2.0) if data == "tiny" else (256, 1.0)
        centres = torch.randn(ncent, d, device=dev) * sigma
        X = torch.randn(rows, d, device=dev)
        if data == "deep":
            X *= 1.5 * torch.arange(1, d + 1, device=dev, dtype=torch.float32) ** -0.75
        X += centres[torch.randint(0, ncent, (rows,), device=dev)]
        if data == "deep":
            X = X / X.norm(dim=1, keepdim=True)
    return X[:n].contiguous(), X[n:].contiguous()


def _parse(targets):
    pairs = [t.split(":") for t in targets.split()]
    return [float(a) for a, _ in pairs], [int(r) for _, r in pairs]


_ctx = _stream = None


def _context():
    """The process's one context, on the stream that the program's own tensors are used on."""
    global _ctx, _stream
    if _ctx is None:
        _stream = torch.cuda.Stream()
        _ctx = rp.rp_create(0, stream=_stream)
    return _ctx


class State(dict):
    """What a program holds: buffers and graph handles; the graphs go when it does."""

    def __del__(self):
        for g in self.pop("held", []):
            rp.rp_graph_free(_ctx, g)


def _base(ctx, data_graph, case):
    """The base graph: Vamana over embeddings, kNN candidates pruned to (1.2, 64) over the others."""
    if case["data"] == "deep":
        return rp.rp_build_vamana(ctx, data_graph, [1.0, 1.2], 64, 75)[0]
    return rp.rp_build_knn_base(ctx, data_graph, min(128, case["n"] - 1), 1.2, 64)


def prepare(case, seed):
    ctx = _context()
    torch.cuda.synchronize()
    with torch.cuda.stream(_stream):
        s = _prepare(ctx, case, seed)
        rp.rp_sync(ctx)
    torch.cuda.synchronize()
    return s


def _prepare(ctx, case, seed):
    kind = case["kind"]
    s = State(case=case, held=[])
    X, Q = _vectors(case, seed, case.get("nq", 0))
    data = rp.rp_load_graph(ctx, X)
    s["held"].append(data)
    s["data"] = data
    if kind == "tune":
        s["base"] = _base(ctx, data, case)
        s["held"].append(s["base"])
        s["alphas"], s["Rs"] = _parse(case["targets"])
    elif kind in ("search", "mixed"):
        base = _base(ctx, data, case)
        alphas, Rs = _parse(case["targets"])
        s["graphs"] = [base] + rp.rp_tune_batch(ctx, base, alphas, Rs)
        s["held"] += s["graphs"]
        host = case.get("host", True)
        s["queries"] = Q.cpu().numpy() if host else Q
        if kind == "mixed":
            r = np.random.default_rng(seed)
            s["q_graph"] = r.integers(0, len(s["graphs"]), case["nq"]).astype(np.int32)
            s["q_L"] = r.integers(case["Lmin"], case["Lmax"] + 1, case["nq"]).astype(np.int32)
    elif kind == "knn":
        s["queries"], s["X"] = Q, X
    elif kind == "load":
        # the stored form of an index: vectors, CSR and, if kept with it, the start vertex
        base = _base(ctx, data, case)
        row_ptr, col = rp.rp_graph_export(ctx, base, device="cuda")
        s["start"] = rp.rp_graph_info(ctx, base)["start"] if case["start"] else -1
        rp.rp_graph_free(ctx, base)
        if case["host"]:
            s["X"], s["row_ptr"], s["col"] = (t.cpu().numpy() for t in (X, row_ptr, col))
        else:
            s["X"], s["row_ptr"], s["col"] = X, row_ptr, col.contiguous()
    if kind in ("tune", "vamana", "load"):
        # where the program keeps the lists of each graph that a pass makes: R entries a node at most
        most = s["Rs"] if kind == "tune" else [case.get("R", 64)]
        s["store"] = [torch.zeros(case["n"] * min(r, 64), dtype=torch.int32, device="cuda") for r in most]
    return s


# ---- one pass -----------------------------------------------------------------------------------------------------
def _take(ctx, g, store):
    """The graph as the program keeps it (CSR on the device, the lists in its own buffer); its handle is released."""
    row_ptr, col = rp.rp_graph_export(ctx, g, device="cuda")
    store[:col.shape[0]].copy_(col)
    rp.rp_graph_free(ctx, g)
    return {"row_ptr": row_ptr, "col": store}


def run(state):
    ctx = _context()
    with torch.cuda.stream(_stream):
        return _run(ctx, state, state["case"])


def _run(ctx, state, case):
    kind = case["kind"]
    if kind == "tune":
        variant = rp.RP_UNSORTED if case["variant"] == "unsorted" else rp.RP_SORTED
        if len(state["alphas"]) == 1:
            graphs = [rp.rp_tune(ctx, state["base"], state["alphas"][0], state["Rs"][0], variant)]
        else:
            graphs = rp.rp_tune_batch(ctx, state["base"], state["alphas"], state["Rs"], variant)
        return [_take(ctx, g, to) for g, to in zip(graphs, state["store"])]
    if kind == "search":
        ids, dists = rp.rp_search(ctx, state["graphs"][1], state["queries"], case["L"], case["k"])
        return {"ids": ids, "dists": dists}
    if kind == "mixed":
        ids, dists = rp.rp_search_multi(ctx, state["graphs"], state["q_graph"], state["q_L"], state["queries"],
                                        case["k"])
        return {"ids": ids, "dists": dists}
    if kind == "vamana":
        g, cut = rp.rp_build_vamana(ctx, state["data"], [1.0, 1.2], case["R"], case["L"])
        return dict(_take(ctx, g, state["store"][0]), cut=cut)
    if kind == "knn":
        ids, dists = rp.rp_knn(ctx, state["data"], state["queries"], case["k"])
        return {"ids": ids, "dists": dists}
    g = rp.rp_load_graph(ctx, state["X"], state["row_ptr"], state["col"], state["start"])
    info = rp.rp_graph_info(ctx, g)
    return dict(_take(ctx, g, state["store"][0]), **info)


# ---- what a pass cannot do without ----------------------------------------------------------------------------------
def work(case):
    """Bytes: inputs read once, outputs written once.  Flops: the distances and Grams of the method itself.

    Degrees are not known from a case: a base of R = 64 holds about 56 edges a
    node, a graph tuned to (alpha, R) about min(R, 16 + 200 (alpha - 1)).
    """
    n, d, b = case["n"], case["d"], 1 if case["data"] == "sift" else 4
    kind, m = case["kind"], 56
    vec, base = n * d * b, (n + 1) * 8 + 4 * n * m
    deg = [min(r, 16 + 200 * (a - 1)) for a, r in zip(*_parse(case["targets"]))] if "targets" in case else [m]
    if kind == "tune":
        out = sum((n + 1) * 8 + 4 * n * k for k in deg)
        return {"bytes": vec + base + out, "flops": n * (3 * m * d + m * m * d)}  # keys, half the Gram
    if kind in ("search", "mixed"):
        nq, k = case["nq"], case["k"]
        L = case["L"] if kind == "search" else (case["Lmin"] + case["Lmax"]) / 2
        mean = sum(deg) / len(deg)
        seen = nq * L * mean * 0.5  # about half the neighbours met are new to their query
        return {"bytes": min(seen, n) * d * b + min(nq * L, n) * (16 + 4 * mean) + nq * (d * b + 8 * k),
                "flops": seen * 3 * d}
    if kind == "vamana":
        pool = 1.3 * case["L"] + case["R"]  # two passes: a search, a prune of its visited points
        return {"bytes": vec + (n + 1) * 8 + 4 * n * case["R"],
                "flops": 2 * n * (1.3 * case["L"] * case["R"] * 0.25 * 3 * d + pool * case["R"] * 3 * d)}
    if kind == "knn":
        return {"bytes": vec + case["nq"] * (d * b + 8 * case["k"]), "flops": 2 * case["nq"] * n * d}
    return {"bytes": 2 * (vec + base) + (0 if case["start"] else 2 * vec), "flops": 0 if case["start"] else 4 * n * d}


def exact(case, seed):
    """Exact neighbours' distances in 64 bits; what else a pass returns are whole
    numbers, or distances of points that a search over this library's graph met."""
    if case["kind"] != "knn":
        return None
    X, Q = _vectors(case, seed, case["nq"])
    X, k = X.double(), case["k"]
    xx = (X * X).sum(1)
    out = []
    for q in Q.double().split(max(1, int(3e8 // case["n"]))):
        near = torch.topk(xx[None, :] - 2.0 * (q @ X.T), k + 8, largest=False).indices  # short of |q|^2
        d2 = torch.cat([((X[i] - r[:, None, :]) ** 2).sum(2) for i, r in zip(near.split(256), q.split(256))])
        out.append(torch.sort(d2, dim=1).values[:, :k])
    return {"ids": None, "dists": torch.cat(out)}
