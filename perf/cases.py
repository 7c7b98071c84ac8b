"""Measured cases: the calls that a program clustering with this package makes.

A K-center solve loads a dataset, takes a farthest-first start, bounds and
tightens batches of branch-and-bound nodes over the samples, evaluates
candidate center sets and loops until the bounds meet.  The cases are those
calls, one by one and as whole solves, through the package's public classes,
from a thousand samples (latency) to a hundred million (one node streamed from
HBM), in float32 and float64, on the shapes of the package's own workloads
(synth.WORKLOADS, bench.py) and of the paper's real data sets (D = 12, 29, 68).

Inputs are Gaussian mixtures as in the package's recipes, drawn on the GPU from
the seed.  Node boxes come in the three forms its calls meet:
  nested    boxes shrinking around one sample per cluster (bench.py's batch);
  frontier  open nodes of a branch and bound: dyadic cells of the root box near
            good centers, as sibling pairs split on their longest side;
  around    boxes of 5 to 40 % of the data's range around the farthest-first
            centers (the package's tightening benchmark).
"""
import math

import torch

import paper_2301_00061_gb300 as kcm

# Component weights, sigma range, range of the means, share of uniform outliers.
MIXES = {
    "blobs": (None, 0.5, 2.0, 20.0, 0.0),             # equal weights, as many blobs as clusters
    "weights": ((0.6, 0.3, 0.1), 1.0, 1.0, 10.0, 0.0),
    "outliers": (None, 1.0, 1.0, 10.0, 0.01),
}


def listed():
    return [
        # one batch of children of a small double-precision instance: a call's latency
        dict(name="bounds-small", op="bounds", dtype="f64", n=1_000, d=2, k=3, b=16, mix="blobs", boxes="frontier"),
        # one node over the largest resident dataset of the benchmark: streams HBM
        dict(name="bounds-node", op="bounds", dtype="f32", n=100_000_000, d=2, k=4, b=1, mix="outliers",
             boxes="frontier"),
        # the package's headline batch
        dict(name="bounds-batch", op="bounds", dtype="f32", n=10_000_000, d=8, k=5, b=256, mix="blobs",
             boxes="nested"),
        # children of a wide instance (the paper's HIGGS has 29 attributes), ragged N
        dict(name="bounds-wide", op="bounds", dtype="f32", n=1_000_003, d=29, k=3, b=64, mix="blobs",
             boxes="frontier"),
        # children bounded over the quarter of the samples that sample reduction left
        dict(name="subset", op="subset", dtype="f32", n=10_000_000, d=4, k=3, b=8, part=4, mix="weights",
             boxes="frontier"),
        # a batch's candidate center sets in double precision
        dict(name="objective", op="objective", dtype="f64", n=1_000_000, d=3, k=3, b=64, mix="weights"),
        # the paper's heuristic column: farthest-first traversal from 100 random starts
        dict(name="fft", op="fft", dtype="f32", n=10_000_000, d=4, k=3, b=100, mix="weights"),
        # one batch of open nodes tightened at the batched-solve shape
        dict(name="tighten", op="tighten", dtype="f32", n=1_000_000, d=4, k=3, b=256, cap=0, mix="weights"),
        # a shape beyond the compiled ones (the paper's Taxi has 12 attributes), ragged N
        dict(name="tighten-wide", op="tighten", dtype="f32", n=200_003, d=12, k=5, b=32, cap=0, mix="blobs"),
        # a dataset from pinned host rows to its root box and first incumbent
        dict(name="load", op="load", dtype="f32", n=10_000_000, d=8, k=5, host=True, mix="blobs"),
        # a whole small solve in double precision (shared sample set, sample reduction)
        dict(name="solve-small", op="solve", dtype="f64", n=1_000, d=2, k=3, nodes=512, mix="blobs"),
        # the first batches of a batched solve (per-node sample lists), where the lists are longest
        dict(name="solve", op="solve", dtype="f32", n=1_000_000, d=4, k=3, nodes=2048, mix="weights"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["bounds", "bounds", "subset", "objective", "fft", "tighten", "load", "solve"])
    dtype = "f32" if op in ("subset", "fft") else rng.choice(["f32", "f32", "f64"])
    mix = rng.choice(list(MIXES))
    c = dict(op=op, dtype=dtype, mix=mix)
    if op == "solve":
        f64 = dtype == "f64"
        return dict(c, n=_log(rng, 500, 5_000 if f64 else 500_000), d=rng.randint(2, 3 if f64 else 4),
                    k=rng.randint(2, 3), nodes=_log(rng, 128, 512 if f64 else 2048))
    if op == "load":
        d = rng.choice([2, 3, 4, 5, 8, 12, 29])
        return dict(c, n=_log(rng, 2_000, 40_000_000 // d if dtype == "f32" else 20_000_000 // d), d=d,
                    k=rng.randint(2, 5), host=rng.random() < 0.5)
    if op == "tighten":
        d = rng.randint(2, 4) if dtype == "f64" else rng.choice([2, 3, 4, 5, 8, 12, 16, 29])
        k = rng.randint(2, 4 if dtype == "f64" else 6)
        b = _log(rng, 4, 256)
        terms = 6e7 if dtype == "f64" else 2e9   # node x sample x cluster x attribute
        n = _log(rng, 1_000, max(2_000, min(1_000_000, terms / (b * k * d))))
        cap = kcm.KC_BALLS_ALL if dtype == "f32" and d <= 4 and n <= 50_000 and b <= 32 and rng.random() < 0.25 else 0
        return dict(c, n=n, d=d, k=k, b=b, cap=cap)
    d = rng.choice([2, 3, 4, 5, 7, 8] if op in ("subset", "fft") else [2, 3, 4, 5, 8, 12, 16, 29, 68])
    k = rng.randint(2, 8)
    b = _log(rng, 1, 64 if op == "subset" else 256)
    terms = 4e9 if dtype == "f64" else 4e10
    n = _log(rng, 1_000, max(2_000, min(20_000_000, 2e8 / d, terms / (b * k * d))))
    c = dict(c, n=n, d=d, k=k, b=b)
    if op in ("bounds", "subset"):
        c["boxes"] = rng.choice(["nested", "frontier", "frontier"])
    if op == "subset":
        c["part"] = rng.choice([1, 2, 4, 16])
    return c


# ------------------------------------------------------------------- inputs

def _dtype(case):
    return torch.float32 if case["dtype"] == "f32" else torch.float64


def _samples(case, g):
    """(n, d) rows of a Gaussian mixture on the GPU."""
    weights, slo, shi, top, out = MIXES[case["mix"]]
    n, d = case["n"], case["d"]
    if weights is None:
        weights = (1.0 / case["k"],) * case["k"]
    m, dt = len(weights), _dtype(case)
    kw = dict(generator=g, device="cuda")
    means = torch.rand(m, d, **kw) * top
    sigma = slo + (shi - slo) * torch.rand(m, 1, **kw)
    edges = torch.tensor(weights, device="cuda").cumsum(0)[:-1].contiguous()
    X = torch.empty(n, d, dtype=dt, device="cuda")
    step = 1 << 24
    for s in range(0, n, step):
        e = min(n, s + step)
        lab = torch.bucketize(torch.rand(e - s, **kw), edges)
        X[s:e] = means[lab] + sigma[lab] * torch.randn(e - s, d, dtype=dt, **kw)
    n_out = int(round(out * n))
    if n_out:
        lo, hi = X.amin(0), X.amax(0)
        pos = torch.randint(0, n, (n_out,), **kw)
        X[pos] = lo + (hi - lo) * torch.rand(n_out, d, dtype=dt, **kw)
    return X


def _far_first(X, k):
    """k row indices: row 0, then the row farthest from those chosen (64 bits)."""
    Y = X[: 1 << 20].double()
    c = [0]
    near = (Y - Y[0]).square().sum(1)
    for _ in range(k - 1):
        c.append(int(near.argmax()))
        near = torch.minimum(near, (Y - Y[c[-1]]).square().sum(1))
    return c, float(near.max())


def _nested(case, X, g):
    k, b, d = case["k"], case["b"], case["d"]
    c = X[torch.randint(0, case["n"], (k,), generator=g, device="cuda")]
    u = torch.rand(b, k, d, generator=g, device="cuda", dtype=X.dtype)
    h = torch.exp(math.log(1e-3) + u * math.log(5.0 / 1e-3)).sort(0, descending=True).values
    return (c - h).cummax(0).values.contiguous(), (c + h).cummin(0).values.contiguous()


def _frontier(case, X, g):
    k, b, d = case["k"], case["b"], case["d"]
    kw = dict(generator=g, device="cuda", dtype=torch.float64)
    root, top = X.amin(0).double(), X.amax(0).double()
    span = top - root
    good = X[_far_first(X, k)[0]].double()
    pairs = (b + 1) // 2
    level = torch.randint(1, 6, (pairs, k, d), generator=g, device="cuda").double()
    at = good + 0.1 * span * torch.randn(pairs, k, d, **kw)
    cells = torch.exp2(level)
    cell = ((at - root) / span * cells).floor().clamp(min=0).minimum(cells - 1)
    lo = root + cell / cells * span
    hi = root + (cell + 1) / cells * span
    lo, hi = lo.reshape(pairs, -1), hi.reshape(pairs, -1)
    v = (hi - lo).argmax(1, keepdim=True)
    mid = 0.5 * (lo.gather(1, v) + hi.gather(1, v))
    lo = torch.stack([lo, lo.scatter(1, v, mid)], 1).reshape(2 * pairs, k, d)[:b]
    hi = torch.stack([hi.scatter(1, v, mid), hi], 1).reshape(2 * pairs, k, d)[:b]
    return lo.to(X.dtype).contiguous(), hi.to(X.dtype).contiguous()


def _around(case, X, g):
    k, b, d = case["k"], case["b"], case["d"]
    kw = dict(generator=g, device="cuda", dtype=torch.float64)
    root, top = X.amin(0).double(), X.amax(0).double()
    c, far = _far_first(X, k)
    width = (0.05 + 0.35 * torch.rand(b, k, d, **kw)) * (top - root)
    lo = (X[c].double() - (0.2 + 0.6 * torch.rand(b, k, d, **kw)) * width).clamp(min=root, max=top)
    hi = (lo + width).clamp(min=root, max=top)
    return lo.to(X.dtype).contiguous(), hi.to(X.dtype).contiguous(), 1.1 * far


def _inputs(case, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    X = _samples(case, g)
    s = dict(case=case, X=X)
    op, n, k = case["op"], case["n"], case["k"]
    if op in ("bounds", "subset"):
        s["lo"], s["hi"] = (_nested if case["boxes"] == "nested" else _frontier)(case, X, g)
    if op == "subset":
        keep = torch.rand(n, generator=g, device="cuda") < 1.0 / case["part"]
        keep[0] = True
        s["ids"] = keep.nonzero().reshape(-1).to(torch.int32)
    if op == "objective":
        # candidates of neighbouring nodes: samples near the farthest-first centers
        c = torch.tensor(_far_first(X, k)[0], device="cuda")
        pool = torch.randint(0, n, (4096,), generator=g, device="cuda")
        near = torch.cdist(X[c].double(), X[pool].double()).topk(64, largest=False).indices
        pick = torch.randint(0, 64, (case["b"], k), generator=g, device="cuda")
        s["sets"] = pool[near[torch.arange(k, device="cuda"), pick]].contiguous()
    if op == "fft":
        s["starts"] = torch.randint(0, n, (case["b"],), generator=g, device="cuda")
    if op == "tighten":
        s["lo"], s["hi"], s["alpha"] = _around(case, X, g)
    return s


def prepare(case, seed):
    s = _inputs(case, seed)
    if case["op"] == "load":
        if case["host"]:
            s["X"] = s["X"].cpu().pin_memory()
        s["like"] = torch.empty(0, device="cuda")
    else:
        s["kc"] = kcm.KCenter(s["X"], case["k"])
        del s["X"]
    torch.cuda.synchronize()
    return s


def run(s):
    case = s["case"]
    op = case["op"]
    if op == "bounds":
        return s["kc"].lower_bounds(s["lo"], s["hi"])
    if op == "subset":
        return s["kc"].lower_bounds_subset(s["ids"], s["lo"], s["hi"])
    if op == "objective":
        return s["kc"].upper_bound(s["sets"])
    if op == "fft":
        return s["kc"].fft_multi(s["starts"])
    if op == "tighten":
        return s["kc"].tighten(s["lo"], s["hi"], s["alpha"], ball_cap=case["cap"])
    if op == "load":
        kc = kcm.KCenter(s["X"], case["k"])
        lo, hi = kc.root_box(s["like"])
        centers, value = kc.fft(0, s["like"])
        kc.close()
        return dict(lo=lo, hi=hi, centers=centers, value=value)
    r = s["kc"].solve(tol=1e-12, node_limit=case["nodes"])
    return {q: r[q] for q in ("objective", "lower_bound", "gap", "fft_objective", "centers", "nodes", "batches",
                              "status")}


def work(case):
    """Samples (and ids or rows) read once, results written once; 4 operations
    per sample, node (or center set), cluster and attribute of the definition."""
    n, d, k, es = case["n"], case["d"], case["k"], 4 if case["dtype"] == "f32" else 8
    b = case.get("b", 1)
    op = case["op"]
    data = n * d * es
    boxes = 2 * b * k * d * es
    if op == "bounds":
        return dict(bytes=data + boxes + 24 * b, flops=4 * n * b * k * d)
    if op == "subset":
        m = n // case["part"]
        return dict(bytes=m * (4 + d * es) + boxes + 24 * b, flops=4 * m * b * k * d)
    if op == "objective":
        return dict(bytes=data + 8 * b * k + 16 * b, flops=3 * n * b * k * d)
    if op == "fft":
        return dict(bytes=data * k + 8 * b * (k + 2), flops=3 * n * b * k * d)
    if op == "tighten":
        return dict(bytes=data + 2 * boxes + b * (16 * k + 9), flops=4 * n * b * k * d)
    if op == "load":
        return dict(bytes=data * (2 + k), flops=3 * n * k * d)
    return dict(bytes=data * (k + 1), flops=4 * n * case["nodes"] * k * d // 8)


# ----------------------------------------------------------- 64-bit values

def _max_min(Y, lo, hi):
    """max over samples of min over clusters of the squared distance to the box
    [lo, hi] (b, k, d), for attribute-major 64-bit samples Y (d, n)."""
    b, k, d = lo.shape
    n = Y.shape[1]
    lo, hi = lo.double(), hi.double()
    best = torch.full((b,), -1.0, dtype=torch.float64, device=Y.device)
    ns = min(n, 1 << 22)
    bs = max(1, (1 << 24) // ns)
    for s in range(0, n, ns):
        y = Y[:, s:s + ns]
        for i in range(0, b, bs):
            near = None
            for j in range(k):
                acc = 0.0
                for a in range(d):
                    t = y[a] - torch.maximum(torch.minimum(y[a], hi[i:i + bs, j, a, None]), lo[i:i + bs, j, a, None])
                    acc = acc + t * t
                near = acc if near is None else torch.minimum(near, acc)
            best[i:i + bs] = torch.maximum(best[i:i + bs], near.amax(1))
    return best


def _far_first_from(Y, starts, k):
    """Farthest-first traversal over attribute-major 64-bit samples from every
    start -> objective of each set."""
    out = []
    for s in starts:
        last, near = int(s), None
        for j in range(k):
            acc = (Y - Y[:, last, None]).square().sum(0)
            near = acc if near is None else torch.minimum(near, acc)
            last = int(near.argmax())
        out.append(float(near[last]))
    return torch.tensor(out, dtype=torch.float64, device=Y.device)


def exact(case, seed):
    s = _inputs(case, seed)
    op, X = case["op"], s.pop("X")
    if op == "load":
        v = _far_first_from(X.t().double(), [0], case["k"])
        return dict(lo=X.amin(0).double(), hi=X.amax(0).double(), centers=None, value=v)
    if op == "subset":
        X = X[s["ids"].long()]
    Y = X.t().contiguous().double()
    if op in ("bounds", "subset"):
        v = _max_min(Y, s["lo"], s["hi"])
        return (v, v, None)
    if op == "objective":
        c = X[s["sets"]]
        return (_max_min(Y, c, c), None)
    if op == "fft":
        return (None, _far_first_from(Y, s["starts"], case["k"]))
    if op == "tighten":
        # the tightened boxes, counts and candidates follow from decisions, not from a formula
        return dict(lo=None, hi=None, count=None, cand=None, lb=_max_min(Y, s["lo"], s["hi"]), status=None)
    # an incumbent at a node limit has no value of its own; the heuristic start has
    return dict(objective=None, lower_bound=None, gap=None, centers=None, nodes=None, batches=None, status=None,
                fft_objective=float(_far_first_from(Y, [0], case["k"])[0]))
