"""What a user of this library has it do, as cases that can be timed and compared.

Every case is one call sequence through the public binding on a seeded synthetic graph: a whole model over every vertex
(`it_infer`), the set-up of a graph (`it_graph_create` + `it_split_hubs`), or what one worker of a vertex-partitioned
pass runs between two exchanges (`it_layer_gather`, `it_aggregate_finish`, `it_layer_update`).  Sizes run from a graph
that fits the L2 cache, where a pass is a latency, to the largest whose state fits a third of the device.

A case is a dict of plain values:
  kind     "infer" | "build" | "worker"
  op       the Gather stage of every layer (mean, sum, max, min, gcn, gat)
  dtype    storage type of features, weights and layer outputs ("f32" | "bf16")
  n, e     vertices and directed edges
  shape    in-degrees: "power" (shifted power law, exponent `gamma`, at most `cap` edges), "hubs" (`hubs` vertices with `cap`
           edges each, the rest uniform) or "even" (uniform destinations)
  dims     widths of the layers, "64-128-64"
  weighted edge weights U(0, 1);  heads: attention heads;  edge_dim: edge features;  msg_dim: learned messages
  split    hub-split threshold
"""
import math

import torch

from paper_2307_00228_b200 import binding as B

DEFAULTS = dict(kind="infer", op="mean", dtype="bf16", n=10_000, e=100_000, shape="power", gamma=2.1, cap=2_000, hubs=0, dims="64-64",
                weighted=False, heads=1, edge_dim=0, msg_dim=0, split=4096)


def _case(**kw):
    return {**DEFAULTS, **kw}


def listed():
    return [
        # The smallest call: a graph that lives in the L2 cache, re-scored on request.  A latency: launches and host work.
        _case(name="small_mean_f32", op="mean", dtype="f32", n=10_000, e=100_000, cap=2_000, dims="64-64-16", split=256),
        # The same kind of request on an attention model.
        _case(name="small_gat_bf16", op="gat", dtype="bf16", n=30_000, e=420_000, gamma=2.0, cap=4_000, heads=4, dims="64-64-64", split=1024),
        # A three-layer GCN on raw features of 100 columns (rows that are no power of two), normalisation in the edge weights.
        _case(name="gcn_f32_odd", op="gcn", dtype="f32", n=610_001, e=15_000_003, cap=20_000, weighted=True, dims="100-128-128-48", split=1024),
        # An ordinary fp32 model with edge weights: 2M vertices, hubs of up to 200k edges.
        _case(name="medium_sum_f32", op="sum", dtype="f32", n=2_000_000, e=40_000_000, cap=200_000, weighted=True, dims="128-128-64", split=1024),
        # An ordinary attention model: two layers of four heads of 32.
        _case(name="gat_bf16", op="gat", dtype="bf16", n=5_000_000, e=100_000_000, gamma=2.0, cap=200_000, heads=4, dims="128-128-128", split=4096),
        # Max pooling on a graph whose edges crowd on a hundred hubs, three layers.
        _case(name="hubs_max_bf16", op="max", dtype="bf16", n=20_000_000, e=200_000_000, shape="hubs", hubs=100, cap=1_000_000, dims="64-64-64-32", split=4096),
        # The largest: a quarter of 100M vertices / 1.5B edges, so that three states fit the device.
        _case(name="large_mean_bf16", op="mean", dtype="bf16", n=25_000_000, e=375_000_000, cap=50_000, dims="64-128-64", split=4096),
        # Wide input features (768 columns, as text embeddings have), reduced by the first layer.
        _case(name="wide_mean_bf16", op="mean", dtype="bf16", n=1_000_000, e=16_000_000, cap=50_000, dims="768-256-64", split=4096),
        # Learned messages on edge features: the general message function of the model family.
        _case(name="messages_bf16", op="mean", dtype="bf16", n=1_000_000, e=16_000_000, cap=50_000, dims="64-64", edge_dim=32, msg_dim=64, split=4096),
        # Attention whose logits read edge features, fp32.
        _case(name="gat_edges_f32", op="gat", dtype="f32", n=500_000, e=8_000_000, cap=50_000, heads=4, dims="64-64", edge_dim=16, split=4096),
        # Set-up of a graph: validation, hub split, degree buckets.
        _case(name="build", kind="build", n=5_000_000, e=100_000_000, gamma=2.0, cap=200_000, split=4096),
        # One of four workers of a source-partitioned layer: raw partial sums for every destination, then its own vertices finished.
        _case(name="worker_sum_bf16", kind="worker", op="sum", dtype="bf16", n=8_000_000, e=30_000_000, cap=50_000, dims="64-64", split=4096),
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """A case of the same ranges: every kind of layer, both types, sizes over their logarithm, widths odd and even."""
    family = rng.choice(["pool", "pool", "pool", "gcn", "gat", "gat", "wide", "messages", "gat_edges", "build", "worker"])
    dtype = rng.choice(["f32", "bf16", "bf16"])
    n = _log_uniform(rng, 8_000, 12_000_000)
    if family in ("wide", "messages", "gat_edges"):
        n = _log_uniform(rng, 8_000, 1_000_000)
    e = int(n * math.exp(rng.uniform(math.log(4), math.log(24)))) + rng.randrange(7)
    shape = rng.choice(["power", "power", "power", "hubs", "even"])
    hubs = rng.randint(1, 100) if shape == "hubs" else 0
    cap = max(64, min(n // 10, 200_000))
    if shape == "hubs":
        cap = max(1, min(cap, e // (3 * hubs)))
    c = dict(dtype=dtype, n=n, e=e, shape=shape, hubs=hubs, cap=cap, gamma=rng.choice([1.9, 2.0, 2.1, 2.4]), split=rng.choice([256, 1024, 4096, 4096, 0]),
             weighted=rng.random() < 0.3)
    step = 4 if dtype == "f32" else 8
    width = lambda: rng.choice([16, 32, 48, 64, 64, 96, 128, 128, step * rng.randint(4, 32)])  # noqa: E731
    if family == "pool":
        c.update(op=rng.choice(["mean", "mean", "sum", "max", "min"]), dims="-".join(str(width()) for _ in range(rng.choice([2, 3, 3, 4]))))
    elif family == "gcn":
        c.update(op="gcn", weighted=True, dims="-".join(str(width()) for _ in range(rng.choice([3, 4]))))
    elif family == "gat":
        heads = rng.choice([2, 4, 4])
        per = rng.choice([16, 32])
        c.update(op="gat", weighted=False, heads=heads, dims="-".join([str(rng.choice([64, 100 if dtype == "f32" else 104, 128]))] + [str(heads * per)] * rng.choice([1, 2])))
    elif family == "wide":
        c.update(op=rng.choice(["mean", "sum", "max"]), dims=rng.choice(["768-256-64", "768-128", "512-128-64", "600-128-40"]))
    elif family == "messages":
        c.update(op=rng.choice(["mean", "sum", "max"]), dims=rng.choice(["64-64", "64-128", "32-64"]), msg_dim=rng.choice([0, 32, 64, 64, 128]), edge_dim=rng.choice([0, 16, 32, 32, 40]))
    elif family == "gat_edges":
        c.update(op="gat", weighted=False, heads=4, dims=rng.choice(["64-64", "128-128", "64-128"]), edge_dim=rng.choice([8, 16, 32]))
    elif family == "build":
        c.update(kind="build", weighted=False, dims="64-64")
    else:
        c.update(kind="worker", op=rng.choice(["sum", "mean", "max"]), dims="-".join(str(width()) for _ in range(2)))
    c = _case(**c)
    while _moved(c) > 0.8 * max(_moved(k) for k in listed()):   # never more than the largest listed case
        for k in ("n", "e", "cap"):
            c[k] = max(1, c[k] // 2)
    return c


def _moved(case):
    """Bytes a pass reads row by row: what its cost goes by."""
    dims, size = _dims(case), 4 if case["dtype"] == "f32" else 2
    rows = sum(case["e"] * size * max(fi if case["op"] in ("max", "min") else min(fi, fo), case["msg_dim"]) for fi, fo in zip(dims[:-1], dims[1:]))
    return rows + work(case)["bytes"]


# ----------------------------------------------------------------------------- inputs

def _dims(case):
    return [int(d) for d in case["dims"].split("-")]


def _power_law_degrees(g, n, e, gamma, cap):
    """n in-degrees from P(k) ~ (k + q)^-gamma on [0, cap], q such that the mean is e / n; nudged to sum to e."""
    k = torch.arange(cap + 1, dtype=torch.float64, device="cuda")
    lo, hi = 1e-6, 1e6
    for _ in range(60):
        mid = math.sqrt(lo * hi)
        p = (k + mid) ** -gamma
        if float((p * k).sum() / p.sum()) < e / n:
            lo = mid
        else:
            hi = mid
    p = (k + math.sqrt(lo * hi)) ** -gamma
    cdf = torch.cumsum(p / p.sum(), 0)
    u = torch.rand(n, generator=g, device="cuda", dtype=torch.float64)
    deg = torch.searchsorted(cdf, u).clamp_(max=cap)
    diff = e - int(deg.sum())
    if diff > 0:      # spread the missing edges evenly
        deg += diff // n
        deg[: diff % n] += 1
    elif diff < 0:    # take the surplus from vertices that have edges
        while diff < 0:
            some = torch.nonzero(deg > 0).flatten()[:-diff]
            deg[some] -= 1
            diff += some.numel()
    return deg


def _degrees(g, case):
    n, e = case["n"], case["e"]
    if case["shape"] == "power":
        return _power_law_degrees(g, n, e, case["gamma"], case["cap"])
    hubs, cap = (case["hubs"], case["cap"]) if case["shape"] == "hubs" else (0, 0)
    deg = torch.zeros(n, dtype=torch.int64, device="cuda")
    rest = e - hubs * cap
    for c0 in range(0, rest, 1 << 26):
        deg += torch.bincount(torch.randint(0, n, (min(1 << 26, rest - c0),), generator=g, device="cuda"), minlength=n)
    if hubs:
        deg[torch.randperm(n, generator=g, device="cuda")[:hubs]] += cap
    return deg


def _graph(g, case, n_sources):
    """CSR by destination: int32 indptr, source ids ascending inside every destination, as a sorted edge list gives them."""
    # One degree sequence for a case, dealt to other vertices with each seed: how many rows a hub split makes then depends on the case alone.
    fixed = torch.Generator(device="cuda")
    fixed.manual_seed(1)
    deg = _degrees(fixed, case)[torch.randperm(case["n"], generator=g, device="cuda")]
    indptr = torch.zeros(case["n"] + 1, dtype=torch.int64, device="cuda")
    torch.cumsum(deg, 0, out=indptr[1:])
    indices = torch.empty(case["e"], dtype=torch.int32, device="cuda")
    v0 = 0
    while v0 < case["n"]:   # whole destinations, about 2^26 edges at a time
        e0 = int(indptr[v0])
        v1 = max(v0 + 1, int(torch.searchsorted(indptr, e0 + (1 << 26), right=True)) - 1)
        e1 = int(indptr[v1])
        if e1 > e0:
            dst = torch.repeat_interleave(torch.arange(v1 - v0, device="cuda"), deg[v0:v1])
            key = (dst << 32) | torch.randint(0, n_sources, (e1 - e0,), generator=g, device="cuda")
            indices[e0:e1] = torch.sort(key).values & 0xFFFFFFFF
        v0 = v1
    return indptr.to(torch.int32), indices


def _layers(g, case):
    dt = torch.float32 if case["dtype"] == "f32" else torch.bfloat16
    dims, op, de, dm, heads = _dims(case), case["op"], case["edge_dim"], case["msg_dim"], case["heads"]

    def glorot(rows, cols, dtype=dt):
        lim = math.sqrt(6.0 / (rows + cols))
        return ((torch.rand(rows, cols, generator=g, device="cuda") * 2 - 1) * lim).to(dtype)

    out = []
    for i in range(len(dims) - 1):
        fi, fo = dims[i], dims[i + 1]
        last = i == len(dims) - 2
        kw = dict(op=op, act="none" if last else ("elu" if op == "gat" else "relu"), in_dim=fi, out_dim=fo,
                  bias=torch.rand(fo, generator=g, device="cuda") * 0.2 - 0.1, use_edge_weights=bool(case["weighted"]), edge_dim=de, msg_dim=dm,
                  allow_reorder=case["kind"] != "worker")
        if op == "gat":
            hd = fo // heads
            att = lambda k: glorot(k, heads, torch.float32).t().contiguous()  # noqa: E731
            kw.update(W=glorot(fi, fo), heads=heads, att_src=att(hd), att_dst=att(hd), att_edge=att(de) if de else None)
        elif dm:
            kw.update(W=glorot(fi + dm if op != "gcn" else dm, fo), W_edge=glorot(fi + de, dm), act_edge="relu",
                      bias_edge=torch.rand(dm, generator=g, device="cuda") * 0.2 - 0.1)
        else:
            kw.update(W=glorot((fi if op != "gcn" else 0) + fi + de, fo))
        out.append(B.LayerDesc(**kw))
    return out


def prepare(case, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    n, e, dims = case["n"], case["e"], _dims(case)
    dt = torch.float32 if case["dtype"] == "f32" else torch.bfloat16
    workers = 4 if case["kind"] == "worker" else 1
    n_sources = -(-n // workers)
    indptr, indices = _graph(g, case, n_sources)
    s = dict(kind=case["kind"], split=case["split"], indptr=indptr, indices=indices)
    if case["kind"] == "build":
        return s
    weights = torch.rand(e, generator=g, device="cuda") if case["weighted"] else None
    s["layers"] = _layers(g, case)
    s["x"] = torch.randn(n_sources, dims[0], generator=g, device="cuda", dtype=dt)
    s["out"] = torch.empty(n_sources, dims[-1], device="cuda", dtype=dt)
    if case["kind"] == "worker":
        s["part"] = B.it_graph_create_part(indptr, indices, n_sources, weights)   # every destination, the worker's own sources
        B.it_split_hubs(s["part"], case["split"])
        own = torch.zeros(n_sources + 1, dtype=torch.int32, device="cuda")        # the worker's own vertices (their update reads no edges)
        s["own"] = B.it_graph_create_part(own, torch.empty(0, dtype=torch.int32, device="cuda"), n_sources)
        if weights is not None:
            s["layers"][0].use_edge_weights = True
        s["raw"] = torch.empty(n, dims[0], device="cuda")
        s["agg"] = torch.empty(n_sources, dims[0], device="cuda", dtype=dt)
        deg = (indptr[1:] - indptr[:-1])[:n_sources].float()
        s["scale"] = torch.where(deg > 0, 1.0 / deg.clamp(min=1) if case["op"] == "mean" else torch.ones_like(deg), torch.zeros_like(deg))
        update = {**vars(s["layers"][0]), "use_edge_weights": False}
        s["update"] = B.LayerDesc(**update)
        s["ws"] = torch.empty(B.it_workspace_bytes(s["part"], s["layers"]), dtype=torch.uint8, device="cuda")
        return s
    s["graph"] = B.it_graph_create(indptr, indices, weights)
    if case["edge_dim"]:
        s["edge_feat"] = torch.randn(e, case["edge_dim"], generator=g, device="cuda", dtype=dt)
        B.it_graph_set_edge_features(s["graph"], s["edge_feat"])
    B.it_split_hubs(s["graph"], case["split"])
    s["ws"] = torch.empty(B.it_workspace_bytes(s["graph"], s["layers"]), dtype=torch.uint8, device="cuda")
    return s


def run(s):
    if s["kind"] == "build":
        g = B.it_graph_create(s["indptr"], s["indices"])
        B.it_split_hubs(g, s["split"])
        return B.it_graph_get_split(g)
    if s["kind"] == "worker":
        layer, per = s["layers"][0], s["x"].shape[0]
        B.it_layer_gather(s["part"], layer, s["x"], None, 0, True, s["raw"], s["ws"])
        B.it_aggregate_finish(s["raw"][:per], s["scale"], s["agg"])   # the block a reduce-scatter would hand this worker
        B.it_layer_update(s["own"], s["update"], s["x"], s["agg"], s["out"], s["ws"])
        return {"raw": s["raw"], "out": s["out"]}
    return B.it_infer(s["graph"], s["layers"], s["x"], s["out"], s["ws"])


# ----------------------------------------------------------------------------- what a pass cannot do without

def work(case):
    """Per layer: the edge arrays, the layer input and the layer output, each once; the products and the reduce."""
    n, e, dims = case["n"], case["e"], _dims(case)
    s = 4 if case["dtype"] == "f32" else 2
    if case["kind"] == "build":   # CSR in; row bounds, owners, bucket lists out
        return {"bytes": 4.0 * (n + 1) + 4.0 * e + n * (8.0 + 4.0 + 8.0 + 4.0), "flops": 0.0}
    if case["kind"] == "worker":
        own = -(-n // 4)
        return {"bytes": e * (8.0 if case["weighted"] else 4.0) + n * (4.0 + 4.0 * dims[0]) + own * s * (dims[0] + dims[1]),
                "flops": float(e) * dims[0] + 4.0 * own * dims[0] * dims[1]}
    total, flops = 0.0, 0.0
    for fi, fo in zip(dims[:-1], dims[1:]):
        fm = case["msg_dim"] or fi
        total += e * (4.0 + (4.0 if case["weighted"] else 0.0) + s * case["edge_dim"]) + 4.0 * n + n * s * (fi + fo)
        if case["op"] == "gat":
            flops += 2.0 * n * fi * fo + 2.0 * e * (fo + case["heads"] * case["edge_dim"])
        else:
            self_term = 0 if case["op"] == "gcn" else fi
            flops += 2.0 * n * (self_term + fm) * fo + e * float(min(fm, fo) if case["op"] in ("mean", "sum", "gcn") and not case["msg_dim"] else fm)
            if case["msg_dim"]:
                flops += 2.0 * n * fi * fm + 2.0 * e * case["edge_dim"] * fm
    return {"bytes": total, "flops": flops}


def tolerance(case):
    if case["kind"] == "build":
        return "exact"
    # Seen: f32 against float64 up to 4e-6 (largest single entry 3e-5 of the rms), bf16 against float64 and against the other order of
    # transform and aggregate up to 4e-3 (largest entry 0.07, once 0.24 on sums over hubs).
    return {"rel": 1e-2, "max": 0.3} if case["dtype"] == "bf16" else {"rel": 1.5e-5, "max": 1.3e-4}
