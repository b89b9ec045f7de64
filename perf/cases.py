"""The work that is timed: what programs have the framework do, through its
public entry points (``Graph.prepare`` / ``fetch_all`` / ``sage_mean_layer``).

Three kinds of pass:

  "sample"  one hyperbatch sampled and its features gathered: prepare, then
            fetch_all (every array of the view is an output);
  "layer"   one GraphSAGE-mean layer over a hop that is already prepared;
  "step"    a model's forward pass: prepare, then one layer per hop.

Graphs are RMAT graphs with the skew of the repository's workloads, made on
the GPU from the seed, with N(0,1) features; targets are distinct random
nodes.  A state holds a graph of its own, loaded, and a ctx that has already
prepared a hyperbatch of the same shape with other targets, as in a loader's
steady state.  The views' arrays are as long as the shape's capacity; what a
hyperbatch does not reach of them is zero here (cleared before the passes).
"""
import functools
import math

import torch

from paper_2601_01473_gb300 import Graph

KB, MB = 1024, 1024 * 1024
M32 = 0xFFFFFFFF
DTYPES = {"f16": torch.float16, "f32": torch.float32}
SKEW = {"rmat": (0.57, 0.19, 0.19), "social": (0.6, 0.2, 0.15)}


def _case(name=None, **kw):
    c = {
        "kind": "sample", "nodes": 10_000_000, "degree": 20, "skew": "rmat", "offsets": 64,
        "dtype": "f16", "dim": 128, "block": MB, "H": 1, "B": 1024, "fanouts": "15,10,5",
        "frontier": "src",      # or "sampled": Algorithm 1's literal frontier update
        "features": "hbm",      # or "host": pinned host memory, read by rows through a cache
        "out": "f32", "width": 128,  # the layers' output type and width
    }
    c.update(kw)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # an online request: a few nodes' neighbourhoods on a small graph; latency only
        _case("request_1x16", nodes=100_000, degree=16, offsets=32, dtype="f32", block=64 * KB,
              H=1, B=16, fanouts="10,5"),
        # the small training configuration: a graph that fits the L2 cache
        _case("train_small_8x1024", nodes=100_000, degree=16, offsets=32, dtype="f32",
              block=64 * KB, H=8, B=1024, fanouts="10,5"),
        # one minibatch per call, three hops: a trainer that does not batch its minibatches
        _case("one_minibatch_1x1024", dtype="f32", H=1),
        # hyperbatches of a mid-sized graph, fp32 features, three hops
        _case("train_mid_16x1024", dtype="f32", H=16),
        # a skewed social graph: hubs, wide rows, a large first fanout
        _case("social_32x1024", nodes=8_000_000, degree=28, skew="social", dim=256, H=32,
              fanouts="25,10"),
        # the paper's minibatch of 1000, a ragged H, feature rows of 400 bytes (not a power of two)
        _case("width100_13x1000", nodes=2_500_000, degree=25, dtype="f32", dim=100, H=13, B=1000,
              fanouts="10,10"),
        # feature rows of 1204 bytes: not a multiple of 16
        _case("width602_8x500", nodes=250_000, degree=40, offsets=32, dim=602, H=8, B=500,
              fanouts="25,10"),
        # Algorithm 1's literal frontier update
        _case("sampled_frontier_16x1024", H=16, frontier="sampled"),
        # evaluation with wide fanouts (past a warp's lanes)
        _case("evaluate_wide_8x256", nodes=2_000_000, degree=28, skew="social", H=8, B=256,
              fanouts="100,20"),
        # features that stay in pinned host memory, read over the host link
        _case("host_features_16x1024", nodes=2_000_000, degree=16, H=16, fanouts="10,5",
              features="host"),
        # layer-wise inference: one layer over all rows of a large one-hop batch
        _case("layer_24x8192", kind="layer", H=24, B=8192, fanouts="15", out="f16"),
        # a training-scale forward pass: a large graph, 128 minibatches of 1024, three layers
        _case("model_128x1024", kind="step", nodes=40_000_000, degree=16, H=128, out="f32",
              width=128),
    ]


def draw(rng):
    def logint(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    while True:
        kind = rng.choice(["sample", "sample", "sample", "layer", "step"])
        c = _case(kind=kind, nodes=logint(50_000, 10_000_000), degree=rng.randint(6, 30),
                  skew=rng.choice(["rmat", "social"]), offsets=rng.choice([32, 64]),
                  dtype=rng.choice(["f16", "f32"]), block=rng.choice([64, 256, 1024]) * KB,
                  H=logint(1, 128), B=logint(16, 2048))
        if kind == "sample":
            hops = rng.randint(1, 3)
            c["fanouts"] = ",".join(str(rng.randint(2, 25)) for _ in range(hops))
            c["dim"] = rng.choice([16, 50, 64, 100, 128, 128, 200, 256, 301])
            option = rng.choice(["", "", "", "sampled", "host", "wide"])
            if option == "sampled":
                c["frontier"] = "sampled"
            elif option == "host":
                c.update(features="host", dtype="f16", dim=rng.choice([64, 128, 200, 256]),
                         nodes=min(c["nodes"], 2_000_000))
            elif option == "wide":
                c["fanouts"] = "%d,%d" % (rng.randint(33, 150), rng.randint(2, 20))
        elif kind == "layer":
            # layer-wise inference: one hop, many targets, every row an output
            c["fanouts"] = str(rng.randint(3, 30))
            c["B"] = logint(256, 16384)
            c["dim"] = 8 * rng.randint(2, 16)
            c["width"] = 32 * rng.randint(1, 6)
            c["out"] = rng.choice(["f16", "f32"])
        else:
            c["fanouts"] = ",".join(str(rng.randint(3, 15)) for _ in range(rng.randint(2, 3)))
            c["dim"] = 8 * rng.randint(4, 16)
            c["width"] = 32 * rng.randint(1, 4)
        cap = _caps(c)
        if (c["H"] * c["B"] <= c["nodes"] and c["H"] * cap[-1] * c["dim"] <= 1 << 31
                and c["H"] * cap[-1] <= 1 << 25):
            return c


def _fanouts(c):
    return [int(k) for k in c["fanouts"].split(",")]


def _caps(c):
    cap = [c["B"]]
    for k in _fanouts(c):
        cap.append(min(c["nodes"], cap[-1] * (1 + k)))
    return cap


# ---- inputs ------------------------------------------------------------------


def _generator(seed, salt):
    g = torch.Generator(device="cuda")
    g.manual_seed(1_000_003 * (int(seed) + 1) + salt)
    return g


def _topology(c, seed):
    """CSR (offsets, indices) of an RMAT graph: each edge picks a quadrant of
    the adjacency matrix per level; duplicate edges are dropped."""
    N, E = c["nodes"], c["nodes"] * c["degree"]
    a, b, cc = SKEW[c["skew"]]
    scale = max(1, math.ceil(math.log2(N)))
    gen = _generator(seed, 1)
    keys = torch.empty(E, dtype=torch.int64, device="cuda")
    for first in range(0, E, 1 << 27):
        n = min(E - first, 1 << 27)
        src = torch.zeros(n, dtype=torch.int32, device="cuda")
        dst = torch.zeros(n, dtype=torch.int32, device="cuda")
        for _ in range(scale):
            u = torch.rand(n, device="cuda", generator=gen)
            src.mul_(2).add_(u >= a + b)
            dst.mul_(2).add_(((u >= a) & (u < a + b)) | (u >= a + b + cc))
        keys[first:first + n] = ((src.long() * N) >> scale) * N + ((dst.long() * N) >> scale)
        del src, dst, u
    keys = torch.unique(keys, sorted=True)
    rows = torch.arange(N + 1, dtype=torch.int64, device="cuda") * N
    offsets = torch.searchsorted(keys, rows)
    del rows
    indices = (keys % N).to(torch.int32)
    del keys
    return offsets.to(torch.int32 if c["offsets"] == 32 else torch.int64), indices


def _features(c, seed):
    return torch.randn(c["nodes"], c["dim"], dtype=DTYPES[c["dtype"]], device="cuda",
                       generator=_generator(seed, 2))


def _targets(c, seed, salt=3):
    ids = torch.randperm(c["nodes"], device="cuda", generator=_generator(seed, salt))
    return ids[:c["H"] * c["B"]].to(torch.int32).view(c["H"], c["B"])


def _layers(c, seed):
    """(weight, bias, output type) of each hop's layer, hop 0 (the targets') first."""
    K = len(_fanouts(c))
    gen = _generator(seed, 4)
    layers = []
    for hop in range(K):
        d_in = c["dim"] if hop == K - 1 else c["width"]
        w = torch.randn(c["width"], 2 * d_in, device="cuda", generator=gen) / (2 * d_in) ** 0.5
        bias = 0.1 * torch.randn(c["width"], device="cuda", generator=gen)
        layers.append((w.to(torch.float16), bias, DTYPES[c["out"] if hop == 0 else "f16"]))
    return layers


def prepare(case, seed):
    c = case
    offsets, indices = _topology(c, seed)
    features = _features(c, seed)
    torch.cuda.empty_cache()  # the library allocates beside torch's pool
    options = {}
    if c["features"] == "host":
        host = torch.empty(features.shape, dtype=features.dtype, pin_memory=True)
        host.copy_(features)
        features = host
        options = {"features_on_host": True, "feature_io": "rows",
                   "feature_cache_bytes": host.numel() * host.element_size() // 4}
    g = Graph(offsets, indices, features, adj_block_bytes=c["block"],
              feat_block_bytes=c["block"], **options)
    if c["frontier"] != "src":
        g.set_frontier(c["frontier"])
    state = {"kind": c["kind"], "graph": g, "fanouts": _fanouts(c), "seed": int(seed),
             "targets": _targets(c, seed)}
    # the loader has been running: an earlier hyperbatch, with other targets
    g.prepare(_targets(c, seed, 5), state["fanouts"], state["seed"] + 1, 10_000)
    view = g.fetch_all()
    for t in [view.nodes, view.feats, *view.indptr, *view.col]:
        t.zero_()
    if c["kind"] != "sample":
        state["layers"] = _layers(c, seed)
    if c["kind"] == "layer":
        g.prepare(state["targets"], state["fanouts"], state["seed"])
        state["x"] = g.fetch_all().feats
    return state


class View(dict):
    """A hyperbatch's arrays; they lie in memory that their graph owns, so
    the graph is kept with them."""

    graph = None


def run(state):
    g = state["graph"]
    if state["kind"] == "layer":
        w, bias, out = state["layers"][0]
        return {"rows": g.sage_mean_layer(0, state["x"], w, bias, out_dtype=out)}
    g.prepare(state["targets"], state["fanouts"], state["seed"])
    view = g.fetch_all()
    sizes = {"node_size": view.node_size, "edges": view.edges, "src_size": view.src_size}
    if state["kind"] == "sample":
        out = View(indptr=view.indptr, col=view.col, nodes=view.nodes, feats=view.feats, **sizes)
        out.graph = g
        return out
    x = view.feats
    for hop in reversed(range(len(state["fanouts"]))):
        w, bias, out = state["layers"][hop]
        x = g.sage_mean_layer(hop, x, w, bias, out_dtype=out)
    return {"logits": x, **sizes}


# ---- the same in plain torch ---------------------------------------------------


def _philox(c0, c1, c2, c3, k0, k1):
    """The first two words of Philox4x32-10 (Salmon et al., SC'11); every
    argument holds 32-bit values in int64."""
    for r in range(10):
        if r:
            k0, k1 = (k0 + 0x9E3779B9) & M32, (k1 + 0xBB67AE85) & M32
        p, q = c0 * 0xD2511F53, c2 * 0xCD9E8D57  # wraps: the low 64 bits are right
        c0, c1, c2, c3 = (((q >> 32) & M32) ^ c1 ^ k0, q & M32, ((p >> 32) & M32) ^ c3 ^ k1,
                          p & M32)
    return c0, c1


def _hops(c, offsets, indices, targets, seed):
    """Per hop: (number of dst rows, src node ids, edges' dst rows, edges'
    src rows), the rows of all minibatches in one list, dst first."""
    N, H = c["nodes"], c["H"]
    offsets = offsets.long()
    mb = torch.arange(H, device="cuda").repeat_interleave(c["B"])
    ids = targets.reshape(-1).long()
    hops = []
    for hop, k in enumerate(_fanouts(c)):
        n = ids.numel()
        first = offsets[ids]
        deg = offsets[ids + 1] - first
        src_rows, dst_rows, chosen = [], [], []
        for s in range(k):
            # Floyd: slot s draws t in [0, J], J = deg - k + s, and takes J if t is taken
            J = (deg - k + s).clamp_(min=0)
            x0, x1 = _philox(ids, ((hop + 1) << 24) | s, mb, 0, seed & M32, seed >> 32)
            t = (x1 * (J + 1) + ((x0 * (J + 1)) >> 32)) >> 32
            taken = torch.zeros(n, dtype=torch.bool, device="cuda")
            for earlier in chosen:
                taken |= earlier == t
            t = torch.where(taken, J, t)
            chosen.append(t)
            has = deg > s
            at = first + torch.where(deg <= k, s, t)
            rows = torch.nonzero(has).flatten()
            src_rows.append(mb[rows] * N + indices[at[rows]].long())
            dst_rows.append(rows)
        del chosen
        keys, dst = torch.cat(src_rows), torch.cat(dst_rows)
        del src_rows, dst_rows
        mine = mb * N + ids
        union = torch.unique(keys)
        ordered, order = torch.sort(mine)
        at = torch.searchsorted(ordered, union).clamp_(max=n - 1)
        new = union[ordered[at] != union]
        src_keys = torch.cat([mine, new])
        ordered, order = torch.sort(src_keys)
        src = order[torch.searchsorted(ordered, keys)]
        hops.append((n, src_keys % N, dst, src))
        after = src_keys if c["frontier"] == "src" else union
        mb, ids = after // N, after % N
    return hops


def _layer64(x, hop, w, bias):
    n, _, dst, src = hop
    total = torch.zeros(n, x.shape[1], dtype=torch.float64, device="cuda")
    for e in range(0, dst.numel(), 1 << 22):
        total.index_add_(0, dst[e:e + (1 << 22)], x[src[e:e + (1 << 22)]].double())
    deg = torch.bincount(dst, minlength=n).clamp_(min=1)
    total /= deg[:, None]
    out = torch.empty(n, w.shape[0], dtype=torch.float64, device="cuda")
    for r in range(0, n, 1 << 20):
        a = torch.cat([x[r:r + (1 << 20)][:n - r].double(), total[r:r + (1 << 20)]], 1)
        out[r:r + (1 << 20)] = torch.relu(a @ w.double().T + bias.double())
    return out


def exact(case, seed):
    c = case
    if c["kind"] == "sample":
        return None  # ids, positions and copied bytes: nothing is computed
    offsets, indices = _topology(c, seed)
    hops = _hops(c, offsets, indices, _targets(c, seed), int(seed))
    del offsets, indices
    features = _features(c, seed)
    x = features[hops[-1][1]]
    del features
    layers = _layers(c, seed)
    for hop in reversed(range(len(hops))):
        x = _layer64(x, hops[hop], layers[hop][0], layers[hop][1])
    out = x.view(c["H"], c["B"], -1)
    if c["kind"] == "layer":
        return {"rows": out}
    return {"logits": out, "node_size": None, "edges": None, "src_size": None}


@functools.lru_cache(maxsize=None)
def _counts(items):
    """Per hop (dst rows, src rows, edges) and the distinct gathered ids of
    one hyperbatch, counted on a graph of this shape."""
    c = dict(items)
    offsets, indices = _topology(c, 0)
    hops = _hops(c, offsets, indices, _targets(c, 0), 0)
    return ([(n, ids.numel(), dst.numel()) for n, ids, dst, _ in hops],
            torch.unique(hops[-1][1]).numel())


def work(case):
    """Bytes: per frontier node two offsets read and an indptr entry written,
    per sampled edge a neighbour id read and a col entry written, per new node
    its id; each distinct feature row read and each gathered row written.  A
    layer reads its src rows, indptr, col and weights and writes its dst rows."""
    c = case
    hops, distinct = _counts(tuple(sorted((k, v) for k, v in c.items() if k != "name")))
    row = c["dim"] * DTYPES[c["dtype"]].itemsize
    bytes_ = flops = 0
    if c["kind"] != "layer":
        for n, n_src, edges in hops:
            bytes_ += n * (2 * c["offsets"] // 8 + 8) + edges * 8 + (n_src - n) * 4
        bytes_ += hops[-1][1] * row + distinct * row
    if c["kind"] != "sample":
        for hop, (n, n_src, edges) in enumerate(hops):
            outer = hop == len(hops) - 1
            d_in = c["dim"] if outer else c["width"]
            x_row = row if outer else 2 * d_in
            out_row = c["width"] * (DTYPES[c["out"]].itemsize if hop == 0 else 2)
            bytes_ += n_src * x_row + n * (8 + out_row) + edges * 4 + 4 * d_in * c["width"]
            flops += 4 * n * d_in * c["width"] + edges * d_in
    return {"bytes": bytes_, "flops": flops}


def tolerance(case):
    """Sampling and gathering are integers and copied bytes.  The layers round
    their inputs, and in half precision their outputs, to fp16 and accumulate
    in fp32: measured against exact, 5e-5 .. 2.1e-4 for one layer and 2.7e-4
    for a model, whose layers pass their rounding on; four times that."""
    if case["kind"] == "sample":
        return "exact"
    return {"rel": 8e-4 if case["kind"] == "layer" else 1.1e-3}
