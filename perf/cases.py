"""The work a user of this framework has it do, as cases that can be timed and compared.

Shapes follow the five named workloads of the benchmark (`tiny`, `seqpart`, `medium`, `dense`, `large`) and the layers
and tools around the aggregation: a whole attention layer with its normalisation, a GraphSage layer, the sum aggregation,
the propagation that post-processes predictions, and graph preparation.  Every case goes through `api`, as a training or
inference program does, and every kind is measured in each direction it has.

A case is a dict of plain values:

  kind   attention | sum | layer | sage | propagate | graph
  n, e   nodes and directed edges (self-loops, where asked for, are part of e)
  hub    expected degree of the heaviest node of a power-law graph (exponent 2.1); 0: endpoints drawn uniformly
  dtype  f32 | bf16: storage of the node features and their gradients
  k      source partitions: 1 = the un-split graph; more = call by call, the running state in device memory
"""
import math

import torch

from paper_2111_06483_b200 import api

SLOPE = 0.2
ALPHA, ITERS = 0.9, 10   # propagation: weight of the neighbours, steps
DTYPES = {"f32": torch.float32, "bf16": torch.bfloat16}


def listed():
    return [
        # One attention layer of a small graph, forward and backward: citation-network size, where launches and host
        # time are what a step costs.
        dict(name="attention-tiny-f32", kind="attention", n=2_000, e=22_000, hub=0, heads=4, feat=16, dtype="f32", k=1,
             backward=True),
        # The paper's own schedule: eight source partitions visited one after the other, running softmax state between
        # the calls (Algorithms 1 and 2), forward and backward.
        dict(name="attention-seqpart-f32-k8", kind="attention", n=100_000, e=2_000_000, hub=2_000, heads=4, feat=32,
             dtype="f32", k=8, backward=True),
        # A hidden layer on a products-sized graph in single precision, forward and backward.
        dict(name="attention-medium-f32", kind="attention", n=2_450_000, e=62_000_000, hub=17_000, heads=4, feat=64,
             dtype="f32", k=1, backward=True),
        # Dense neighbourhoods (200 edges per node, hubs of tens of thousands), eight heads, bf16 storage.
        dict(name="attention-dense-bf16", kind="attention", n=1_000_000, e=200_000_000, hub=50_000, heads=8, feat=32,
             dtype="bf16", k=1, backward=True),
        # One layer of the largest single-GPU graph.
        dict(name="attention-large-bf16", kind="attention", n=20_000_000, e=300_000_000, hub=100_000, heads=4, feat=32,
             dtype="bf16", k=1, backward=True),
        # The layer that ends a classifier: one head as wide as there are classes (47 on ogbn-products), so that rows
        # are no whole number of 16-byte words.
        dict(name="attention-classes-bf16", kind="attention", n=170_000, e=2_500_000, hub=1_500, heads=1, feat=47,
             dtype="bf16", k=1, backward=True),
        # Inference with a two-head layer on a mid-sized graph: forward only, one launch chain.
        dict(name="attention-inference-bf16", kind="attention", n=233_000, e=11_600_000, hub=4_000, heads=2, feat=64,
             dtype="bf16", k=1, backward=False),
        # Sum aggregation of the products-sized graph with 256 columns, forward and backward (the transposed graph).
        dict(name="sum-medium-f32", kind="sum", n=2_450_000, e=62_000_000, hub=17_000, feat=256, dtype="f32"),
        # A whole hidden layer of a training step: projection, scores, attention, batch normalisation, and all of
        # their backward passes.
        dict(name="layer-bf16", kind="layer", n=1_000_000, e=15_000_000, hub=9_000, d_in=128, heads=4, feat=32,
             dtype="bf16"),
        # A GraphSage layer of hidden size 256 on the products-sized graph, forward and backward.
        dict(name="sage-medium-bf16", kind="sage", n=2_450_000, e=62_000_000, hub=17_000, d_in=256, d_out=256,
             dtype="bf16"),
        # Smoothing of class predictions over the graph: ten steps on as many columns as there are classes.
        dict(name="propagate-classes-f32", kind="propagate", n=500_000, e=10_000_000, hub=5_000, feat=47, dtype="f32"),
        # Graph preparation of the products-sized graph: CSR, CSC, long-row plans and four source partitions.
        dict(name="graph-medium-k4", kind="graph", n=2_450_000, e=62_000_000, hub=17_000, k=4),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _edges(rng, n, budget):
    """Edge count for n nodes: 4 to 100 per node, at most `budget`."""
    return max(16, min(int(n * math.exp(rng.uniform(math.log(4.0), math.log(100.0)))), int(budget)))


def _hub(rng, n, most=0.75):
    return 0 if rng.random() < 0.25 else max(8, int(n ** rng.uniform(0.55, most)))


def draw(rng):
    """One more case of the ranges above: sizes log-uniform from some hundreds of nodes to some millions."""
    kind = rng.choice(["attention"] * 6 + ["sum", "layer", "sage", "propagate", "graph"])
    dtype = rng.choice(["f32", "bf16"])
    if kind == "graph":
        n = _log_int(rng, 500, 4_000_000)
        return dict(kind=kind, n=n, e=_edges(rng, n, 80e6), hub=_hub(rng, n), k=rng.choice([1, 2, 3, 4, 6]))
    if kind in ("layer", "sage"):   # the projections take bf16 and widths that are multiples of eight
        n = _log_int(rng, 500, 2_000_000)
        hub = _hub(rng, n)
        d_in = 8 * _log_int(rng, 4, 32)
        if kind == "layer":
            heads, feat = rng.choice([(1, 64), (2, 32), (2, 64), (4, 16), (4, 32), (4, 64), (8, 16), (8, 32)])
            return dict(kind=kind, n=n, e=_edges(rng, n, 40e6), hub=hub, d_in=d_in, heads=heads, feat=feat, dtype="bf16")
        return dict(kind=kind, n=n, e=_edges(rng, n, 40e6), hub=hub, d_in=d_in, d_out=8 * _log_int(rng, 4, 32), dtype="bf16")
    if kind in ("sum", "propagate"):
        n = _log_int(rng, 500, 2_000_000)
        if rng.random() < 0.5:
            feat = 8 * _log_int(rng, 2, 32)
        else:                       # as many columns as there are classes
            feat = rng.randint(3, 180)
        steps = ITERS if kind == "propagate" else 2
        hub = _hub(rng, n, 0.62 if feat % 8 else 0.75)
        return dict(kind=kind, n=n, e=_edges(rng, n, min(40e6, 2e10 / (steps * feat))), hub=hub, feat=feat,
                    dtype=dtype if kind == "sum" else "f32")
    heads = rng.choice([1, 2, 3, 4, 4, 6, 8])
    whole = rng.random() < 0.75
    if whole:
        feat = rng.choice([f for f in (8, 16, 24, 32, 48, 64, 128) if heads * f <= 512])
    else:                           # rows that are no whole number of 16-byte words
        feat = rng.randint(3, max(5, 120 // heads))
    n = _log_int(rng, 500, 3_000_000 if whole else 400_000)
    e = _edges(rng, n, min(60e6, 8e9 / (heads * feat)) if whole else min(8e6, 3e8 / (heads * feat)))
    return dict(kind=kind, n=n, e=e, hub=_hub(rng, n, 0.75 if whole else 0.6), heads=heads, feat=feat, dtype=dtype,
                k=rng.choice([1, 1, 1, 2, 4, 8, 16]), backward=rng.random() < 0.75)


# ---- inputs ----------------------------------------------------------------------------------------------------------

def _graph_edges(n, e, hub, gen, dev):
    """(src, dst) int32: a power-law graph (weights (rank + c)^(-1/1.1), source and destination drawn independently,
    ranks scattered over the ids by a random permutation), or, with hub = 0, uniform endpoints and one self-loop per node."""
    if hub == 0:
        src = torch.randint(0, n, (e,), generator=gen, device=dev, dtype=torch.int32)
        dst = torch.randint(0, n, (e,), generator=gen, device=dev, dtype=torch.int32)
        loops = min(n, e)
        src[e - loops:] = torch.arange(loops, device=dev, dtype=torch.int32)
        dst[e - loops:] = torch.arange(loops, device=dev, dtype=torch.int32)
        return src, dst
    b = 1.0 - 1.0 / 1.1   # the cumulative weight of rank x is ((x + c)^b - c^b) / ((n + c)^b - c^b)
    lo, hi = 1e-3, float(n)
    for _ in range(50):
        c = math.sqrt(lo * hi)
        heaviest = e * ((1.0 + c) ** b - c ** b) / ((n + c) ** b - c ** b)
        lo, hi = (c, hi) if heaviest > hub else (lo, c)
    perm = torch.randperm(n, generator=gen, device=dev, dtype=torch.int32)
    ends = []
    for _ in range(2):
        x = torch.empty(e, dtype=torch.int32, device=dev)
        for at in range(0, e, 1 << 26):
            u = torch.rand(min(e - at, 1 << 26), generator=gen, device=dev, dtype=torch.float64)
            rank = u.mul_((n + c) ** b - c ** b).add_(c ** b).pow_(1.0 / b).sub_(c).to(torch.int64).clamp_(0, n - 1)
            x[at:at + rank.numel()] = perm[rank]
        ends.append(x)
    return ends[0], ends[1]


def prepare(case, seed):
    dev = torch.device("cuda")
    gen = torch.Generator(device=dev)
    gen.manual_seed(int(seed))
    kind, n, e = case["kind"], case["n"], case["e"]
    dt = DTYPES[case.get("dtype", "f32")]

    def normal(*shape, dtype=torch.float32, scale=1.0):
        x = torch.randn(*shape, generator=gen, device=dev, dtype=dtype)
        return x if scale == 1.0 else x.mul_(scale)

    src, dst = _graph_edges(n, e, case["hub"], gen, dev)
    s = dict(case=case)
    if kind == "graph":
        s.update(src=src, dst=dst)
        return s
    k = case.get("k", 1)
    s["g"] = g = api.Graph.from_coo(n, src, dst, k=k, build_parts=k > 1)
    del src, dst
    if kind == "attention":
        H, F = case["heads"], case["feat"]
        s.update(feat=normal(n, H, F, dtype=dt), el=normal(n, H), er=normal(n, H))
        if case["backward"]:
            s["gout"] = normal(n, H, F, dtype=dt)
    elif kind == "sum":
        s.update(x=normal(n, case["feat"], dtype=dt), gout=normal(n, case["feat"], dtype=dt), gt=g.whole.transposed())
    elif kind == "propagate":
        s["x0"] = torch.softmax(normal(n, case["feat"]).mul_(2.0), dim=1).to(dt)
        s["src_scale"], s["dst_scale"] = api.sym_norm_scales(g)
    elif kind == "layer":
        H, F, d_in = case["heads"], case["feat"], case["d_in"]
        s.update(h=normal(n, d_in, dtype=dt), W=normal(d_in, H * F, dtype=dt, scale=d_in ** -0.5),
                 a_l=normal(H, F, scale=F ** -0.5), a_r=normal(H, F, scale=F ** -0.5),
                 gamma=normal(H * F, scale=0.1).add_(1.0), beta=normal(H * F, scale=0.1), gy=normal(n, H * F, dtype=dt))
    elif kind == "sage":
        d_in, d_out = case["d_in"], case["d_out"]
        s.update(h=normal(n, d_in, dtype=dt), W=normal(d_in, d_out, dtype=dt, scale=d_in ** -0.5),
                 W_res=normal(d_in, d_out, dtype=dt, scale=d_in ** -0.5), gpre=normal(n, d_out, dtype=dt),
                 inv=api.rgcn_inv_degrees([g])[0])
    return s


# ---- one pass --------------------------------------------------------------------------------------------------------

def _graph_outputs(g, e):
    """A prepared graph as arrays whose sizes do not depend on the edges drawn: the long-row plans one after the other and
    filled up with -1, the partitions' indices one after the other (their CSC indices are slices of the whole graph's)."""
    w, pieces = g.whole, [g.whole] + g.parts
    plans = [x for p in pieces for sp in (p.split, p.t_split) for x in (sp.long_row, sp.long_seg)]
    room = 8 * (e // api.DEFAULT_THRESHOLD) + 2 * len(pieces)
    plan = torch.full((room,), -1, dtype=torch.int64, device=w.indptr.device)
    torch.cat(plans, out=plan[:sum(x.numel() for x in plans)])
    out = dict(whole=[w.indptr, w.indices, w.t_indptr, w.t_indices], plan=plan,
               counts=[x for p in pieces for x in (p.nnz, p.split.n_long, p.split.n_seg, p.t_split.n_long, p.t_split.n_seg)])
    if g.parts:
        out["indptr"] = [x for p in g.parts for x in (p.indptr, p.t_indptr)]
        out["indices"] = torch.cat([p.indices for p in g.parts])
    return out


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "graph":
        g = api.Graph.from_coo(case["n"], s["src"], s["dst"], k=case["k"], build_parts=case["k"] > 1)
        return _graph_outputs(g, case["e"])
    g = s["g"]
    if kind == "attention":
        feat, el, er = s["feat"], s["el"], s["er"]
        if case["k"] == 1:
            out, m, d = api.gat_forward(g, feat, el, er, SLOPE)
            if not case["backward"]:
                return dict(out=out, m=m, d=d)
            dfeat, del_, der = api.gat_backward(g, feat, el, er, m, d, s["gout"], SLOPE)
        else:
            # with bf16 storage the numerator is kept, so that the row dot does not see the rounding of `out`
            keep = case["dtype"] == "bf16" and case["backward"]
            out, m, d, *acc = api.gat_forward(g, feat, el, er, SLOPE, mode="stateful", keep_numerator=keep)
            if not case["backward"]:
                return dict(out=out, m=m, d=d)
            dfeat, del_, der = api.gat_backward(g, feat, el, er, m, d, s["gout"], SLOPE, out=out, mode="stateful",
                                                acc=acc[0] if keep else None)
        return dict(out=out, m=m, d=d, dfeat=dfeat, del_=del_, der=der)
    if kind == "sum":
        return dict(out=api.spmm_sum(g.whole, s["x"]), dx=api.spmm_sum(s["gt"], s["gout"]))
    if kind == "propagate":
        return api.propagate(g, s["x0"], ALPHA, ITERS, s["src_scale"], s["dst_scale"])
    if kind == "layer":
        h, W, a_l, a_r = s["h"], s["W"], s["a_l"], s["a_r"]
        out, saved = api.full_layer_forward(g, h, W, a_l, a_r, SLOPE, relu_input=True)
        x = out.view(case["n"], -1)
        y, stats = api.bn_forward(x, gamma=s["gamma"], beta=s["beta"])
        gx, dgamma, dbeta = api.bn_backward(x, s["gy"], stats, gamma=s["gamma"])
        dh, dW, da_l, da_r = api.full_layer_backward(g, h, W, a_l, a_r, saved, gx.view(out.shape), SLOPE, relu_input=True)
        return dict(y=y, dh=dh, dW=dW, da_l=da_l, da_r=da_r, dgamma=dgamma, dbeta=dbeta)
    if kind == "sage":
        pre, saved = api.sage_layer_forward(g, s["h"], s["W"], s["W_res"], s["inv"])
        dh, dW, dW_res = api.sage_layer_backward(g, s["h"], s["W"], s["W_res"], saved, s["gpre"])
        return dict(pre=pre, dh=dh, dW=dW, dW_res=dW_res)
    raise ValueError(kind)


# ---- what a pass cannot do without -----------------------------------------------------------------------------------

def work(case):
    """Bytes: every distinct input read once, every output written once (an array that a later pass of the same step reads
    again is counted again).  Operations: the multiplications and additions of the equations."""
    kind, n, e = case["kind"], case["n"], case["e"]
    index = 8 * (n + 1) + 4 * e
    b = 2 if case.get("dtype") == "bf16" else 4
    if kind == "graph":
        out = 2 * index
        if case["k"] > 1:
            out += case["k"] * 8 * (n + 1) + 4 * e + 8 * (n + case["k"])
        return {"bytes": 8 * e + out, "flops": 0}
    if kind == "attention":
        H, F = case["heads"], case["feat"]
        if not case["backward"]:
            return {"bytes": index + 2 * n * H * F * b + 16 * n * H, "flops": e * H * (2 * F + 4)}
        return {"bytes": 3 * index + 4 * n * H * F * b + 40 * n * H, "flops": e * H * (6 * F + 16)}
    if kind == "sum":
        return {"bytes": 2 * index + 4 * n * case["feat"] * b, "flops": 2 * e * case["feat"]}
    if kind == "propagate":
        return {"bytes": ITERS * (index + 8 * n + 3 * n * case["feat"] * b), "flops": ITERS * (2 * e + 3 * n) * case["feat"]}
    if kind == "layer":
        d, c = case["d_in"], case["heads"] * case["feat"]
        attention = 3 * index + 4 * n * c * b + 40 * n * case["heads"]
        dense = 3 * n * (d + c) * b               # h W, dz W^T, h^T dz
        norm = 5 * n * c * b                      # x -> y; x, gy -> gx
        return {"bytes": attention + dense + norm, "flops": 6 * n * d * c + e * (6 * c + 16 * case["heads"]) + 20 * n * c}
    if kind == "sage":
        d, c = case["d_in"], case["d_out"]
        sums = 2 * (index + 2 * n * d * b)
        dense = n * (2 * d + c) * b + n * (2 * d + c) * b + n * (c + 2 * d) * b   # forward, weights, inputs
        return {"bytes": sums + dense, "flops": 12 * n * d * c + 4 * e * d}
    raise ValueError(kind)


def tolerance(case):
    """Whole numbers are unique.  float32: sums of products in another order.  bf16: one rounding of each stored value,
    and what it does to the values computed from it."""
    if case["kind"] == "graph":
        return "exact"
    return {"rel": 1e-5, "max": 1e-3} if case["dtype"] == "f32" else {"rel": 1e-2, "max": 5e-2}
