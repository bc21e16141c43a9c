"""Performance cases of the route-maintenance library: what a user of it runs, through its public
entry points, from the smallest configuration to the largest.

Kinds of case
  layers   one forward pass of a model's routing: RouteLedger.route_anchor / route_relay layer
           after layer on one stream, inputs resident on the GPU (bf16 or fp32, with and without
           the causal mask, global sentinels, token ranges)
  buckets  the same with heads of different route widths: BucketSet.route_layer
  host     the same from pinned host buffers: RouteLedger.route_layers_host, routes copied back
  attend   the consumer of the routes (Eq. 3): attend_token_ranges over an anchor's token ranges

The ids inside a route or sentinel row are a set (their order carries no meaning by the library's
contract), so `run` returns those rows sorted.
"""
import math

import torch

from paper_2609_07306_b200 import binding as B
from paper_2609_07306_b200.ledger import BucketSet, RouteLedger, attend_token_ranges

GLOBAL_SINK, GLOBAL_RECENT = 1, 2


def _layers(name, problems, n_q, n_k, d, k, m, r, layers, anchor_every, rho, **kw):
    c = dict(name=name, kind="layers", problems=problems, n_q=n_q, n_k=n_k, d=d, k=k, m=m, r=r,
             layers=layers, anchor_every=anchor_every, rho=rho, dtype="bf16", causal=True,
             offset=0, centroids=64, redraw=False, global_sentinels=0, chunk_tokens=0, coalesce=False)
    c.update(kw)
    return c


def listed():
    return [
        # the smallest configuration: one head, fp32 inputs -- latency of the calls themselves
        _layers("tiny_f32", 1, 128, 128, 64, 8, 4, 4, 4, 4, 0.05, dtype="f32", causal=False, centroids=16),
        # a short prompt of an eight-head model: a few CTAs per layer, launch- and latency-bound
        _layers("moderate", 8, 256, 256, 128, 16, 8, 8, 12, 6, 0.15, centroids=32),
        # odd sizes: a prompt appended to a cached prefix (n_k > n_q, causal offset), ragged in
        # every dimension, both mandatory global sentinels, ranges of adjacent chunks merged
        _layers("ragged", 15, 389, 777, 64, 20, 10, 7, 12, 6, 0.10, offset=388, centroids=50,
                global_sentinels=GLOBAL_SINK | GLOBAL_RECENT, chunk_tokens=32, coalesce=True),
        # the shape of the method's own experiments: fp32, ten seeds of 384 x 192 chunks, no mask
        _layers("paper_f32", 10, 384, 192, 64, 12, 24, 12, 16, 8, 0.03, dtype="f32", causal=False, centroids=24),
        # the chunk sweep's largest point: one sequence of a 32-head model
        _layers("sweep_1024", 32, 1024, 1024, 128, 32, 16, 16, 16, 8, 0.30),
        # many short sequences with one anchor (the sentinel ablation's shape)
        _layers("ablation", 256, 256, 256, 128, 12, 12, 12, 24, 24, 0.003, causal=False, centroids=32),
        # a batch of eight 32-head sequences, strong drift: nearly every row is routed again
        _layers("high_drift", 256, 1024, 1024, 128, 32, 16, 16, 16, 8, 0.30, redraw=True),
        # the same in the regime the method is built for: few rows are routed again
        _layers("low_drift", 256, 1024, 1024, 128, 32, 16, 16, 16, 8, 0.005),
        # long context: 2048 chunks, wide routes, token ranges for the attention backend
        _layers("long_ctx", 64, 2048, 2048, 128, 64, 32, 32, 8, 8, 0.15, centroids=128, chunk_tokens=64),
        # heads with their own route widths (8, 16 and 32), four sequences
        _layers("buckets", 128, 512, 512, 128, 0, 16, 16, 8, 8, 0.05, kind="buckets", w0=8, w1=16, w2=32),
        # one 32-head sequence from pinned host memory, every layer's routes copied back
        _layers("host", 32, 512, 512, 128, 32, 16, 16, 8, 8, 0.15, kind="host"),
        # attention of eight heads over the tokens their routes select
        _layers("attend", 8, 256, 256, 128, 16, 8, 8, 1, 1, 0.15, kind="attend", centroids=32,
                chunk_tokens=64),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _unnamed(*args, **kw):
    c = _layers("", *args, **kw)
    del c["name"]
    return c


def draw(rng):
    kind = rng.choices(["layers", "buckets", "host", "attend"], [9, 1, 1, 1])[0]
    d = rng.choice([64, 128])
    if kind == "attend":
        return _unnamed(_log(rng, 1, 12), _log(rng, 64, 300), _log(rng, 64, 300), d, rng.randint(6, 20),
                        rng.randint(0, 12), rng.randint(0, 12), 1, 1, 0.15, kind=kind, centroids=32,
                        causal=rng.random() < 0.7, chunk_tokens=rng.choice([16, 32, 48, 64]),
                        coalesce=rng.random() < 0.5, dtype=rng.choice(["bf16", "bf16", "f32"]))
    f32 = kind == "layers" and rng.random() < 0.2
    n_q, n_k = _log(rng, 100, 2048), _log(rng, 128, 2048)
    if rng.random() < 0.5:
        n_k = n_q = max(n_q, 128)
    if f32:
        n_q, n_k = min(n_q, 600), min(n_k, 600)
    # half of the largest listed case's score pairs at most, spread over the logarithm
    most = min(256, int(0.5 * 16 * 256 * 1024 * 1024 / (12 * n_q * n_k)))
    problems = _log(rng, 1, max(1, min(most, 24) if f32 else most))
    if kind == "host":                                     # one sequence
        problems, n_q, n_k = min(problems, 32), min(n_q, 1024), min(n_k, 1024)
    top = min(64, n_k // 4)
    k, m, r = _log(rng, 6, top), rng.randint(0, min(32, top)), rng.randint(0, min(32, top))
    layers = rng.randint(4, 12)
    causal = rng.random() < 0.7
    kw = dict(kind=kind, causal=causal, offset=max(0, n_k - n_q) if causal else 0,
              centroids=rng.choice([24, 32, 64]), dtype="f32" if f32 else "bf16")
    if kind == "layers":
        kw.update(global_sentinels=rng.choice([0, 0, 0, 3]), chunk_tokens=rng.choice([0, 0, 64]))
        kw.update(coalesce=kw["chunk_tokens"] > 0 and rng.random() < 0.5)
    if kind == "buckets":
        kw.update(w0=max(2, k // 4), w1=max(3, k // 2), w2=max(4, k))
    return _unnamed(problems, n_q, n_k, d, k, m, r, layers, rng.choice([4, 8, 16]),
                    math.exp(rng.uniform(math.log(0.003), math.log(0.3))), **kw)


# ------------------------------------------------------------------------------------ inputs
def _drifting_inputs(c, seed):
    """Chunk representations that drift from layer to layer: rows around the centroids their
    problem's queries and keys share, X <- sqrt(1 - rho^2) X + rho G per layer; with `redraw` a
    tenth of the centroids (and the rows around them) is drawn anew every fourth layer."""
    dev = torch.device("cuda")
    g = torch.Generator(device=dev).manual_seed(int(seed))
    P, d, C, rho = c["problems"], c["d"], c["centroids"], c["rho"]
    dt = torch.float32 if c["dtype"] == "f32" else torch.bfloat16
    inv = d ** -0.5

    def normal(*shape):
        return torch.randn(shape, generator=g, device=dev).mul_(inv)

    mu = normal(P, C, d)
    sides = []
    for n in (c["n_q"], c["n_k"]):
        assign = torch.randint(0, C, (P, n), generator=g, device=dev)
        pick = assign[:, :, None].expand(P, n, d)
        sides.append([assign, pick, mu.gather(1, pick) + 0.5 * normal(P, n, d)])
    out = []
    for layer in range(c["layers"]):
        if layer:
            for s in sides:
                s[2].mul_(math.sqrt(1.0 - rho * rho)).add_(normal(*s[2].shape), alpha=rho)
            if c["redraw"] and layer % 4 == 0:
                new = torch.rand((P, C), generator=g, device=dev).argsort(1) < max(1, round(0.1 * C))
                mu = torch.where(new[:, :, None], normal(P, C, d), mu)
                for s in sides:
                    fresh = mu.gather(1, s[1]) + 0.5 * normal(*s[2].shape)
                    s[2] = torch.where(new.gather(1, s[0])[:, :, None], fresh, s[2])
        out.append(tuple(s[2].to(dt).contiguous() for s in sides))
    return out


def _config(c):
    return B.rr_config(batch=1, heads=c["problems"], n_q=c["n_q"], n_k=c["n_k"], d=c["d"], k=max(1, c["k"]),
                       m=c["m"], r=c["r"], dtype=B.RR_F32 if c["dtype"] == "f32" else B.RR_BF16,
                       causal=1 if c["causal"] else 0, causal_offset=c["offset"], gamma=0.0, seed=1,
                       chunk_tokens=c["chunk_tokens"], coalesce_ranges=1 if c["coalesce"] else 0,
                       global_sentinels=c["global_sentinels"])


def _widths(c):
    return [(c["w0"], c["w1"], c["w2"])[p % 3] for p in range(c["problems"])]


def prepare(case, seed):
    c = case
    inputs = _drifting_inputs(c, seed)
    s = {"case": c, "anchors": [l % c["anchor_every"] == 0 for l in range(c["layers"])]}
    if c["kind"] == "buckets":
        s["set"] = BucketSet(_config(c), _widths(c))
        s["inputs"] = inputs              # (already bucket-major: problems are drawn alike)
        return s
    led = s["ledger"] = RouteLedger(_config(c))
    if c["kind"] == "host":
        s["qc"] = [q.cpu().pin_memory() for q, _ in inputs]
        s["kc"] = [k.cpu().pin_memory() for _, k in inputs]
        s["dev_q"] = [torch.empty_like(inputs[0][0]) for _ in range(2)]
        s["dev_k"] = [torch.empty_like(inputs[0][1]) for _ in range(2)]
        s["dev_r"] = [torch.empty_like(led.routes) for _ in range(2)]
        s["routes"] = [torch.empty((led.rows, c["k"]), dtype=torch.int32).pin_memory() for _ in inputs]
        s["up"], s["down"] = torch.cuda.Stream(), torch.cuda.Stream()
    elif c["kind"] == "attend":
        g = torch.Generator(device="cuda").manual_seed(int(seed) + 1)
        led.route_anchor(*inputs[0], 0)
        s["ranges"] = led.token_ranges.contiguous()
        dt, tokens = inputs[0][0].dtype, c["n_k"] * c["chunk_tokens"]
        s["q"] = torch.randn((led.rows, c["d"]), generator=g, device="cuda").to(dt)
        s["keys"], s["values"] = (torch.randn((c["problems"], tokens, c["d"]), generator=g, device="cuda").to(dt)
                                  for _ in range(2))
        s["inputs"] = inputs              # (the ledger's work is done; kept until it has run)
    else:
        s["inputs"] = inputs
        s["slots"] = torch.arange(led.rows, device="cuda", dtype=torch.int32)
    return s


# --------------------------------------------------------------------------------------- run
def _sets(ids):
    return torch.sort(ids, dim=1).values


def _state(led):
    """The ledger and the last layer's per-row outputs."""
    return {"routes": _sets(led.routes), "sentinels": _sets(led.sentinels), "ages": led.ages,
            "kth_score": led.kth_score, "margin": led.margin, "flags": led.flags, "alpha": led.alpha,
            "beta": led.beta, "refresh_count": led.refresh_count, "problem_offsets": led.problem_offsets}


def run(state):
    c = state["case"]
    if c["kind"] == "attend":
        return attend_token_ranges(state["ranges"], c["n_q"], state["q"], state["keys"], state["values"],
                                   c["d"] ** -0.5)
    if c["kind"] == "buckets":
        bs = state["set"]
        for l, (qc, kc) in enumerate(state["inputs"]):
            bs.route_layer(qc, kc, l, state["anchors"][l])
        return [_state(led) for led in bs.buckets]
    led = state["ledger"]
    if c["kind"] == "host":
        led.route_layers_host(state["qc"], state["kc"], state["anchors"], 0, state["dev_q"], state["dev_k"],
                              state["dev_r"], state["routes"], state["up"], state["down"])
        # the caller's side of the contract: every stream is done before the routes are read
        for st in (state["up"], state["down"], torch.cuda.current_stream()):
            st.synchronize()
        return {"host_routes": state["routes"], "ages": led.ages, "kth_score": led.kth_score,
                "margin": led.margin, "flags": led.flags, "alpha": led.alpha, "beta": led.beta,
                "sentinels": _sets(led.sentinels)}
    for l, (qc, kc) in enumerate(state["inputs"]):
        (led.route_anchor if state["anchors"][l] else led.route_relay)(qc, kc, l)
    out = _state(led)
    # the refresh list is defined up to its count
    out["refresh_rows"] = torch.where(state["slots"] < led.refresh_count, led.refresh_rows, -1)
    if c["chunk_tokens"]:
        out["token_ranges"] = led.token_ranges
    return out


# ------------------------------------------------------------------------------ floor, accuracy
def _valid_pairs(c):
    if not c["causal"]:
        return c["n_q"] * c["n_k"]
    return sum(min(c["n_k"], i + 1 + c["offset"]) for i in range(c["n_q"]))


def work(case):
    c = case
    es = 4 if c["dtype"] == "f32" else 2
    if c["kind"] == "attend":
        rows, tokens = c["problems"] * c["n_q"], c["n_k"] * c["chunk_tokens"]
        picked = sum(min(c["k"], min(c["n_k"], i + 1) if c["causal"] else c["n_k"]) for i in range(c["n_q"]))
        return {"bytes": 2 * c["problems"] * tokens * c["d"] * es + rows * (c["k"] * 8 + c["d"] * (es + 4)),
                "flops": 4.0 * c["problems"] * picked * c["chunk_tokens"] * c["d"]}
    P, rows = c["problems"], c["problems"] * c["n_q"]
    k = c["k"] if c["kind"] != "buckets" else (c["w0"] + c["w1"] + c["w2"]) / 3
    sw = c["m"] + c["r"] + bin(c["global_sentinels"]).count("1")
    anchors = sum(l % c["anchor_every"] == 0 for l in range(c["layers"]))
    relays = c["layers"] - anchors
    # every layer reads its inputs; an anchor writes the ledger rows (ids, k-th score, margin, age)
    # and a relay reads them and writes flag, alpha, beta, age; re-routed rows come on top
    moved = c["layers"] * P * (c["n_q"] + c["n_k"]) * c["d"] * es
    moved += anchors * rows * ((k + sw) * 4 + 12 + (8 * k if c["chunk_tokens"] else 0))
    moved += relays * rows * ((k + sw) * 4 + 13)
    if c["kind"] == "host":
        moved += c["layers"] * rows * k * 4
    # an anchor scores every valid pair, a relay at least every row's candidates
    return {"bytes": moved, "flops": 2.0 * c["d"] * P * (anchors * _valid_pairs(c) + relays * c["n_q"] * (k + sw))}


def tolerance(case):
    # fp32 accumulation of exact products everywhere (attend: fp32 softmax as well); ids may differ
    # where two scores agree to the last bits
    return {"rel": 1e-5, "max": 1e-3, "differ": 1e-4}
