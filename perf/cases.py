"""What the performance of this framework is measured on.

Each case is one piece of work that a program serving a pruned-pool MoE model
has the library do, through the Python binding of its C ABI:

  decode      one MoE layer of a decode step (batches of 1 to 512 tokens) over
              the full pool or a retained pool, with or without a shared expert,
              with a caller's workspace or through the entry point that needs
              none
  stack       several layers of one decode step back to back on one stream,
              each with its own weights, under skewed expert popularity
  prefill     the full-pool layer on a prompt chunk of 1024 to 8192 tokens
              (pruning masks decode only, so prefill runs every expert)
  calibrate   one calibration batch of importance statistics and the retained
              set chosen from them
  compact     the compact checkpoint of a layer's retained experts
  route       routing and grouping alone, as a program runs them to count the
              experts that a batch touches

Layers are the Tiny, Qwen-class and Qwen3.6-shaped ones of this repository;
weights are bf16 ~ N(0, 0.02), the router fp32 ~ N(0, 0.02), hidden states
bf16 ~ N(0, 1).  Skewed popularity is a Zipf(1.1) rank bias on the router
logits, realised by one constant hidden element.
"""
from __future__ import annotations

import math

import torch

import paper_2609_34117_gb300 as sw
from paper_2609_34117_gb300 import binding

# name: (hidden, experts, expert intermediate width, top-k)
LAYERS = {
    "tiny": (256, 16, 128, 2),
    "qwen": (2048, 128, 768, 8),
    "qwen36": (2048, 256, 512, 8),
}
SHARED_INTER = 1024  # the Qwen3.6-shaped decoder's two merged shared experts of 512
ZIPF = 1.1


def _case(name, kind, layer, batch, retained=0, skew=False, shared=False, noalloc=False, layers=1,
          criterion="", shuffled=False):
    """retained: size of the retained pool, 0 for the full pool."""
    c = dict(kind=kind, layer=layer, batch=batch, retained=retained, skew=skew, shared=shared,
             noalloc=noalloc, layers=layers, criterion=criterion, shuffled=shuffled)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the smallest call: a toy layer, where launches and latency are everything
        _case("tiny_p50_b4", "decode", "tiny", 4, 8),
        # one user, one token at a time, in an engine that gives no workspace
        _case("qwen_p50_b1_noalloc", "decode", "qwen", 1, 64, noalloc=True),
        # a few dozen concurrent requests on an aggressively pruned pool, ragged batch
        _case("qwen_p75_b37", "decode", "qwen", 37, 32),
        # the unpruned decode layer at the batch the headline is quoted on
        _case("qwen_full_b64", "decode", "qwen", 64),
        # a heavily loaded pruned server
        _case("qwen_p50_b500", "decode", "qwen", 500, 64),
        # the distilled decoder: pruned pool plus the gated shared expert
        _case("qwen36_shared_p50_b96", "decode", "qwen36", 96, 128, shared=True),
        # one decode step through consecutive layers with popular experts
        _case("stack8_skew_p50_b256", "stack", "qwen", 256, 64, skew=True, layers=8),
        # a prompt chunk of odd length with popular experts, full pool
        _case("prefill_skew_b4001", "prefill", "qwen", 4001, skew=True),
        # the largest prompt chunk, many small experts and the shared expert
        _case("prefill_qwen36_shared_b8192", "prefill", "qwen36", 8192, shared=True),
        # a calibration batch, and the half of the pool that it keeps
        _case("calibrate_b2048", "calibrate", "qwen", 2048, 64, criterion="reap"),
        # a decode instance loading only its retained experts
        _case("compact_p50", "compact", "qwen", 0, 64, shuffled=True),
        # counting the experts that a batch touches
        _case("route_p25_b300", "route", "qwen", 300, 96),
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _pool(rng, layer):
    """A retained-pool size: the full pool, a usual pruning ratio or any size between."""
    _, E, _, k = LAYERS[layer]
    m = rng.choice([0, 3 * E // 4, E // 2, E // 4, rng.randint(max(k, E // 5), E - 1)])
    return m


def draw(rng):
    kind = rng.choice(["decode", "decode", "decode", "decode", "stack", "prefill", "prefill",
                       "calibrate", "compact", "route"])
    layer = rng.choice(["qwen", "qwen", "qwen36"])
    shuffled = rng.random() < 0.25
    if kind == "decode":
        layer = rng.choice(["tiny", "qwen", "qwen", "qwen36", "qwen36"])
        batch = _log_int(rng, 1, 512)
        shared = layer == "qwen36" and rng.random() < 0.5
        # the entry point without a workspace holds the Qwen-class layers up to 128 tokens
        noalloc = not shared and batch <= 128 and rng.random() < 0.25
        return _case("", kind, layer, batch, _pool(rng, layer), rng.random() < 0.3, shared, noalloc,
                     shuffled=shuffled)
    if kind == "stack":
        return _case("", kind, layer, _log_int(rng, 16, 512), _pool(rng, layer), rng.random() < 0.7,
                     layers=rng.randint(2, 5), shuffled=shuffled)
    if kind == "prefill":
        return _case("", kind, layer, _log_int(rng, 1024, 8192), 0, rng.random() < 0.5,
                     layer == "qwen36" and rng.random() < 0.5)
    if kind == "calibrate":
        _, E, _, k = LAYERS[layer]
        return _case("", kind, layer, _log_int(rng, 256, 4096), rng.randint(E // 4, 3 * E // 4),
                     rng.random() < 0.5, criterion=rng.choice(["mass", "ean", "reap"]))
    if kind == "compact":
        _, E, _, k = LAYERS[layer]
        return _case("", kind, layer, 0, rng.randint(E // 4, 3 * E // 4), shuffled=shuffled)
    return _case("", "route", layer, _log_int(rng, 1, 4096), _pool(rng, layer), rng.random() < 0.5,
                 shuffled=shuffled)


# --------------------------------------------------------------------------
# inputs, from the seed alone
# --------------------------------------------------------------------------
def _normal(shape, std, dtype, g):
    return torch.empty(shape, dtype=dtype, device="cuda").normal_(0.0, std, generator=g)


def _zipf_bias(E, g):
    rank = torch.randperm(E, generator=g, device="cuda").to(torch.float32) + 1.0
    return -ZIPF * torch.log(rank)


def _inputs(case, seed):
    """One dict of tensors per layer."""
    H, E, I, _ = LAYERS[case["layer"]]
    layers = []
    for n in range(case["layers"]):
        g = torch.Generator(device="cuda")
        g.manual_seed(1000 * int(seed) + n)
        d = {"router": _normal((E, H), 0.02, torch.float32, g)}
        if case["batch"]:
            d["x"] = _normal((case["batch"], H), 1.0, torch.bfloat16, g)
        if case["skew"]:
            d["x"][:, -1] = 1.0
            d["router"][:, -1] = _zipf_bias(E, g)
        if case["kind"] != "route":
            d["gate_up"] = _normal((E, 2 * I, H), 0.02, torch.bfloat16, g)
            d["down"] = _normal((E, H, I), 0.02, torch.bfloat16, g)
        # the ids of the experts with the highest importance score
        d["retained"] = None
        if case["retained"] and case["kind"] != "calibrate":
            ids = torch.rand(E, generator=g, device="cuda").argsort()[: case["retained"]]
            if not case["shuffled"]:
                ids = ids.sort().values
            d["retained"] = ids.to(torch.int32).contiguous()
        if case["shared"]:
            d["s_gate"] = _normal((H,), 0.05, torch.float32, g)
            d["s_gate_up"] = _normal((2 * SHARED_INTER, H), 0.02, torch.bfloat16, g)
            d["s_down"] = _normal((H, SHARED_INTER), 0.02, torch.bfloat16, g)
        layers.append(d)
    return layers


def prepare(case, seed):
    """The inputs, and the workspace and output buffers that a serving program keeps."""
    H, E, I, k = LAYERS[case["layer"]]
    B = case["batch"]
    layers = _inputs(case, seed)
    state = {"case": case, "layers": layers, "workspace": None}
    if case["kind"] != "compact" and not case["noalloc"]:
        if case["shared"]:
            n = sw.slimwise_moe_shared_workspace_size(B, H, E, I, k, SHARED_INTER)
            state["workspace"] = torch.empty(n, dtype=torch.uint8, device="cuda")
        else:
            # routing alone is sized for the smallest expert, as the binding's default
            inter = 64 if case["kind"] == "route" else I
            state["workspace"] = sw.alloc_workspace(B, H, E, inter, k)
    if case["kind"] in ("decode", "stack", "prefill", "calibrate"):
        for d in layers:
            d["out"] = torch.empty((B, H), dtype=torch.bfloat16, device="cuda")
    return state


# --------------------------------------------------------------------------
# one pass
# --------------------------------------------------------------------------
def _layer(case, d, workspace, k):
    if case["noalloc"]:
        return binding.slimwise_moe_decode_noalloc(d["x"], d["router"], d["retained"], d["gate_up"],
                                                   d["down"], k, d["out"])
    if case["shared"]:
        return sw.slimwise_moe_decode_shared(d["x"], d["router"], d["retained"], d["gate_up"],
                                             d["down"], k, d["s_gate"], d["s_gate_up"],
                                             d["s_down"], out=d["out"], workspace=workspace)
    if d["retained"] is None:
        return sw.slimwise_moe_decode_full(d["x"], d["router"], d["gate_up"], d["down"], k,
                                           out=d["out"], workspace=workspace)
    return sw.slimwise_moe_decode(d["x"], d["router"], d["retained"], d["gate_up"], d["down"], k,
                                  out=d["out"], workspace=workspace)


def run(state):
    case, layers, workspace = state["case"], state["layers"], state["workspace"]
    _, E, _, k = LAYERS[case["layer"]]
    kind = case["kind"]
    if kind == "compact":
        d = layers[0]
        return sw.slimwise_moe_compact_layer(d["gate_up"], d["down"], d["router"], d["retained"])
    if kind == "route":
        d = layers[0]
        return sw.slimwise_moe_route(d["x"], d["router"], d["retained"], k, E, workspace=workspace)
    if kind == "calibrate":
        d = layers[0]
        stats, out = sw.slimwise_moe_expert_stats(d["x"], d["router"], d["gate_up"], d["down"], k,
                                                  out=d["out"], workspace=workspace)
        ids = sw.slimwise_moe_select_retained(stats, case["retained"], case["criterion"])
        return {"out": out, "stats": stats, "retained": ids}
    return [_layer(case, d, workspace, k) for d in layers]


# --------------------------------------------------------------------------
# what a pass cannot do without
# --------------------------------------------------------------------------
def _pool_size(case):
    _, E, _, _ = LAYERS[case["layer"]]
    return E if case["kind"] == "calibrate" or not case["retained"] else case["retained"]


def _expected_union(case):
    """Distinct experts that a batch selects, from one simulated batch of logits."""
    H, E, _, k = LAYERS[case["layer"]]
    m, B = _pool_size(case), case["batch"]
    g = torch.Generator().manual_seed(5)
    z = torch.randn((B, m), generator=g) * (0.02 * math.sqrt(H))
    if case["skew"]:
        rank = torch.randperm(E, generator=g)[:m].to(torch.float32) + 1.0
        z = z - ZIPF * torch.log(rank)
    return int(torch.unique(torch.topk(z, k, dim=1).indices).numel())


def work(case):
    H, E, I, k = LAYERS[case["layer"]]
    m, B = _pool_size(case), case["batch"]
    expert = 3 * I * H * 2
    if case["kind"] == "compact":
        return {"bytes": 2 * m * (expert + H * 4), "flops": 0}
    route_bytes = m * H * 4 + B * H * 2
    route_flops = 2 * B * m * H
    if case["kind"] == "route":
        return {"bytes": route_bytes + B * k * 16 + 3 * E * 4, "flops": route_flops}
    nbytes = route_bytes + B * H * 2 + _expected_union(case) * expert
    flops = route_flops + 6 * B * k * H * I
    if case["shared"]:
        nbytes += 3 * SHARED_INTER * H * 2 + H * 4
        flops += 6 * B * H * SHARED_INTER
    if case["kind"] == "calibrate":
        nbytes += E * 32
    return {"bytes": case["layers"] * nbytes, "flops": case["layers"] * flops}


def tolerance(case):
    if case["kind"] == "compact":
        return "exact"  # a copy
    if case["kind"] == "route":
        return {"rel": 2e-6}  # ids and counts are whole numbers; gates are fp32
    if case["kind"] == "calibrate":
        # one expert changing places at the edge of the retained set shifts the
        # sorted ids between its old place and its new one
        return {"rel": 1e-2, "differ": 0.05}
    # bf16 activations between the two products, bf16 expert outputs and results:
    # 2.9e-3 from the 64-bit result
    return {"rel": 1e-2, "max": 0.06}


# --------------------------------------------------------------------------
# the same in 64 bits, in plain torch
# --------------------------------------------------------------------------
def _select64(d, k):
    x, router = d["x"].double(), d["router"].double()
    E = router.shape[0]
    pool = torch.arange(E, device=x.device) if d["retained"] is None else d["retained"].long()
    pool = pool.sort().values
    z = x @ router[pool].T
    top, at = torch.sort(z, dim=1, descending=True, stable=True)
    return pool[at[:, :k]], torch.softmax(top[:, :k], dim=1)


def _swiglu64(x, gate_up, down):
    h = x @ gate_up.double().T
    inter = h.shape[1] // 2
    return (torch.nn.functional.silu(h[:, :inter]) * h[:, inter:]) @ down.double().T


def _layer64(d, k, shared, stats=None):
    x = d["x"].double()
    idx, gates = _select64(d, k)
    out = torch.zeros_like(x)
    for e in torch.unique(idx).tolist():
        tok, slot = (idx == e).nonzero(as_tuple=True)
        y = _swiglu64(x[tok], d["gate_up"][e], d["down"][e])
        g = gates[tok, slot]
        out.index_add_(0, tok, g[:, None] * y)
        if stats is not None:
            norm = y.norm(dim=1)
            stats[e] = torch.stack([torch.tensor(float(tok.numel()), device=x.device,
                                                 dtype=torch.float64),
                                    g.sum(), norm.sum(), (g * norm).sum()])
    if shared:
        s = torch.sigmoid(x @ d["s_gate"].double())
        out += s[:, None] * _swiglu64(x, d["s_gate_up"], d["s_down"])
    return out


def exact(case, seed):
    _, E, _, k = LAYERS[case["layer"]]
    layers = _inputs(case, seed)
    if case["kind"] == "compact":
        d = layers[0]
        ids = d["retained"].sort().values
        rows = ids.long()
        return d["gate_up"][rows], d["down"][rows], d["router"][rows], ids
    if case["kind"] == "route":
        idx, gates = _select64(layers[0], k)
        B = idx.shape[0]
        flat = idx.flatten()
        counts = torch.bincount(flat, minlength=E)
        perm = torch.sort(flat, stable=True).indices
        union = counts.nonzero().flatten()
        ids = torch.full((E,), -1, device=flat.device, dtype=torch.int64)
        ids[: union.numel()] = union
        pos = torch.empty_like(perm)
        pos[perm] = torch.arange(B * k, device=flat.device)
        offsets = torch.zeros(E + 1, device=flat.device, dtype=torch.int64)
        offsets[1:] = counts.cumsum(0)
        res = {"topk_idx": idx, "topk_gate": gates, "counts": counts, "offsets": offsets,
               "union_ids": ids, "union_size": torch.tensor([union.numel()], device=flat.device),
               "perm": perm, "pos": pos}
        return {n: t if n == "topk_gate" else t.to(torch.int32) for n, t in res.items()}
    if case["kind"] == "calibrate":
        stats = torch.zeros((E, 4), dtype=torch.float64, device="cuda")
        out = _layer64(layers[0], k, False, stats)
        # the scores of neighbouring experts can be closer than 16-bit outputs
        # resolve: only the routing mass ranks the same at every precision
        ids = None
        if case["criterion"] == "mass":
            order = torch.sort(stats[:, 1], descending=True, stable=True).indices
            ids = order[: case["retained"]].sort().values.to(torch.int32)
        return {"out": out, "stats": stats, "retained": ids}
    return [_layer64(d, k, case["shared"]) for d in layers]
