"""Performance cases of the streaming-MoE decode library: what its users have it do, through its public calls.

Kinds of work (``case["kind"]``):

* ``steps``  -- a decoder's loop: one ``moe_layer_decode`` per layer on an ordinary stream (attention and the
  rest of the block run between two of them, so nothing is chained); every layer predicts its successor's
  routing on the way.
* ``chain``  -- data-dependent layer-steps, ``moe_layer_decode_dependent``, chained and replayed from a CUDA
  graph: tokens one after the other, each through all layers, x of a layer being the state the layer
  before it wrote.
* ``burst``  -- layer-steps that depend on one another through the routing only, chained and replayed from
  a CUDA graph (the throughput form; the repository's headline benchmark).
* ``stack``  -- ``StackDecoder``: a token through a stack of layers, experts staged from the pinned-host
  tier as the prediction says (``slots`` < ``E``), or all resident (``slots`` == ``E``).
* ``ffn``    -- T tokens at once: routing (a prerouter head, or a router's logits with Zipf popularity), then
  ``moe_expert_ffn_int4_lora`` over a resident layer: batched decode, chunked prefill, prefill.
* ``heads``  -- the full (MLP) prerouter heads of a stack in one flush.
* ``gate``   -- sigmoid-group routing of given router logits.

Shapes are those of the repository's configurations (a small layer H=1024 I=256 E=16; the 35B-class layer
H=2048 I=512 E=256 int4 g64 with rank-16 adapters) and of its tests; value distributions are those of
``workloads/synth.py``.  ``draw`` varies sizes, types and options over the same ranges.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2609_18063_b200 as edg
from paper_2609_18063_b200 import layer_io
from paper_2609_18063_b200.decoder import StackDecoder

# the two layer shapes of the configurations
SMALL = dict(H=1024, I=256, E=16, K=2, group=32, rank=8, head="f32")
LARGE = dict(H=2048, I=512, E=256, K=8, group=64, rank=16, head="f16")
COMMON = dict(out="f32", per_expert_adapters=False)


def listed():
    return [
        # the smallest call there is: one layer-step of a small model, fp32 head
        dict(COMMON, name="step_small", kind="steps", layers=1, shared=False, **SMALL),
        # batch-1 decode inside a decoder: eight layers of the 35B class, one launch each, fp16 head
        dict(COMMON, name="steps_35b", kind="steps", layers=8, shared=False, **LARGE),
        # batch-1 decode as a captured chain of dependent layer-steps: 16 tokens of 8 layers
        dict(COMMON, name="chain_35b", kind="chain", layers=8, steps=128, **LARGE),
        # the headline workload: layer-steps that depend on one another through the routing alone
        dict(COMMON, name="burst_35b", kind="burst", layers=8, steps=1280, **LARGE),
        # a token of the shipped K = 4 profile through a resident stack, host loop included
        dict(COMMON, name="stack_resident", kind="stack", layers=12, slots=256, **dict(LARGE, K=4)),
        # the same loop when the experts do not fit: 32 slots a layer, missing experts come from pinned memory
        dict(COMMON, name="stack_streaming", kind="stack", layers=4, slots=32, **LARGE),
        # the heads of a 40-layer stack at their full form, one flush per token
        dict(COMMON, name="heads_40", kind="heads", heads=40, width=512, **LARGE),
        # routing of a prefill chunk of the 8B tier: 128 experts in 8 groups, 4 kept
        dict(name="gate_4096", kind="gate", T=4096, E=128, K=8, groups=8, keep=4, bias=True),
        # a handful of concurrent requests, through four layers
        dict(COMMON, name="batch_5", kind="ffn", T=5, layers=4, router="head", **LARGE),
        # batched decode: 64 concurrent tokens
        dict(COMMON, name="batch_64", kind="ffn", T=64, layers=1, router="head", **LARGE),
        # a ragged prefill chunk, bf16 output, one adapter per expert
        dict(name="chunk_333", kind="ffn", T=333, layers=1, router="zipf", out="bf16", per_expert_adapters=True, **LARGE),
        # prefill: 4096 tokens with Zipf(1.1) popularity of the experts
        dict(COMMON, name="prefill_4096", kind="ffn", T=4096, layers=1, router="zipf", **LARGE),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, round(math.exp(rng.uniform(math.log(lo), math.log(hi))))))


def draw(rng):
    kind = rng.choice(["steps", "chain", "burst", "stack", "heads", "gate", "ffn", "ffn", "ffn", "ffn"])
    if kind == "gate":
        groups = rng.choice([4, 8, 16])
        keep = rng.randint(max(1, groups // 4), groups)
        E = groups * rng.choice([8, 16, 24])
        return dict(kind=kind, T=_log_int(rng, 1, 4096), E=E, K=rng.randint(1, min(8, keep * E // groups)), groups=groups,
                    keep=keep, bias=rng.random() < 0.5)
    big = rng.random() < 0.7
    shape = dict(LARGE if big else SMALL)
    shape.update(K=rng.choice([1, 2, 4, 6, 8]) if big else rng.choice([1, 2, 4]),
                 E=rng.choice([64, 128, 160, 256]) if big else rng.choice([16, 32]),
                 group=rng.choice([32, 64, 128] if big else [32, 64]), rank=rng.choice([0, 8, 16]))
    case = dict(COMMON, kind=kind, out=rng.choice(["f32", "f32", "f16", "bf16"]), **shape)
    if kind == "steps":
        case.update(layers=rng.randint(1, 8), shared=rng.random() < 0.3,
                    per_expert_adapters=rng.random() < 0.3)
    elif kind == "chain":
        case.update(layers=8, steps=128, K=max(2, case["K"]))
    elif kind == "burst":
        case.update(layers=8, steps=128 * rng.randint(2, 10), K=rng.choice([2, 4, 8]) if big else 2)
    elif kind == "stack":
        streaming = rng.random() < 0.5
        case.update(layers=rng.randint(2, 4) if streaming else rng.randint(2, 12))
        case["slots"] = rng.choice([max(8, case["K"]), 24, 32]) if streaming and big else case["E"]
    elif kind == "heads":
        case.update(heads=rng.randint(1, 40), width=rng.choice([256, 512]), K=min(case["K"], 8))
    else:
        T = _log_int(rng, 2, 4096)
        case.update(T=T, layers=rng.randint(1, 4) if T < 16 else 1, router=rng.choice(["head", "zipf"]),
                    head=rng.choice(["f16", "f16", "f32"]), rank=rng.choice([0, 8, 16, 16, 32]),
                    per_expert_adapters=rng.random() < 0.25)
    return case


# ---------------------------------------------------------------- inputs

def _desc(c, slots=None):
    return edg.make_desc(None, H=c["H"], I=c["I"], E=c["E"], K=c["K"], group=c["group"], rank=c["rank"],
                         n_adapters=c["E"] if c.get("per_expert_adapters") else 1, n_slots=slots or c["E"],
                         pre_dtype=c["head"], lora_scale=2.0, out_dtype=c["out"])


def _records(c, desc, rng, count, gain=1.0):
    """`count` distinct experts, packed: uniform int4 codes, fp16 scales U(0.005, 0.02) * gain, integer zero points."""
    shapes = {"gate": (c["I"], c["H"]), "up": (c["I"], c["H"]), "down": (c["H"], c["I"])}
    out = np.empty((count, edg.record_bytes(desc)), np.uint8)
    for e in range(count):
        ex = {}
        for proj, (n, kd) in shapes.items():
            ng = kd // c["group"]
            ex[proj] = (rng.integers(0, 256, size=(n, kd // 2), dtype=np.uint8),
                        rng.uniform(0.005 * gain, 0.02 * gain, size=(n, ng)).astype(np.float16),
                        rng.integers(0, 16, size=(n, ng)).astype(np.float16))
        edg.pack_expert(desc, ex, out[e])
    return torch.from_numpy(out)


def _layer(records, E, pin):
    """The E records of a layer in host memory (distinct experts repeat beyond the first ones)."""
    host = torch.empty((E, records.shape[1]), dtype=torch.uint8, pin_memory=pin)
    for e0 in range(0, E, records.shape[0]):
        n = min(records.shape[0], E - e0)
        host[e0:e0 + n] = records[:n]
    return host


def _adapters(c, gen):
    """LoRA factors of one layer, A ~ N(0, 0.02), B ~ N(0, 0.01), bf16; None without an adapter."""
    if c["rank"] == 0:
        return None, []
    n, r, H, I = c["E"] if c.get("per_expert_adapters") else 1, c["rank"], c["H"], c["I"]

    def rnd(std, *shape):
        return (torch.randn(shape, generator=gen, device="cuda") * std).to(torch.bfloat16)
    t = [rnd(0.02, n, r, H), rnd(0.01, n, I, r), rnd(0.02, n, r, H), rnd(0.01, n, I, r), rnd(0.02, n, r, I), rnd(0.01, n, H, r)]
    return edg.make_lora(*t), t


def _heads(c, n, gen):
    w = torch.randn((n, c["E"], c["H"]), generator=gen, device="cuda") * 0.02
    return w.to(torch.float16) if c["head"] == "f16" else w


def _states(gen, *shape):
    return torch.randn(shape, generator=gen, device="cuda").to(torch.bfloat16)


def _out(c, *shape):
    return torch.zeros(shape, dtype={"f32": torch.float32, "f16": torch.float16, "bf16": torch.bfloat16}[c["out"]], device="cuda")


def _routing(*shape):
    return torch.zeros(shape, dtype=torch.int32, device="cuda"), torch.zeros(shape, dtype=torch.float32, device="cuda")


def _distinct(c):
    return min(c["E"], 48)


def _store(c, rng, gen, slots=None, gain=1.0):
    """A store of `layers` layers over one pinned host layer (layers may alias), resident when slots == E."""
    slots = slots or c["E"]
    desc = _desc(c, slots)
    host = _layer(_records(c, desc, rng, _distinct(c), gain), c["E"], pin=True)
    L = c["layers"]
    pool = torch.empty((L, slots, host.shape[1]), dtype=torch.uint8, device="cuda")
    tables = torch.empty((L, c["E"]), dtype=torch.int32, device="cuda")
    loras, keep = zip(*[_adapters(c, gen) for _ in range(L)])
    copies = torch.cuda.Stream()
    store = edg.Store(desc, [host] * L, pool, tables, list(loras) if c["rank"] else None, copies)
    if slots == c["E"]:
        for l in range(L):
            store.load_whole_layer(l)
            store.wait_staged(l)
    return desc, store, dict(host=host, pool=pool, tables=tables, keep=keep, copies=copies)


def prepare(case, seed):
    c = dict(case)
    rng = np.random.default_rng([int(seed), 17])
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed))
    return {"case": c, **globals()["_prepare_" + c["kind"]](c, rng, gen)}


def _prepare_steps(c, rng, gen):
    desc, store, keep = _store(c, rng, gen)
    L, K, H = c["layers"], c["K"], c["H"]
    s = dict(store=store, keep=keep, W=_heads(c, L, gen), X=_states(gen, L, H), Y=_out(c, L, H), ws=layer_io.new_workspace(desc))
    if c["shared"]:
        s["shared"] = _records(c, desc, rng, 1).cuda()
        for l in range(L):
            store.set_shared_expert(l, s["shared"][0])
    s["cur"], s["nxt"] = _routing(L, K), _routing(L, K)
    # the routing of this token, predicted from the token before it
    edg.prerouter_topk(desc, s["W"], _states(gen, L, H), L, *s["cur"])
    # a decoder keeps each layer's buffers: x, the routing it executes, its head, the routing it predicts, y
    (ci, cg), (ni, ng) = s["cur"], s["nxt"]
    s["calls"] = [(l, s["X"][l], ci[l], cg[l], s["W"][l], ni[(l + 1) % L], ng[(l + 1) % L], None, s["Y"][l], s["ws"])
                  for l in range(L)]
    return s


def _prepare_chain(c, rng, gen):
    # a layer adds a few per cent to the state it is given, as in a residual stream
    desc, store, keep = _store(c, rng, gen, gain=0.2)
    L, K, H, n = c["layers"], c["K"], c["H"], c["steps"]
    tokens = n // L
    W = _heads(c, L, gen)
    s = dict(store=store, keep=keep, W=W, x0=_states(gen, tokens, H), Y=_out(c, n, H), ws=layer_io.new_workspace(desc),
             xn=torch.zeros((n, H), dtype=torch.bfloat16, device="cuda"))
    s["first"], s["nxt"] = _routing(tokens, K), _routing(n, K)
    edg.prerouter_topk_tokens(desc, W[0], _states(gen, tokens, H), tokens, *s["first"])

    def step(i):
        l, t = i % L, i // L
        x = s["x0"][t] if l == 0 else s["xn"][i - 1]
        inds, gates = (s["first"][0][t], s["first"][1][t]) if l == 0 else (s["nxt"][0][i - 1], s["nxt"][1][i - 1])
        edg.moe_layer_decode_dependent(store, l, x, inds, gates, W[(l + 1) % L], s["nxt"][0][i], s["nxt"][1][i], None,
                                       s["Y"][i], s["xn"][i], s["ws"])
    s["graph"] = _capture(store, step, L, n)
    return s


def _prepare_burst(c, rng, gen):
    desc, store, keep = _store(c, rng, gen)
    L, K, H, n, NX = c["layers"], c["K"], c["H"], c["steps"], 64
    W = _heads(c, L, gen)
    s = dict(store=store, keep=keep, W=W, X=_states(gen, NX, H), Y=_out(c, NX, H), ws=layer_io.new_workspace(desc))
    s["inds"], s["gates"] = _routing(n + 1, K)
    edg.prerouter_topk(desc, W[0], _states(gen, 1, H), 1, s["inds"][0], s["gates"][0])

    def step(i):
        edg.moe_layer_decode(store, i % L, s["X"][i % NX], s["inds"][i], s["gates"][i], W[(i + 1) % L], s["inds"][i + 1],
                             s["gates"][i + 1], None, s["Y"][i % NX], s["ws"])
    s["graph"] = _capture(store, step, L, n)
    return s


def _capture(store, step, L, n):
    """The n chained steps as one graph (a multiple of 128, as the hand-off ring asks); every layer runs once before it."""
    for i in range(L):
        step(i)
    torch.cuda.synchronize()
    store.set_chaining(1)
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        for i in range(n):
            step(i)
    return g


def _prepare_stack(c, rng, gen):
    desc, store, keep = _store(c, rng, gen, slots=c["slots"])
    L, H, NX = c["layers"], c["H"], 16
    # consecutive tokens agree on part of their routing, as decode traces do
    X = torch.empty((NX, L, H), device="cuda")
    X[0] = torch.randn((L, H), generator=gen, device="cuda")
    for t in range(1, NX):
        X[t] = 0.6 * X[t - 1] + 0.8 * torch.randn((L, H), generator=gen, device="cuda")
    X = X.to(torch.bfloat16)
    dec = StackDecoder(desc, store, _heads(c, L, gen), prefetch=True)
    dec.prime(X[NX - 1])
    return dict(store=store, keep=keep, dec=dec, X=list(X), Y=_out(c, L, H), t=0)


def _prepare_ffn(c, rng, gen):
    desc = _desc(c)
    records = _records(c, desc, rng, _distinct(c)).cuda()
    order = torch.arange(c["E"], device="cuda") % records.shape[0]
    T, K, L = c["T"], c["K"], c["layers"]
    pool = torch.stack([records[order] for _ in range(L)])
    s = dict(desc=desc, pool=pool, table=torch.arange(c["E"], dtype=torch.int32, device="cuda"), X=_states(gen, L, T, c["H"]),
             Y=_out(c, L, T, c["H"]), ws=layer_io.new_workspace(desc, T), loras=[_adapters(c, gen) for _ in range(L)])
    s["inds"], s["gates"] = _routing(L, T, K)
    if c["router"] == "head":
        s["W"] = _heads(c, L, gen)
    else:
        rank = torch.argsort(torch.rand((L, 1, c["E"]), generator=gen, device="cuda"), dim=-1).float() + 1
        gumbel = -torch.log(-torch.log(torch.rand((L, T, c["E"]), generator=gen, device="cuda").clamp(1e-9, 1 - 1e-7)))
        s["logits"] = (-1.1 * torch.log(rank) + gumbel).contiguous()
    s["layers"] = [(s["inds"][l], s["gates"][l], s["X"][l], s["W" if c["router"] == "head" else "logits"][l], pool[l],
                    s["loras"][l][0], s["Y"][l]) for l in range(L)]
    return s


def _prepare_heads(c, rng, gen):
    desc = _desc(c)
    n, D, E, H, K = c["heads"], c["width"], c["E"], c["H"], c["K"]

    def rnd(std, *shape):
        return (torch.randn(shape, generator=gen, device="cuda") * std).to(torch.float16)

    def some():
        return torch.argsort(torch.rand((n, E), generator=gen, device="cuda"), dim=-1)[:, :K].to(torch.int32).sort(-1).values.contiguous()
    s = dict(desc=desc, W1=rnd(0.02, n, D, H + 2 * E), b1=rnd(0.01, n, D), W2=rnd(0.02, n, E, D), b2=rnd(0.01, n, E),
             W_res=_heads(c, n, gen), x=_states(gen, n, H), cur=some(), prev=some())
    s["inds"], s["gates"] = _routing(n, K)
    s["logits"] = torch.zeros((n, E), device="cuda")
    return s


def _prepare_gate(c, rng, gen):
    s = dict(logits=torch.randn((c["T"], c["E"]), generator=gen, device="cuda"),
             bias=torch.randn((c["E"],), generator=gen, device="cuda") * 0.05 if c["bias"] else None)
    s["inds"], s["gates"] = _routing(c["T"], c["K"])
    return s


# ---------------------------------------------------------------- one pass

def run(state):
    return globals()["_run_" + state["case"]["kind"]](state, state["case"])


def _run_steps(s, c):
    for call in s["calls"]:
        edg.moe_layer_decode(s["store"], *call)
    return s["Y"], s["nxt"][0], s["nxt"][1]


def _run_chain(s, c):
    s["graph"].replay()
    return s["Y"], s["xn"], s["nxt"][0], s["nxt"][1]


def _run_burst(s, c):
    s["graph"].replay()
    return s["Y"], s["inds"], s["gates"]


def _run_stack(s, c):
    t = s["t"]
    s["dec"].step(t, s["X"][t % len(s["X"])], s["Y"])
    s["t"] = t + 1
    return s["Y"], s["dec"].inds[(t + 1) % 2], s["dec"].gates[(t + 1) % 2]


def _run_ffn(s, c):
    T, head = c["T"], c["router"] == "head"
    for inds, gates, x, router, pool, lora, y in s["layers"]:
        if head:
            edg.prerouter_topk_tokens(s["desc"], router, x, T, inds, gates)
        else:
            edg.softmax_topk_rows(s["desc"], router, T, inds, gates)
        edg.moe_expert_ffn_int4_lora(s["desc"], pool, s["table"], T, inds, None, gates, x, lora, y, s["ws"])
    return s["Y"], s["inds"], s["gates"]


def _run_heads(s, c):
    edg.prerouter_mlp_topk(s["desc"], s["W1"], s["b1"], s["W2"], s["b2"], s["W_res"], c["width"], s["x"], s["cur"], s["prev"],
                           c["heads"], s["inds"], s["gates"], s["logits"])
    return s["inds"], s["gates"], s["logits"]


def _run_gate(s, c):
    edg.sigmoid_group_topk_rows(s["logits"], c["T"], c["E"], c["K"], c["groups"], c["keep"], 2.5, s["bias"], s["inds"], s["gates"])
    return s["inds"], s["gates"]


# ---------------------------------------------------------------- what a pass cannot do without

def work(case):
    c = case
    if c["kind"] == "gate":
        return {"bytes": c["T"] * (4 * c["E"] + 8 * c["K"]), "flops": 4 * c["T"] * c["E"]}
    H, I, E, K, r = c["H"], c["I"], c["E"], c["K"], c["rank"]
    hb, ob = (2 if c["head"] == "f16" else 4), (4 if c["out"] == "f32" else 2)
    if c["kind"] == "heads":
        D = c["width"]
        per = 2 * D * (H + 2 * K) + 2 * E * D + hb * E * H + 2 * (D + E) + 2 * H + 4 * E + 16 * K
        return {"bytes": c["heads"] * per, "flops": c["heads"] * 2 * (D * (H + 2 * K) + E * D + E * H)}
    record = 3 * H * I // 2 + 3 * (H * I // c["group"]) * 4
    one_adapter = 2 * r * (3 * H + 3 * I)
    pair_flops = 6 * H * I + 2 * r * (3 * H + 3 * I)
    if c["kind"] == "ffn":
        T, L = c["T"], c["layers"]
        if c["router"] == "head":
            p = np.full(E, 1 / E)
            route_bytes, route_flops = hb * E * H, 2 * T * E * H
        else:
            p = np.arange(1, E + 1, dtype=np.float64) ** -1.1
            p /= p.sum()
            route_bytes, route_flops = 4 * T * E, 0
        touched = float((1 - (1 - np.minimum(1.0, K * p)) ** T).sum())       # experts that some token is routed to
        adapters = touched if c["per_expert_adapters"] else 1
        return {"bytes": L * (touched * record + adapters * one_adapter + route_bytes + T * H * (2 + ob) + 8 * T * K),
                "flops": L * (T * K * pair_flops + route_flops)}
    n = c["steps"] if c["kind"] in ("chain", "burst") else c["layers"]
    experts = K + (1 if c.get("shared") else 0)
    adapters = K if c.get("per_expert_adapters") else 1
    per = experts * record + adapters * one_adapter + hb * E * H + H * (2 + ob) + 16 * K + (2 * H if c["kind"] == "chain" else 0)
    return {"bytes": n * per, "flops": n * (experts * pair_flops + 2 * E * H)}


def tolerance(case):
    """About four times what the path differs by from its fp64 evaluation (measured on a B200: fp32 outputs 4e-5 relative,
    the adapter's fp16 operands and the order of fp32 sums; bf16 outputs 1.7e-3, their rounding), and the share of expert
    indices that near-ties may move."""
    c = case
    if c["kind"] in ("gate", "heads"):
        return {"rel": 1e-5, "max": 1e-4, "differ": 1e-4}
    if c["kind"] == "chain":
        # the state is rounded to bf16 after every layer: a rounding that falls the other way is carried on
        return {"rel": 1e-2, "max": 0.5, "differ": 5e-3}
    rel, most = {"f32": (1.5e-4, 8e-4), "f16": (6e-4, 3e-3), "bf16": (6e-3, 2e-2)}[c["out"]]
    return {"rel": rel, "max": most, "differ": 1e-3}
