"""The latency form of the layer-step -- alone, and as a link of a chain of dependent steps -- where it can go wrong: both widths of
the state and of the experts, every scale group, no adapter / the smallest / the largest rank, one expert and the most it
takes (more CTAs than SMs), adapters per expert, a shared expert, heads of whole and of broken tiles; and several chains at once on
streams of their own, whose launches find the SMs taken.  Each step against the oracle on the state the GPU itself handed on; bars
as everywhere."""
import dataclasses

import numpy as np
import pytest
import torch

import paper_2609_18063_b200 as edg
from oracle import moe_oracle as orc
from paper_2609_18063_b200 import layer_io
from workloads import synth

from _gpu_util import x_dev
from test_gpu_parity import _assert_close, _check_routing, _make_store

pytestmark = pytest.mark.gpu

SHARED_ID = 1000


class _Chain:
    """`steps` dependent layer-steps of one layer: buffers, and the calls"""

    def __init__(self, cfg, steps, shared, seed):
        self.store, self.d, _, _, self.tables, self.cs, self.keep = _make_store(cfg, n_slots=cfg.E)
        for e0 in range(0, cfg.E, 32):
            edg.stage_experts_to_slots(self.store, 0, np.arange(e0, min(cfg.E, e0 + 32), dtype=np.int32))
        self.shared = synth.expert_tensors(cfg, 0, SHARED_ID) if shared else None
        self.slo = synth.lora_tensors(cfg, 0, SHARED_ID) if shared and cfg.rank else None
        if shared:
            self.rec = torch.from_numpy(edg.pack_expert(self.d, self.shared)).cuda()
            lo, self.keep2 = layer_io.lora_to_device(edg.make_desc(cfg, n_adapters=1), [self.slo]) if cfg.rank else (None, None)
            self.store.set_shared_expert(0, self.rec, lo)
        self.W_np = synth.prerouter_weights(cfg)
        self.W = torch.from_numpy(self.W_np).cuda()
        x0 = synth.hidden_states(cfg, 2, stream=seed)
        self.xs = torch.zeros((steps + 1, cfg.H), dtype=torch.bfloat16, device="cuda")
        self.xs[0] = x_dev(x0[0])
        self.inds = torch.zeros((steps + 1, cfg.K), dtype=torch.int32, device="cuda")
        self.gates = torch.zeros((steps + 1, cfg.K), dtype=torch.float32, device="cuda")
        self.logits = torch.zeros((steps + 1, cfg.E), dtype=torch.float32, device="cuda")
        self.y = torch.zeros((steps, cfg.H), dtype=torch.float32, device="cuda")
        self.ws = layer_io.new_workspace(self.d)
        self.cfg, self.steps = cfg, steps
        edg.prerouter_topk(self.d, self.W, x_dev(x0[1]), 1, self.inds[0], self.gates[0], self.logits[0])
        self.store.set_chaining(2)
        torch.cuda.synchronize()

    def run(self, t):
        edg.moe_layer_decode_dependent(self.store, 0, self.xs[t], self.inds[t], self.gates[t], self.W, self.inds[t + 1], self.gates[t + 1],
                                       self.logits[t + 1], self.y[t], self.xs[t + 1], self.ws)

    def result(self):
        assert edg.workspace_status(self.ws) == 0
        return [a.clone() for a in (self.xs, self.inds, self.gates, self.logits, self.y)]


def _cfg(H, I, group, E, K, rank, n_adapters):
    return dataclasses.replace(synth.CONFIGS["cfg1"], name=f"H{H}I{I}g{group}E{E}K{K}r{rank}a{n_adapters}", H=H, I=I, group=group, E=E, K=K,
                               rank=rank, n_adapters=n_adapters, n_slots=E, seed=29)


@pytest.mark.parametrize("H,I,group,E,K,rank,n_adapters,shared", [
    (1024, 256, 32, 16, 1, 0, 1, False),     # the smallest: 16 CTAs of gate/up work, 64 of down work
    (1024, 512, 128, 40, 4, 24, 1, False),   # a head of 40 rows: a broken tile; a rank that is no power of two
    (2048, 256, 64, 24, 2, 64, 24, False),   # the largest rank, adapters per expert
    (2048, 512, 32, 32, 6, 8, 1, True),      # the smallest groups, a shared expert
    (2048, 512, 64, 96, 8, 16, 1, True),     # 144 expert CTAs: six head tiles share four CTAs
    (1024, 256, 64, 32, 16, 8, 32, False),   # the most experts: more CTAs than SMs, two passes over h
])
def test_alone_and_as_a_link_of_a_chain(H, I, group, E, K, rank, n_adapters, shared):
    cfg, steps = _cfg(H, I, group, E, K, rank, n_adapters), 5
    c = _Chain(cfg, steps, shared, 67)
    for t in range(steps):
        c.run(t)
    torch.cuda.synchronize()
    xs, inds, gates, logits, y = [a.cpu().numpy() if a.dtype != torch.bfloat16 else a.view(torch.int16).cpu().numpy().view(np.uint16)
                                  for a in c.result()]
    # the same states once more, each step alone
    alone = torch.zeros_like(c.y)
    c.store.set_chaining(0)
    for t in range(steps):
        edg.moe_layer_decode(c.store, 0, c.xs[t], c.inds[t], c.gates[t], c.W, torch.zeros_like(c.inds[0]), torch.zeros_like(c.gates[0]), None,
                             alone[t], c.ws)
    torch.cuda.synchronize()
    assert edg.workspace_status(c.ws) == 0
    experts = {}
    get = lambda e: experts.setdefault(e, synth.expert_tensors(cfg, 0, e))
    lora = (lambda e: synth.lora_tensors(cfg, 0, e if n_adapters > 1 else 0)) if rank else None
    for t in range(steps):
        g = gates[t].astype(np.float64)
        ref = (orc.moe_ffn_with_shared(xs[t], inds[t], g, get, lora, c.shared, c.slo, cfg.lora_scale, cfg.group) if shared else
               orc.moe_ffn(xs[t], inds[t], g, get, lora, cfg.lora_scale, cfg.group))
        _assert_close(y[t], ref)
        _assert_close(alone[t].cpu().numpy(), ref)
        _check_routing(logits[t + 1], inds[t + 1], gates[t + 1], c.W_np.astype(np.float32), xs[t], K)
        nxt = orc.next_hidden_state(xs[t], y[t].astype(np.float64), 1e-6)
        # one bf16 step: the norm is summed in fp32
        key = lambda b: np.where(b.astype(np.int32) & 0x8000, -(b.astype(np.int32) & 0x7FFF), b.astype(np.int32))
        assert np.abs(key(np.asarray(nxt)) - key(xs[t + 1])).max() <= 1
    c.store.close()


def test_chains_on_streams_of_their_own():
    """Four chains at once: their launches together want four times the CTAs that fit, so some wait for SMs while others, partly
    resident, wait for them.  Every result is the one the chain gives when it has the GPU to itself, bit for bit."""
    cfg, steps = _cfg(2048, 512, 64, 32, 8, 16, 1), 96
    chains = [_Chain(cfg, steps, False, 71 + i) for i in range(4)]
    want = []
    for c in chains:
        for t in range(steps):
            c.run(t)
        torch.cuda.synchronize()
        want.append(c.result())
    streams = [torch.cuda.Stream() for _ in chains]
    for rep in range(3):
        for c, w in zip(chains, want):
            for a in (c.xs[1:], c.inds[1:], c.gates[1:], c.logits[1:], c.y):
                a.zero_()
        torch.cuda.synchronize()
        for t in range(steps):
            for c, st in zip(chains, streams):
                with torch.cuda.stream(st):
                    c.run(t)
        torch.cuda.synchronize()
        for c, w in zip(chains, want):
            for a, b in zip(c.result(), w):
                assert torch.equal(a, b)
    for c in chains:
        c.store.close()


@pytest.mark.parametrize("E,then", [(256, "dependent"), (1024, "dependent"), (256, "throughput"), (1024, "throughput")])
def test_the_logits_a_link_hands_on(E, then):
    """150 chained links -- the hand-off ring wraps -- of a layer with the most experts there can be: the logits every link leaves, with the
    next one under way on the routing made of them; and steps chained through the routing alone behind one that runs by itself."""
    cfg, steps, n = dataclasses.replace(_cfg(1024, 256, 64, E, 8, 8, 1), pre_dtype="f16"), 150, 8
    d = edg.make_desc(cfg, n_slots=E)
    some = torch.from_numpy(np.stack([edg.pack_expert(d, synth.expert_tensors(cfg, 0, e)) for e in range(n)]))
    host = some[torch.arange(E) % n].contiguous().pin_memory()
    pool, tables = torch.empty((1, E, host.shape[1]), dtype=torch.uint8, device="cuda"), torch.empty((1, E), dtype=torch.int32, device="cuda")
    lora, keep = layer_io.lora_to_device(d, [synth.lora_tensors(cfg, 0, 0)])
    store = edg.Store(d, [host], pool, tables, [lora], torch.cuda.Stream())
    store.load_whole_layer(0)
    W_np = synth.prerouter_weights(cfg)
    W, ws = torch.from_numpy(W_np).cuda(), layer_io.new_workspace(d)
    X = synth.hidden_states(cfg, steps + 1, stream=83)
    xs = x_dev(X)
    inds, gates = torch.zeros((steps + 1, 8), dtype=torch.int32, device="cuda"), torch.zeros((steps + 1, 8), device="cuda")
    logits, y = torch.full((steps + 1, E), float("nan"), device="cuda"), torch.zeros((steps, cfg.H), device="cuda")
    edg.prerouter_topk(d, W, xs[steps], 1, inds[0], gates[0], logits[0])
    store.set_chaining(2)
    for t in range(steps):
        if then == "dependent":
            edg.moe_layer_decode_dependent(store, 0, xs[t], inds[t], gates[t], W, inds[t + 1], gates[t + 1], logits[t + 1], y[t], xs[t + 1], ws)
        else:
            edg.moe_layer_decode(store, 0, xs[t], inds[t], gates[t], W, inds[t + 1], gates[t + 1], logits[t + 1], y[t], ws)
    assert edg.workspace_status(ws) == 0
    bits, lh, ih, gh = xs.view(torch.int16).cpu().numpy().view(np.uint16), logits.cpu().numpy(), inds.cpu().numpy(), gates.cpu().numpy()
    for t in range(steps):
        _check_routing(lh[t + 1], ih[t + 1], gh[t + 1], W_np.astype(np.float32), bits[t], 8)
    for t in range(0, steps, 29):
        _assert_close(y[t].cpu().numpy(), orc.moe_ffn(bits[t], ih[t], gh[t].astype(np.float64), lambda e: synth.expert_tensors(cfg, 0, e % n),
                                                      lambda e: synth.lora_tensors(cfg, 0, 0), cfg.lora_scale, cfg.group))
    store.close()


def test_traced_steps_run_in_the_throughput_form():
    """With a trace buffer set, lone steps (head CTAs of their own behind those of the experts) and dependent chains (norm and state handed on
    by the reducers) of shapes that otherwise take the latency form: right results, and a stamp of every expert CTA's end."""
    cfg, steps = _cfg(2048, 512, 64, 64, 8, 16, 1), 4
    cfg = dataclasses.replace(cfg, pre_dtype="f16")
    c = _Chain(cfg, steps, False, 91)
    n_ctas = 16 * (cfg.K + 1) + cfg.E // 16 + 3
    trace = torch.zeros((n_ctas, 32), dtype=torch.int64, device="cuda")
    alone = torch.zeros_like(c.y)
    edg.set_trace_buffer(trace)
    try:
        for t in range(steps):
            c.run(t)
        torch.cuda.synchronize()
        ends = int((trace[:, 9] > 0).sum())
        xs, inds, gates, logits, y = [a.cpu().numpy() if a.dtype != torch.bfloat16 else a.view(torch.int16).cpu().numpy().view(np.uint16)
                                      for a in c.result()]
        c.store.set_chaining(0)
        for t in range(steps):
            edg.moe_layer_decode(c.store, 0, c.xs[t], c.inds[t], c.gates[t], c.W, torch.zeros_like(c.inds[0]), torch.zeros_like(c.gates[0]), None,
                                 alone[t], c.ws)
        torch.cuda.synchronize()
    finally:
        edg.set_trace_buffer(None)
    assert ends >= 16 * cfg.K and edg.workspace_status(c.ws) == 0
    experts = {}
    for t in range(steps):
        ref = orc.moe_ffn(xs[t], inds[t], gates[t].astype(np.float64), lambda e: experts.setdefault(e, synth.expert_tensors(cfg, 0, e)),
                          lambda e: synth.lora_tensors(cfg, 0, 0), cfg.lora_scale, cfg.group)
        _assert_close(y[t], ref)
        _assert_close(alone[t].cpu().numpy(), ref)
        _check_routing(logits[t + 1], inds[t + 1], gates[t + 1], c.W_np.astype(np.float32), xs[t], cfg.K)
    c.store.close()
