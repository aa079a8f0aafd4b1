"""A workspace is scratch: only its control block lasts from call to call.  Layer-steps -- with a head of their own, without one, with
a full head, dependent ones, in a chain -- before and after whatever else may have used the memory: a prompt of the same layer, steps of
a layer of another shape and store, a new owner that has zeroed it or left anything behind the control block.  Every output against the
oracle (bars as everywhere), and no status raised."""
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

SMALL = dataclasses.replace(synth.CONFIGS["cfg1"], name="ws_small", n_slots=16, seed=31)
WIDE = dataclasses.replace(synth.CONFIGS["cfg2"], name="ws_wide", E=32, n_slots=32, seed=32)
MANY = dataclasses.replace(synth.CONFIGS["cfg1"], name="ws_many", E=32, K=24, group=64, n_slots=32, seed=33)   # beyond the latency form
PROMPT = {"ws_small": 800, "ws_wide": 390, "ws_many": 140}       # tokens of a prompt that takes the 128-token tiles (over 96 pairs a slot)


class _Layer:
    def __init__(self, cfg):
        self.cfg = cfg
        self.store, self.d, _, self.slots, self.tables, _, self.keep = _make_store(cfg, n_slots=cfg.E)
        self.lora = layer_io.lora_to_device(self.d, [synth.lora_tensors(cfg, 0, 0)])
        edg.stage_experts_to_slots(self.store, 0, np.arange(cfg.E, dtype=np.int32))
        self.W_np = synth.prerouter_weights(cfg)
        self.W = torch.from_numpy(self.W_np).cuda()
        self.X = synth.hidden_states(cfg, 8, stream=41)
        self.xd = x_dev(self.X)
        self.inds, self.gates = torch.zeros((8, cfg.K), dtype=torch.int32, device="cuda"), torch.zeros((8, cfg.K), device="cuda")
        edg.prerouter_topk_tokens(self.d, self.W, self.xd, 8, self.inds, self.gates)
        torch.cuda.synchronize()
        self.experts, self.t = {}, 0

    def expert(self, e):
        return self.experts.setdefault(e, synth.expert_tensors(self.cfg, 0, e))

    def check(self, y, x_bits, inds, gates):
        lora = synth.lora_tensors(self.cfg, 0, 0)
        _assert_close(y.cpu().numpy(), orc.moe_ffn(x_bits, inds, gates.astype(np.float64), self.expert, lambda e: lora, self.cfg.lora_scale, self.cfg.group))

    def step(self, ws, head=True, dependent=False):
        """one layer-step on the next state; checked"""
        t, K = self.t % 8, self.cfg.K
        self.t += 1
        y = torch.full((self.cfg.H,), float("nan"), device="cuda")
        inds, gates, logits = torch.full((K,), -1, dtype=torch.int32, device="cuda"), torch.zeros(K, device="cuda"), torch.zeros(self.cfg.E, device="cuda")
        args = (self.store, 0, self.xd[t], self.inds[t], self.gates[t]) + ((self.W, inds, gates, logits) if head else (None,) * 4)
        if dependent:
            xn = torch.zeros(self.cfg.H, dtype=torch.bfloat16, device="cuda")
            edg.moe_layer_decode_dependent(*args, y, xn, ws)
        else:
            edg.moe_layer_decode(*args, y, ws)
        assert edg.workspace_status(ws) == 0
        self.check(y, self.X[t], self.inds[t].cpu().numpy(), self.gates[t].cpu().numpy())
        if head:
            _check_routing(logits.cpu().numpy(), inds.cpu().numpy(), gates.cpu().numpy(), self.W_np.astype(np.float32), self.X[t], K)
        if dependent:
            want = orc.bf16_to_f64(orc.next_hidden_state(self.X[t], y.cpu().numpy().astype(np.float64), 1e-6))
            assert np.abs(xn.float().cpu().numpy() - want).max() <= 2.0 ** -7 * np.abs(want).max()      # a bf16 step at the largest value

    def chain(self, ws, n=5, leave_on=False):
        """n dependent steps, chained; each checked on the state the GPU handed on"""
        K = self.cfg.K
        xs = torch.zeros((n + 1, self.cfg.H), dtype=torch.bfloat16, device="cuda")
        xs[0] = self.xd[0]
        inds, gates = torch.zeros((n + 1, K), dtype=torch.int32, device="cuda"), torch.zeros((n + 1, K), device="cuda")
        inds[0], gates[0] = self.inds[0], self.gates[0]
        logits, y = torch.zeros((n + 1, self.cfg.E), device="cuda"), torch.zeros((n, self.cfg.H), device="cuda")
        self.store.set_chaining(2)
        for t in range(n):
            edg.moe_layer_decode_dependent(self.store, 0, xs[t], inds[t], gates[t], self.W, inds[t + 1], gates[t + 1], logits[t + 1], y[t], xs[t + 1], ws)
        assert edg.workspace_status(ws) == 0
        if not leave_on:
            self.store.set_chaining(0)
        bits = xs.view(torch.int16).cpu().numpy().view(np.uint16)
        for t in range(n):
            self.check(y[t], bits[t], inds[t].cpu().numpy(), gates[t].cpu().numpy())
            _check_routing(logits[t + 1].cpu().numpy(), inds[t + 1].cpu().numpy(), gates[t + 1].cpu().numpy(), self.W_np.astype(np.float32), bits[t], K)

    def prompt(self, ws, T):
        X = synth.hidden_states(self.cfg, T, stream=43)
        xd, K = x_dev(X), self.cfg.K
        inds, gates = torch.zeros((T, K), dtype=torch.int32, device="cuda"), torch.zeros((T, K), device="cuda")
        edg.prerouter_topk_tokens(self.d, self.W, xd, T, inds, gates)
        y = torch.zeros((T, self.cfg.H), device="cuda")
        edg.moe_expert_ffn_int4_lora(self.d, self.slots[0], self.tables[0], T, inds, None, gates, xd, self.lora[0], y, ws)
        assert edg.workspace_status(ws) == 0
        for t in (0, T - 1):
            self.check(y[t], X[t], inds[t].cpu().numpy(), gates[t].cpu().numpy())


@pytest.fixture(scope="module")
def layers():
    made = {}

    def get(cfg):
        if cfg.name not in made:
            made[cfg.name] = _Layer(cfg)
        return made[cfg.name]
    yield get
    for l in made.values():
        l.store.close()


@pytest.mark.parametrize("cfg", [SMALL, WIDE, MANY], ids=lambda c: c.name)
def test_steps_around_a_prompt_in_one_workspace(layers, cfg):
    L, T = layers(cfg), PROMPT[cfg.name]
    ws = layer_io.new_workspace(L.d, T)
    for tokens in (T, 3):                       # the 128-token tiles, the streaming form
        for head in (True, False):
            L.step(ws, head)
            L.prompt(ws, tokens)
            L.step(ws, head)
        L.step(ws, dependent=True)
        L.prompt(ws, tokens)
        L.step(ws, dependent=True)
        L.chain(ws)


@pytest.mark.parametrize("cfg", [SMALL, WIDE, MANY], ids=lambda c: c.name)
def test_a_workspace_that_changes_hands_at_the_same_address(layers, cfg):
    L = layers(cfg)
    ws = layer_io.new_workspace(L.d)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(3)
    for fill in ("zeros", "anything", "zeros"):
        L.step(ws)
        L.step(ws, head=False)
        L.chain(ws)
        if fill == "zeros":
            ws.zero_()
        else:                                   # (the control block is zeroed, as before any first use)
            ws.view(torch.int32).random_(-2 ** 31, 2 ** 31 - 1, generator=gen)
            ws[:4096] = 0
        L.step(ws, head=False)
        L.step(ws)
        L.step(ws, dependent=True)
        L.chain(ws)


@pytest.mark.parametrize("cfg", [SMALL, WIDE, MANY], ids=lambda c: c.name)
def test_chains_with_anything_else_in_the_workspace_between_them(layers, cfg):
    """Chaining stays on: what a chain before it left in the hand-off ring, or another use of the workspace, is nothing to the next one."""
    L = layers(cfg)
    ws = layer_io.new_workspace(L.d)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(4)
    L.chain(ws, leave_on=True)
    for _ in range(2):
        ws[4096:].view(torch.int32).random_(-2 ** 31, 2 ** 31 - 1, generator=gen)
        L.chain(ws, leave_on=True)
    for head in (True, False, True):            # steps whose routing nobody takes from the ring
        L.step(ws, head)
    L.chain(ws)


def test_two_stores_of_different_shapes_in_one_workspace(layers):
    a, b, c = layers(SMALL), layers(WIDE), layers(MANY)
    ws = torch.zeros(max(edg.ffn_workspace_bytes(l.d) for l in (a, b, c)), dtype=torch.uint8, device="cuda")
    for head in (True, False, True):
        for l in (a, b, c, b, a, c):
            l.step(ws, head)
            l.step(ws, dependent=True)
    for l in (a, b, c, a):
        l.chain(ws)
        b.step(ws)


def test_a_layer_with_a_full_head_around_a_prompt(layers):
    L, T = layers(SMALL), PROMPT["ws_small"]
    cfg, rng = L.cfg, np.random.default_rng(9)
    W1, W2 = (rng.standard_normal((64, cfg.H + 2 * cfg.E)) * 0.02).astype(np.float16), (rng.standard_normal((cfg.E, 64)) * 0.02).astype(np.float16)
    dev = [torch.from_numpy(w).cuda() for w in (W1, W2)]
    L.store.set_mlp_head(0, dev[0], None, dev[1], None, None, 64)
    ws = layer_io.new_workspace(L.d, T)
    y, inds, gates = torch.zeros(cfg.H, device="cuda"), torch.zeros(cfg.K, dtype=torch.int32, device="cuda"), torch.zeros(cfg.K, device="cuda")
    for t in range(3):
        edg.moe_layer_decode(L.store, 0, L.xd[t], L.inds[t], L.gates[t], None, inds, gates, None, y, ws)
        assert edg.workspace_status(ws) == 0
        L.check(y, L.X[t], L.inds[t].cpu().numpy(), L.gates[t].cpu().numpy())
        L.prompt(ws, T)
    L.store.set_mlp_head(0)


@pytest.mark.parametrize("cfg", [SMALL, WIDE, MANY], ids=lambda c: c.name)
def test_captured_steps_replayed_without_chaining(layers, cfg):
    """Steps with a head of their own in a CUDA graph, chaining off: a replay starts on what the replay before it left in the workspace."""
    L, K = layers(cfg), cfg.K
    ws = layer_io.new_workspace(L.d)
    y = torch.zeros((3, cfg.H), device="cuda")
    inds, gates, logits = torch.zeros((3, K), dtype=torch.int32, device="cuda"), torch.zeros((3, K), device="cuda"), torch.zeros((3, cfg.E), device="cuda")

    def steps():
        for t in range(3):
            edg.moe_layer_decode(L.store, 0, L.xd[t], L.inds[t], L.gates[t], L.W, inds[t], gates[t], logits[t], y[t], ws)
    steps()
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        steps()
    for _ in range(3):
        for a in (y, inds, gates, logits):
            a.zero_()
        g.replay()
        assert edg.workspace_status(ws) == 0
        for t in range(3):
            L.check(y[t], L.X[t], L.inds[t].cpu().numpy(), L.gates[t].cpu().numpy())
            _check_routing(logits[t].cpu().numpy(), inds[t].cpu().numpy(), gates[t].cpu().numpy(), L.W_np.astype(np.float32), L.X[t], K)
