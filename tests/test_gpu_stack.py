"""Config-3-shaped decode through the expert stack (small: 3 layers, 5 tokens): prediction-driven
staging across layers, every layer-step checked against the oracle on the same inputs."""
import numpy as np
import pytest
import torch

import paper_2609_18063_b200 as edg
from oracle import moe_oracle as orc
from paper_2609_18063_b200 import layer_io
from paper_2609_18063_b200.decoder import StackDecoder
from workloads import synth

from _gpu_util import TOL_MAX_ABS, TOL_REL_L2

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_slots,prefetch", [(8, True), (16, True), (8, False)])
def test_stack_decode_matches_oracle(n_slots, prefetch):
    cfg = synth.CONFIGS["cfg3"].with_(n_layers=3)
    L, T, K, E = cfg.n_layers, 5, cfg.K, cfg.E
    d = edg.make_desc(cfg, n_slots=n_slots)
    R = edg.record_bytes(d)
    experts = {}
    get = lambda l, e: experts.setdefault((l, e), synth.expert_tensors(cfg, l, e))
    hosts = [layer_io.host_layer(d, lambda e, l=l: get(l, e)) for l in range(L)]
    loras_np = [synth.lora_tensors(cfg, l, 0) for l in range(L)]
    loras, keep = zip(*[layer_io.lora_to_device(d, [ln]) for ln in loras_np])
    slots = torch.zeros((L, n_slots, R), dtype=torch.uint8, device="cuda")
    tables = torch.zeros((L, E), dtype=torch.int32, device="cuda")
    store = edg.Store(d, hosts, slots, tables, list(loras), torch.cuda.Stream())
    W_np = np.stack([synth.prerouter_weights(cfg, l) for l in range(L)])
    W = torch.from_numpy(W_np).cuda()
    X_np = np.stack([synth.hidden_states(cfg, T + 1, layer=l, stream=21) for l in range(L)])   # [L][T+1][H]
    X = layer_io.bits_to_device(X_np, torch.bfloat16)
    dec = StackDecoder(d, store, W, prefetch=prefetch)
    dec.prime(X[:, T].contiguous())
    Y = torch.zeros((T, L, cfg.H), dtype=torch.float32, device="cuda")
    logits = torch.zeros((T, L, E), dtype=torch.float32, device="cuda")
    allocs = [orc.SlotAllocator(E, n_slots) for _ in range(L)]
    routing = []
    for t in range(T):
        dec.step(t, X[:, t].contiguous(), Y[t], logits[t])
        torch.cuda.synchronize()
        routing.append((dec.inds[t % 2].cpu().numpy().copy(), dec.gates[t % 2].cpu().numpy().copy()))
    assert edg.workspace_status(dec.ws) == 0
    Yh, lg = Y.cpu().numpy(), logits.cpu().numpy()
    want_miss = 0
    for t in range(T):
        inds_t, gates_t = routing[t]
        for l in range(L):
            want_miss += len(allocs[l].stage(inds_t[l].tolist())[1])
            ref = orc.moe_ffn(X_np[l, t], inds_t[l], gates_t[l].astype(np.float64), lambda e, l=l: get(l, e),
                              lambda e, l=l: loras_np[l], cfg.lora_scale, cfg.group)
            assert orc.max_abs(Yh[t, l], ref) <= TOL_MAX_ABS and orc.rel_l2(Yh[t, l], ref) <= TOL_REL_L2
            # the head owned by layer l predicted layer (l+1) % L of the next token
            ln = (l + 1) % L
            l_ref = orc.prerouter_logits(W_np[l], X_np[l, t])
            assert np.abs(lg[t, ln] - l_ref).max() <= 1e-5
            if t + 1 < T:
                i_ref, _ = orc.softmax_topk(l_ref, K)
                srt = np.sort(l_ref)[::-1]
                if srt[K - 1] - srt[K] > 1e-4:
                    assert routing[t + 1][0][ln].tolist() == i_ref.tolist()
    assert dec.misses == want_miss == store.stats()["misses"]
    for l in range(L):
        eos, soe = store.snapshot(l)
        assert eos.tolist() == allocs[l].expert_of_slot and soe.tolist() == allocs[l].slot_of_expert
    store.close()


def _resident_stack(cfg, n_layers, stream):
    """A store of resident layers, its decoder's heads, and per-layer inputs of a few tokens."""
    d = edg.make_desc(cfg, n_slots=cfg.E)
    host = layer_io.host_layer(d, lambda e: synth.expert_tensors(cfg, 0, e))
    slots = torch.zeros((n_layers, cfg.E, edg.record_bytes(d)), dtype=torch.uint8, device="cuda")
    tables = torch.zeros((n_layers, cfg.E), dtype=torch.int32, device="cuda")
    loras, keep = zip(*[layer_io.lora_to_device(d, [synth.lora_tensors(cfg, l, a) for a in range(cfg.n_adapters)]) for l in range(n_layers)])
    store = edg.Store(d, [host] * n_layers, slots, tables, list(loras), torch.cuda.Stream())
    for l in range(n_layers):
        store.load_whole_layer(l)
        store.wait_staged(l)
    W = torch.from_numpy(np.stack([synth.prerouter_weights(cfg, l) for l in range(n_layers)])).cuda()
    X = layer_io.bits_to_device(np.stack([synth.hidden_states(cfg, 9, layer=l, stream=stream) for l in range(n_layers)], axis=1), torch.bfloat16)
    torch.cuda.synchronize()
    return d, store, W, X, (slots, tables, keep)


@pytest.mark.parametrize("name,kw,n_layers", [
    ("cfg1", {}, 7),                                            # more layers than a workspace has exchange buffers, fp32 head
    ("cfg2", dict(E=32, K=4, n_slots=32), 6),
    ("cfg2", dict(E=32, K=8, n_slots=32, n_adapters=32), 3),    # all SMs in gate/up, an adapter per expert
    ("cfg2", dict(E=32, K=12, n_slots=32, rank=0), 5),          # more CTAs than SMs
])
def test_layers_of_a_token_side_by_side_are_the_layer_steps(name, kw, n_layers):
    """Resident layers run beside one another; every output is that of one moe_layer_decode after the other, bit for bit, with two
    stacks at once on two streams as well."""
    cfg = synth.CONFIGS[name].with_(**kw)
    stacks = [_resident_stack(cfg, n_layers, 71 + i) for i in range(2)]
    want = []
    for d, store, W, X, _ in stacks:
        ref = StackDecoder(d, store, W)
        ref.prime(X[8])
        rows = []
        for t in range(8):
            cur, nxt = t % 2, (t + 1) % 2
            y, lg = torch.zeros((n_layers, cfg.H), device="cuda"), torch.zeros((n_layers, cfg.E), device="cuda")
            for l in range(n_layers):
                n = (l + 1) % n_layers
                edg.moe_layer_decode(store, l, X[t, l], ref.inds[cur, l], ref.gates[cur, l], W[l], ref.inds[nxt, n], ref.gates[nxt, n], lg[n], y[l], ref.ws)
            rows.append((y, lg, ref.inds[nxt].clone(), ref.gates[nxt].clone()))
        torch.cuda.synchronize()
        assert edg.workspace_status(ref.ws) == 0
        want.append(rows)
    for both in (False, True):
        decs, got = [], [[], []]
        for d, store, W, X, _ in stacks:
            decs.append(StackDecoder(d, store, W))
            decs[-1].prime(X[8])
        streams = [torch.cuda.Stream() for _ in stacks]
        torch.cuda.synchronize()
        for t in range(8):
            for i, (d, store, W, X, _) in enumerate(stacks):
                if i == 1 and not both:
                    continue
                with torch.cuda.stream(streams[i]):
                    y, lg = torch.zeros((n_layers, cfg.H), device="cuda"), torch.zeros((n_layers, cfg.E), device="cuda")
                    decs[i].step(t, X[t], y, lg)
                    got[i].append((y, lg, decs[i].inds[(t + 1) % 2].clone(), decs[i].gates[(t + 1) % 2].clone()))
        torch.cuda.synchronize()
        for i in range(1 + both):
            assert edg.workspace_status(decs[i].ws) == 0
            for t in range(8):
                for a, b in zip(got[i][t], want[i][t]):
                    assert torch.equal(a, b), (i, t)
    for _, store, _, _, _ in stacks:
        store.close()


def _tokens(cfg, n_layers, n, stream):
    """Layer inputs of n tokens of which three in a row are the same: the second and third of each find their experts where the first has put them."""
    X = np.stack([synth.hidden_states(cfg, (n + 2) // 3, layer=l, stream=stream) for l in range(n_layers)], axis=1)
    return layer_io.bits_to_device(np.repeat(X, 3, axis=0)[:n], torch.bfloat16)


def _shared(store, cfg, layers):
    d = edg.make_desc(cfg, n_slots=cfg.E)
    rec = torch.from_numpy(edg.pack_expert(d, synth.expert_tensors(cfg, 1, 0))).cuda()
    for l in layers:
        store.set_shared_expert(l, rec)


@pytest.mark.parametrize("n_slots,shared", [(8, ()), (5, ()), (8, (0, 2)), (32, (1, 3, 4))])
def test_layers_side_by_side_in_a_pool_that_evicts_and_beside_shared_experts(n_slots, shared):
    """Tokens that copy experts and tokens that find them, in pools smaller than the layer, shared experts on some layers: every output is that
    of one layer-step after the other over resident layers, bit for bit."""
    cfg, n_layers, T = synth.CONFIGS["cfg2"].with_(E=32, K=4, n_slots=32), 5, 18
    d, store, W, _, keep = _resident_stack(cfg, n_layers, 81)
    _shared(store, cfg, shared)
    X = _tokens(cfg, n_layers, T + 1, 82)
    ref, want = StackDecoder(d, store, W), []
    ref.prime(X[T])
    for t in range(T):
        cur, nxt = t % 2, (t + 1) % 2
        y, lg = torch.zeros((n_layers, cfg.H), device="cuda"), torch.zeros((n_layers, cfg.E), device="cuda")
        for l in range(n_layers):
            n = (l + 1) % n_layers
            edg.moe_layer_decode(store, l, X[t, l], ref.inds[cur, l], ref.gates[cur, l], W[l], ref.inds[nxt, n], ref.gates[nxt, n], lg[n], y[l], ref.ws)
        want.append((y, lg, ref.inds[nxt].clone(), ref.gates[nxt].clone()))
    torch.cuda.synchronize()
    store.close()
    d = edg.make_desc(cfg, n_slots=n_slots)
    host = layer_io.host_layer(d, lambda e: synth.expert_tensors(cfg, 0, e))
    slots = torch.zeros((n_layers, n_slots, edg.record_bytes(d)), dtype=torch.uint8, device="cuda")
    tables = torch.zeros((n_layers, cfg.E), dtype=torch.int32, device="cuda")
    loras, keep2 = zip(*[layer_io.lora_to_device(d, [synth.lora_tensors(cfg, l, 0)]) for l in range(n_layers)])
    store = edg.Store(d, [host] * n_layers, slots, tables, list(loras), torch.cuda.Stream())
    _shared(store, cfg, shared)
    dec, got, found = StackDecoder(d, store, W), [], 0
    dec.prime(X[T])
    for t in range(T):
        before = dec.misses
        y, lg = torch.zeros((n_layers, cfg.H), device="cuda"), torch.zeros((n_layers, cfg.E), device="cuda")
        dec.step(t, X[t], y, lg)
        found += dec.misses == before
        got.append((y, lg, dec.inds[(t + 1) % 2].clone(), dec.gates[(t + 1) % 2].clone()))
    torch.cuda.synchronize()
    assert edg.workspace_status(dec.ws) == 0
    assert 4 <= found < T and dec.misses > n_layers * cfg.K
    for t in range(T):
        for a, b in zip(got[t], want[t]):
            assert torch.equal(a, b), t
    store.close()


def test_a_token_whose_outputs_lie_on_inputs_that_have_been_used():
    """y of a layer on the input of the layer before it: the layers then run one after the other, with the results of separate buffers."""
    cfg, n_layers, T = synth.CONFIGS["cfg2"].with_(E=32, K=4, n_slots=32), 5, 6
    d, store, W, _, keep = _resident_stack(cfg, n_layers, 83)
    store.close()
    d = edg.make_desc(cfg, n_slots=32, out_dtype="bf16")
    slots, tables, kept = keep
    host = layer_io.host_layer(d, lambda e: synth.expert_tensors(cfg, 0, e))
    loras, keep2 = zip(*[layer_io.lora_to_device(d, [synth.lora_tensors(cfg, l, 0)]) for l in range(n_layers)])
    store = edg.Store(d, [host] * n_layers, slots, tables, list(loras), torch.cuda.Stream())
    for l in range(n_layers):
        store.load_whole_layer(l)
        store.wait_staged(l)
    X = _tokens(cfg, n_layers, T + 1, 84)
    rows = []
    for apart in (True, False):
        dec = StackDecoder(d, store, W)
        dec.prime(X[T])
        out = []
        for t in range(T):
            both = torch.zeros((n_layers + 1, cfg.H), dtype=torch.bfloat16, device="cuda")
            both[1:] = X[t]
            y = torch.zeros((n_layers, cfg.H), dtype=torch.bfloat16, device="cuda") if apart else both[:n_layers]
            dec.step(t, both[1:], y)
            out.append((y, dec.inds[(t + 1) % 2].clone()))
        torch.cuda.synchronize()
        assert edg.workspace_status(dec.ws) == 0
        rows.append(out)
    for a, b in zip(*rows):
        assert torch.equal(a[0], b[0]) and torch.equal(a[1], b[1])
    store.close()
