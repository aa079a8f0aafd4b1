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
