"""The grouped path where it can go wrong: edges of its tiles (8, 16 and 32 pairs) and of its units (narrow layers whose last unit
is partly empty), down slices of 32, 64 and 128 columns, every scale group, ranks that are no multiple of 8 or 16, adapters per
expert, the sort for pools beyond what shared memory counts, and the first sizes that take the tcgen05 tiles.  Every token
against the oracle; bars as everywhere (fp32 sums of exact int4 x bf16 products; the adapter's fp16 operands)."""
import dataclasses

import numpy as np
import pytest
import torch

import paper_2609_18063_b200 as edg
from oracle import moe_oracle as orc
from paper_2609_18063_b200 import layer_io
from workloads import synth

from _gpu_util import DeviceLayer, out_tensor, x_dev
from test_gpu_grouped import _check_tokens, _ffn_tokens

pytestmark = pytest.mark.gpu


def _layer(H, I, group, rank, E, K, n_adapters=1):
    cfg = dataclasses.replace(synth.CONFIGS["cfg1"], name=f"H{H}I{I}g{group}r{rank}", H=H, I=I, group=group, rank=rank, E=E, K=K,
                              n_slots=E, n_adapters=n_adapters, seed=23)
    return DeviceLayer(cfg)


def _routing(rng, T, E, K, pop=None):
    inds = np.stack([np.sort(rng.choice(E, K, replace=False, p=pop)) for _ in range(T)]).astype(np.int32)
    return inds, rng.dirichlet(np.ones(K), size=T).astype(np.float32)


@pytest.mark.parametrize("H,I,group,rank,E,K,n_adapters,T", [
    (256, 128, 32, 5, 4, 1, 1, 2),          # slices of 32 columns, odd rank, one unit of each kind and that one half empty
    (512, 256, 64, 8, 8, 2, 8, 17),         # tiles of up to 8: runs of 8 and 9 pairs
    (1024, 256, 32, 24, 8, 2, 1, 33),       # tiles of up to 16, second 16 ranks partly empty
    (2048, 512, 128, 16, 4, 2, 4, 50),      # tiles of up to 32: three columns and a remainder of one pair
    (1024, 1024, 64, 64, 4, 1, 1, 97),      # slices of two stages, the largest rank
    (4096, 512, 64, 0, 4, 2, 1, 70),        # wide state, no adapter
    # beyond 128 pairs, where a kernel sorts:
    (512, 256, 64, 24, 32, 2, 32, 100),     # tiles of up to 16, an adapter per expert
    (1024, 256, 32, 8, 32, 2, 1, 120),      # and one for all
    (512, 256, 64, 8, 8, 2, 8, 150),        # tiles of up to 32
    (2048, 512, 32, 16, 4, 2, 1, 150),
    (512, 256, 64, 16, 8, 1, 8, 320),       # the last size before the tcgen05 tiles
    (512, 512, 128, 16, 8, 1, 1, 320),
])
def test_streaming_form_at_tile_edges(H, I, group, rank, E, K, n_adapters, T):
    L = _layer(H, I, group, rank, E, K, n_adapters)
    X = synth.hidden_states(L.cfg, T, stream=61)
    inds_h, gates_h = _routing(np.random.default_rng(5), T, E, K, np.array([0.6] + [0.4 / (E - 1)] * (E - 1)))
    assert T * K <= (40 if group >= 64 else 96) * E                  # (the streaming form's line)
    Y = _ffn_tokens(L, L.desc, X, torch.from_numpy(inds_h).cuda(), torch.from_numpy(gates_h).cuda(), T)
    _check_tokens(L, X, inds_h, gates_h, Y, range(T))
    assert np.array_equal(Y, _ffn_tokens(L, L.desc, X, torch.from_numpy(inds_h).cuda(), torch.from_numpy(gates_h).cuda(), T))


@pytest.mark.parametrize("H,I,group,rank,E,K,n_adapters,T", [
    (512, 256, 32, 8, 32, 2, 32, 63),       # 126 pairs: the tiles find themselves
    (512, 256, 64, 24, 32, 2, 1, 64),       # 128: the last size that does
    (512, 256, 64, 24, 32, 2, 1, 65),       # 130: sorted
    (2048, 512, 64, 0, 64, 1, 1, 61),       # 61 pairs: the last narrow units of the larger layer, about
    (2048, 128, 32, 16, 64, 1, 64, 40),     # two narrow units a matrix
])
def test_few_pairs_find_their_tiles(H, I, group, rank, E, K, n_adapters, T):
    """Up to 128 pairs, tiles of 8: a slot of 20 pairs, single ones, a choice that is no slot, one named twice by a token."""
    L = _layer(H, I, group, rank, E, K, n_adapters)
    X = synth.hidden_states(L.cfg, T, stream=66)
    rng = np.random.default_rng(11)
    inds_h, gates_h = _routing(rng, T, E, K)
    inds_h[5:25, 0] = E - 2
    if K > 1:
        inds_h[5:25, 1] = E - 1
        inds_h[30] = 3
    inds, gates = torch.from_numpy(inds_h).cuda(), torch.from_numpy(gates_h).cuda()
    Y = _ffn_tokens(L, L.desc, X, inds, gates, T)
    _check_tokens(L, X, inds_h, gates_h, Y, range(T))
    assert np.array_equal(Y, _ffn_tokens(L, L.desc, X, inds, gates, T, use_table=False))
    bad = inds_h.copy()
    bad[7, K - 1] = -3
    y = out_tensor(L.desc, T)
    table = torch.arange(E, dtype=torch.int32, device="cuda")
    edg.moe_expert_ffn_int4_lora(L.desc, L.pool, table, T, torch.from_numpy(bad).cuda(), None, gates, x_dev(X), L.lora, y, L.ws)
    torch.cuda.synchronize()
    assert edg.workspace_status(L.ws) == -4
    got = y.cpu().numpy()
    assert np.array_equal(np.delete(got, 7, axis=0), np.delete(Y, 7, axis=0))
    if K > 1:
        _check_tokens(L, X, inds_h[:, :1], gates_h[:, :1], got, [7])
    else:
        assert not got[7].any()


@pytest.mark.parametrize("n_adapters", [1, 16])
def test_first_size_of_the_tensor_memory_tiles(n_adapters):
    """97 pairs per slot on the small layer: groups of 32, rank 8, ragged tiles, an expert that spans many tiles."""
    L = _layer(1024, 256, 32, 8, 16, 2, n_adapters)
    T = 776 + 1
    X = synth.hidden_states(L.cfg, T, stream=62)
    inds_h, gates_h = _routing(np.random.default_rng(6), T, 16, 2, np.array([0.3] + [0.7 / 15] * 15))
    assert T * 2 > 96 * 16
    Y = _ffn_tokens(L, L.desc, X, torch.from_numpy(inds_h).cuda(), torch.from_numpy(gates_h).cuda(), T)
    _check_tokens(L, X, inds_h, gates_h, Y, list(range(0, T, 9)) + [T - 1])


@pytest.mark.parametrize("I,group,rank,n_adapters", [(256, 64, 16, 8), (512, 128, 16, 1)])
def test_first_size_of_the_tensor_memory_tiles_in_wide_groups(I, group, rank, n_adapters):
    """41 pairs in a slot of eight and 40 in the others: one pair beyond the line of groups of 64 and more."""
    L = _layer(512, I, group, rank, 8, 1, n_adapters)
    T = 40 * 8 + 1
    X = synth.hidden_states(L.cfg, T, stream=69)
    inds_h = np.random.default_rng(14).permutation(np.arange(T, dtype=np.int32) % 8).reshape(T, 1)
    gates_h = np.random.default_rng(15).uniform(0.1, 1.0, size=(T, 1)).astype(np.float32)
    Y = _ffn_tokens(L, L.desc, X, torch.from_numpy(inds_h).cuda(), torch.from_numpy(gates_h).cuda(), T)
    _check_tokens(L, X, inds_h, gates_h, Y, list(range(0, T, 5)) + [T - 1])


def test_states_that_are_no_numbers_stay_in_their_rows_of_the_tensor_memory_tiles():
    """An infinity, a NaN and states whose h leaves fp16: their tokens' outputs are not finite, every other token's are the same bits."""
    L = _layer(512, 256, 64, 8, 4, 1)
    T = 300
    X = synth.hidden_states(L.cfg, T, stream=70)
    inds_h = np.random.default_rng(16).integers(0, 4, size=(T, 1)).astype(np.int32)
    inds, gates = torch.from_numpy(inds_h).cuda(), torch.ones((T, 1), device="cuda")
    clean = _ffn_tokens(L, L.desc, X, inds, gates, T)
    bad = X.copy()
    bad[17, 3], bad[120, 500] = 0x7F80, 0x7FC0
    bad[299] = synth.f32_to_bf16_bits(synth.bf16_bits_to_f32(X[299]) * np.float32(2.0 ** 12))
    Y = _ffn_tokens(L, L.desc, bad, inds, gates, T)
    odd = [17, 120, 299]
    assert not np.isfinite(Y[odd]).any()
    assert np.array_equal(np.delete(Y, odd, axis=0), np.delete(clean, odd, axis=0))


# pairs of the eight experts: edges of the tensor-memory tiles' rounding (16) and of the tiles (128), an unused expert, one of several tiles
_RUNS = [1, 16, 17, 127, 128, 129, 0, 452]


@pytest.mark.parametrize("H,I,group,rank,n_adapters", [
    (256, 128, 32, 0, 1),                   # the smallest layer: four stages a kernel, two sums per stage, no adapter
    (512, 256, 64, 8, 8),                   # half a k-step of ranks in down
    (1024, 512, 128, 40, 1),                # a sum over two stages; two stages of adapter in both kernels, the second partly empty
    (2048, 512, 32, 24, 8),
    (1024, 1024, 64, 64, 1),                # the largest rank
    (4096, 512, 128, 16, 1),                # wide state
])
def test_tensor_memory_tiles_at_their_edges(H, I, group, rank, n_adapters):
    L = _layer(H, I, group, rank, 8, 1, n_adapters)
    T = sum(_RUNS)
    X = synth.hidden_states(L.cfg, T, stream=64)
    order = np.random.default_rng(8).permutation(T)
    inds_h = np.repeat(np.arange(8, dtype=np.int32), _RUNS)[order].reshape(T, 1)
    gates_h = np.random.default_rng(9).uniform(0.1, 1.0, size=(T, 1)).astype(np.float32)
    assert T > 96 * 8
    inds, gates = torch.from_numpy(inds_h).cuda(), torch.from_numpy(gates_h).cuda()
    Y = _ffn_tokens(L, L.desc, X, inds, gates, T)
    assert np.isfinite(Y).all()
    last = [int(np.nonzero(inds_h[:, 0] == e)[0][j]) for e in range(8) if _RUNS[e] for j in {0, _RUNS[e] - 1, min(127, _RUNS[e] - 1)}]
    _check_tokens(L, X, inds_h, gates_h, Y, sorted(set(last) | set(range(0, T, 31))))
    assert np.array_equal(Y, _ffn_tokens(L, L.desc, X, inds, gates, T, use_table=False))


def test_tensor_memory_tiles_a_slot_named_twice_and_one_out_of_range():
    """More pairs of a slot than there are tokens; a choice that is no slot leaves its share out and is reported."""
    L = _layer(512, 256, 64, 8, 4, 2)
    T = 200
    X = synth.hidden_states(L.cfg, T, stream=65)
    inds_h = np.full((T, 2), 1, np.int32)
    inds_h[::5] = [0, 3]
    gates_h = np.random.default_rng(10).dirichlet(np.ones(2), size=T).astype(np.float32)
    assert T * 2 > 40 * 4
    gates = torch.from_numpy(gates_h).cuda()
    Y = _ffn_tokens(L, L.desc, X, torch.from_numpy(inds_h).cuda(), gates, T)
    _check_tokens(L, X, inds_h, gates_h, Y, range(0, T, 7))
    bad = inds_h.copy()
    bad[7, 1] = 4
    y = out_tensor(L.desc, T)
    edg.moe_expert_ffn_int4_lora(L.desc, L.pool, None, T, torch.from_numpy(bad).cuda(), torch.from_numpy(bad).cuda(), gates, x_dev(X), L.lora, y, L.ws)
    torch.cuda.synchronize()
    assert edg.workspace_status(L.ws) == -4
    got = y.cpu().numpy()
    assert np.array_equal(np.delete(got, 7, axis=0), np.delete(Y, 7, axis=0))
    ref = orc.moe_ffn(X[7], bad[7, :1], gates_h[7, :1].astype(np.float64), L.expert, L.get_lora, L.cfg.lora_scale, L.cfg.group)
    assert orc.max_abs(got[7], ref) <= 2e-2 and orc.rel_l2(got[7], ref) <= 1e-3


@pytest.mark.parametrize("x_exp,a_exp,b_exp", [(5, -19, 13), (-12, 22, 0)])
@pytest.mark.parametrize("I,rank,n_adapters", [(256, 8, 4), (256, 40, 1), (1024, 8, 1)])
def test_tensor_memory_tiles_and_the_magnitude_of_h_and_its_adapter(I, rank, n_adapters, x_exp, a_exp, b_exp):
    """Adapters per expert, of more than 32 ranks, or of layers that are not 256 or 512 wide: rows of A_down near 2^-19 beside an h near 2^11, and
    near 2^22 beside an h near 2^-23, keep the bits that fp16 would take from them.  The adapter's share is the larger one; what is left is
    the fp16 of sigma A h, 2^-12 of each rank's share."""
    L = _layer(512, I, 64, rank, 4, 1, n_adapters)
    two = lambda bits, e: synth.f32_to_bf16_bits(np.ldexp(synth.bf16_bits_to_f32(bits), e))
    unit = {p: 1 / s for p, s in (("A", 0.02), ("B", 0.01))}         # synth's standard deviations
    ident = lambda bits, k: synth.f32_to_bf16_bits(synth.bf16_bits_to_f32(bits) * np.float32(unit[k]))
    for ad in L.adapters:
        ad["down"] = (two(ident(ad["down"][0], "A"), a_exp), two(ident(ad["down"][1], "B"), b_exp))
    L.lora, L._keep = layer_io.lora_to_device(L.desc, L.adapters)
    for e in range(4):
        codes, scales, zeros = L.expert(e)["down"]
        L.expert(e)["down"] = (codes, (scales / 64).astype(np.float16), zeros)
    L.pool = layer_io.host_layer(L.desc, L.expert).cuda()
    T = 200
    X = two(synth.hidden_states(L.cfg, T, stream=67), x_exp)
    inds_h = np.random.default_rng(12).integers(0, 4, size=(T, 1)).astype(np.int32)
    gates_h = np.ones((T, 1), np.float32)
    assert T > 40 * 4
    Y = _ffn_tokens(L, L.desc, X, torch.from_numpy(inds_h).cuda(), torch.from_numpy(gates_h).cuda(), T)
    for t in range(0, T, 9):
        ref = orc.moe_ffn(X[t], inds_h[t], [1.0], L.expert, L.get_lora, L.cfg.lora_scale, L.cfg.group)
        bare = orc.moe_ffn(X[t], inds_h[t], [1.0], L.expert, lambda e: {**L.get_lora(e), "down": (L.get_lora(e)["down"][0], np.zeros_like(L.get_lora(e)["down"][1]))},
                           L.cfg.lora_scale, L.cfg.group)
        assert np.linalg.norm(ref - bare) > 0.5 * np.linalg.norm(ref)
        assert orc.rel_l2(Y[t], ref) <= 2.0 ** -11


def test_both_forms_activate_alike():
    """One code per row that is not its zero point: gate, up and down are single exact products, so what is left is silu(gate) up, and the
    128-token tiles give the bits of the streaming form."""
    L = _layer(512, 256, 64, 0, 4, 1)
    def one_hot(n, kd, first):
        q = np.full((n, kd), 8, np.uint8)
        q[np.arange(n), (np.arange(n) + first) % kd] = 9
        return q[:, 0::2] | q[:, 1::2] << 4, np.ones((n, kd // 64), np.float16), np.full((n, kd // 64), 8, np.float16)
    for e in range(4):
        L._experts[e] = {"gate": one_hot(256, 512, e), "up": one_hot(256, 512, 100 + e), "down": one_hot(512, 256, e)}
    L.pool = layer_io.host_layer(L.desc, L.expert).cuda()
    T, rng = 200, np.random.default_rng(13)
    X = synth.f32_to_bf16_bits(rng.uniform(-30, 30, size=(T, 512)).astype(np.float32))
    inds_h = rng.integers(0, 4, size=(T, 1)).astype(np.int32)
    inds, gates = torch.from_numpy(inds_h).cuda(), torch.ones((T, 1), device="cuda")
    assert T > 40 * 4
    Y = _ffn_tokens(L, L.desc, X, inds, gates, T)
    _check_tokens(L, X, inds_h, np.ones((T, 1), np.float32), Y, range(0, T, 50))
    few = np.concatenate([_ffn_tokens(L, L.desc, X[t:t + 50], inds[t:t + 50].contiguous(), gates[t:t + 50], 50) for t in range(0, T, 50)])
    assert np.array_equal(Y, few)


@pytest.mark.parametrize("T", [9, 70])
def test_pool_with_more_slots_than_shared_memory_counts(T):
    """26,000 slots: the sort of 140 pairs keeps its counters in the workspace (18 pairs find their tiles without one, as up to 128 do).  The
    experts live in the first, a middle, the last and another slot."""
    cfg = _layer(256, 128, 32, 8, 4, 2).cfg
    S = 26000
    desc = edg.make_desc(cfg, n_slots=S)
    R = edg.record_bytes(desc)
    pool = torch.empty((S, R), dtype=torch.uint8, device="cuda")
    where = [0, 13001, 25999, 7]
    for e, s in enumerate(where):
        pool[s] = torch.from_numpy(edg.pack_expert(desc, synth.expert_tensors(cfg, 0, e))).cuda()
    table = torch.tensor(where, dtype=torch.int32, device="cuda")
    lora, keep = layer_io.lora_to_device(desc, [synth.lora_tensors(cfg, 0, 0)])
    X = synth.hidden_states(cfg, T, stream=63)
    inds_h, gates_h = _routing(np.random.default_rng(7), T, 4, 2)
    ws, y = layer_io.new_workspace(desc, T), out_tensor(desc, T)
    edg.moe_expert_ffn_int4_lora(desc, pool, table, T, torch.from_numpy(inds_h).cuda(), None, torch.from_numpy(gates_h).cuda(), x_dev(X),
                                 lora, y, ws)
    torch.cuda.synchronize()
    assert edg.workspace_status(ws) == 0
    for t in range(T):
        ref = orc.moe_ffn(X[t], inds_h[t], gates_h[t].astype(np.float64), lambda e: synth.expert_tensors(cfg, 0, e),
                          lambda e: synth.lora_tensors(cfg, 0, 0), cfg.lora_scale, cfg.group)
        assert orc.max_abs(y[t].cpu().numpy(), ref) <= 2e-2 and orc.rel_l2(y[t].cpu().numpy(), ref) <= 1e-3
