"""The full head's streaming rings and the register form of the sigmoid-group gate at the sizes where they can go wrong: rows of half a
slot, of one, of several and of a broken one, warps and CTAs without rows, fp32 residual rows; every number of entries
per lane, one expert group per lane, ties and NaN.  The checks are those of test_gpu_routing."""
import ctypes as C
import dataclasses
import os
import shutil
import subprocess

import numpy as np
import pytest
import torch

import paper_2609_18063_b200 as edg
from oracle import moe_oracle as orc
from workloads import synth

import test_gpu_routing as routing

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.mark.parametrize("H,E,K,pre,width,n_heads,variant", [
    (512, 40, 3, "f16", 24, 2, "full"),           # half a slot; five rows per CTA for eight warps, three of fc1
    (1024, 16, 2, "f32", 264, 2, "full"),         # fp32 residual rows of two slots; fc2 rows of 33 pieces
    (4096, 24, 2, "f16", 1032, 1, "full"),        # rows of four slots; fc2 rows of one slot and one piece
    (2048, 8, 2, "f16", 8, 1, "no_residual"),     # one row of either kind per CTA
])
def test_full_head_at_the_edges_of_its_rings(monkeypatch, H, E, K, pre, width, n_heads, variant):
    cfg = dataclasses.replace(synth.CONFIGS["cfg1"], name="edge", H=H, E=E, K=K, pre_dtype=pre, n_slots=E)
    monkeypatch.setitem(synth.CONFIGS, "edge", cfg)
    routing.test_mlp_head_matches_the_oracle("edge", width, n_heads, variant)


@pytest.mark.parametrize("E,n,G,K,T,with_bias", [(32, 4, 2, 3, 9, True), (64, 32, 5, 4, 40, False), (96, 4, 4, 8, 33, True),
                                                 (160, 8, 4, 8, 17, True), (192, 8, 3, 8, 33, False), (384, 16, 8, 8, 25, True),
                                                 (512, 32, 8, 32, 11, False), (448, 16, 4, 8, 9, True)])
def test_group_gate_in_registers(E, n, G, K, T, with_bias):
    routing.test_sigmoid_group_rows_match_the_oracle(E, n, G, K, T, with_bias)


def test_group_gate_ties_and_nans():
    """Row 0: all equal; row 1: ties across lanes and inside one; row 2: a NaN is no candidate."""
    l = np.zeros((3, 128), np.float32)
    l[1, [5, 6, 70, 71, 127]] = 2.0
    l[2] = np.linspace(-1, 1, 128, dtype=np.float32)
    l[2, 127] = np.nan
    inds = torch.zeros((3, 4), dtype=torch.int32, device="cuda")
    gates = torch.zeros((3, 4), dtype=torch.float32, device="cuda")
    edg.sigmoid_group_topk_rows(torch.from_numpy(l).cuda(), 3, 128, 4, 8, 4, 2.5, None, inds, gates)
    torch.cuda.synchronize()
    got = inds.cpu().numpy().tolist()
    assert got[0] == [0, 1, 2, 3] and got[2] == [123, 124, 125, 126]
    want_i, want_w = orc.sigmoid_group_topk(l[1], 4, 8, 4, 2.5)
    assert got[1] == want_i.tolist() == [5, 6, 70, 71]
    assert np.allclose(gates.cpu().numpy()[1], want_w, rtol=2e-6)


@pytest.mark.parametrize("pre,variant", [("f16", "full"), ("f32", "full"), ("f16", "no_residual")])
def test_full_head_whose_copies_do_not_come_in_time(tmp_path, pre, variant):
    """The library's heads built with no polls at all: every wait for a copy runs out at once, the rows come straight from memory, and the
    results are those of the rings, bit for bit."""
    so = str(tmp_path / "late.so")
    csrc = os.path.join(ROOT, "paper_2609_18063_b200", "csrc")
    subprocess.run([shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc", "-gencode", "arch=compute_100a,code=sm_100a", "-std=c++17", "-shared", "-Xcompiler",
                    "-fPIC", "-Xlinker", "-Bsymbolic", "-DEDG_MLP_RING_POLLS=0", "-I", os.path.join(ROOT, "include"), "-o", so,
                    os.path.join(csrc, "edg_prerouter.cu"), os.path.join(csrc, "edg_pack.cu")], check=True)
    late = C.CDLL(so, mode=os.RTLD_LAZY)
    n, H, E, K, D = 3, 1024, 40, 4, 520
    d = edg.make_desc(None, H=H, I=256, E=E, K=K, group=32, rank=0, n_adapters=1, n_slots=E, pre_dtype=pre)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(4)

    def rnd(*shape):
        return (torch.randn(shape, generator=gen, device="cuda") * 0.03).half()
    W1, b1, W2, b2, Wr, x = rnd(n, D, H + 2 * E), rnd(n, D), rnd(n, E, D), rnd(n, E), rnd(n, E, H), torch.randn((n, H), generator=gen, device="cuda").bfloat16()
    Wr = (Wr.float() if pre == "f32" else Wr) if variant == "full" else None
    cur = torch.arange(n * K, dtype=torch.int32, device="cuda").view(n, K)
    out = [(torch.zeros((n, K), dtype=torch.int32, device="cuda"), torch.zeros((n, K), device="cuda"), torch.zeros((n, E), device="cuda")) for _ in range(2)]
    edg.prerouter_mlp_topk(d, W1, b1, W2, b2, Wr, D, x, cur, cur, n, *out[0])
    ptr = lambda t: None if t is None else C.c_void_p(t.data_ptr())
    head = edg.binding.MlpHead(*[None if t is None else t.data_ptr() for t in (W1, b1, W2, b2, Wr)], D)
    torch.cuda.synchronize()
    assert late.prerouter_mlp_topk(C.byref(d), C.byref(head), ptr(x), ptr(cur), ptr(cur), n, *[ptr(t) for t in out[1]], None) == 0
    torch.cuda.synchronize()
    for a, b in zip(*out):
        assert torch.equal(a, b)
    assert out[0][2].abs().max() > 0


@pytest.mark.parametrize("H,E,K,dtype", [(256, 16, 3, "f32"), (1024, 48, 4, "f16"), (2048, 64, 8, "f32"), (512, 160, 2, "f16"), (2048, 160, 6, "f32")])
@pytest.mark.parametrize("T", [2, 15, 16, 17, 95, 96, 97, 517])
def test_many_tokens_of_a_head_in_sixteens(H, E, K, dtype, T):
    """Blocks of 16 tokens, ragged, and the form for other sizes, states from 1e-20 to 1e6: fp32 weights are summed from three bf16
    parts without loss.  Bar: sums of H products in fp32, 2^-24 of the sum of their magnitudes each way of adding."""
    d = edg.make_desc(None, H=H, I=128, E=E, K=K, group=32, rank=0, n_adapters=1, n_slots=E, pre_dtype=dtype, lora_scale=1.0, out_dtype="f32")
    gen = torch.Generator(device="cuda")
    gen.manual_seed(T)
    W = torch.randn((E, H), generator=gen, device="cuda") * 0.02
    if dtype == "f16":
        W = W.half()
    mag = 10.0 ** (torch.arange(T, device="cuda") % 27 - 20).double()
    X = (torch.randn((T, H), generator=gen, device="cuda").double() * mag[:, None]).bfloat16()
    inds, gates, logits = torch.full((T, K), -1, dtype=torch.int32, device="cuda"), torch.zeros((T, K), device="cuda"), torch.zeros((T, E), device="cuda")
    edg.prerouter_topk_tokens(d, W, X, T, inds, gates, logits)
    torch.cuda.synchronize()
    want, size = X.double() @ W.double().T, X.double().abs() @ W.double().abs().T
    assert ((logits.double() - want).abs() <= 4 * 2.0 ** -24 * size).all()
    top = torch.topk(logits, K).indices.sort(-1).values
    assert torch.equal(inds.long(), top)
    picked = torch.gather(logits.double(), 1, top)
    assert torch.allclose(gates.double(), torch.softmax(picked, -1), rtol=2e-5, atol=1e-7)


@pytest.mark.parametrize("H,E,K,dtype,line", [(256, 16, 3, "f32", 320), (256, 48, 4, "f16", 256), (512, 32, 2, "f32", 6), (1024, 48, 4, "f32", 128), (1024, 64, 4, "f16", 4),
                                              (1024, 160, 6, "f32", 384), (2048, 64, 8, "f32", 128), (2048, 144, 2, "f16", 6), (4096, 64, 3, "f32", 8),
                                              (4096, 320, 8, "f32", 256), (4096, 320, 8, "f16", 128)])
def test_a_head_on_both_sides_of_the_line_between_its_forms(H, E, K, dtype, line):
    """The last number of tokens of one form and the first of the other."""
    for T in (line - 1, line):
        test_many_tokens_of_a_head_in_sixteens(H, E, K, dtype, T)


@pytest.mark.parametrize("dtype", ["f32", "f16"])
def test_infinities_in_a_head_of_many_tokens(dtype):
    """An infinite weight or state makes the logits it makes in plain arithmetic, and no others."""
    H, E, T = 512, 32, 33
    d = edg.make_desc(None, H=H, I=128, E=E, K=2, group=32, rank=0, n_adapters=1, n_slots=E, pre_dtype=dtype, lora_scale=1.0, out_dtype="f32")
    W = torch.randn((E, H), device="cuda") * 0.02
    W[3, 5], W[9, 40] = float("inf"), -float("inf")
    W = W.half() if dtype == "f16" else W
    X = torch.randn((T, H), device="cuda").bfloat16()
    X[7, 11], X[20, 5] = float("inf"), 0.0
    inds, gates, logits = torch.zeros((T, 2), dtype=torch.int32, device="cuda"), torch.zeros((T, 2), device="cuda"), torch.zeros((T, E), device="cuda")
    edg.prerouter_topk_tokens(d, W, X, T, inds, gates, logits)
    torch.cuda.synchronize()
    want = (X.double().cpu()[:, None, :] * W.double().cpu()[None]).sum(-1)
    got = logits.double().cpu()
    assert torch.equal(torch.isnan(got), torch.isnan(want)) and torch.equal(torch.isinf(got), torch.isinf(want))
    inf, fin = torch.isinf(want), torch.isfinite(want)
    assert torch.equal(got[inf], want[inf]) and (got[fin] - want[fin]).abs().max() <= 1e-5


@pytest.mark.parametrize("dtype", ["f32", "f16"])
def test_padding_that_is_not_a_number_in_a_head_of_many_tokens(dtype):
    """States and weights that are no numbers make the logits that are none, and such a state in every block of tokens costs next to nothing
    (at most the time of the call once more)."""
    H, E, T = 2048, 160, 1024
    d = edg.make_desc(None, H=H, I=128, E=E, K=2, group=32, rank=0, n_adapters=1, n_slots=E, pre_dtype=dtype, lora_scale=1.0, out_dtype="f32")
    W = torch.randn((E, H), device="cuda") * 0.02
    W = W.half() if dtype == "f16" else W
    X = torch.randn((T, H), device="cuda").bfloat16()
    inds, gates, logits = torch.zeros((T, 2), dtype=torch.int32, device="cuda"), torch.zeros((T, 2), device="cuda"), torch.zeros((T, E), device="cuda")

    def us():
        call = lambda: edg.prerouter_topk_tokens(d, W, X, T, inds, gates, logits)
        call()
        times = []
        for _ in range(7):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            torch.cuda.synchronize()
            a.record()
            for _ in range(10):
                call()
            b.record()
            torch.cuda.synchronize()
            times.append(a.elapsed_time(b))
        return sorted(times)[3]
    plain, clean = us(), logits.clone()
    X[11::16, 77] = float("nan")
    assert us() <= 2 * plain
    pad = torch.arange(T, device="cuda") % 16 == 11
    assert torch.isnan(logits[pad]).all() and torch.equal(logits[~pad], clean[~pad])
    W[37, 1203] = float("nan")
    edg.prerouter_topk_tokens(d, W, X, T, inds, gates, logits)
    torch.cuda.synchronize()
    assert torch.isnan(logits[:, 37]).all()
    rest = torch.arange(E, device="cuda") != 37
    assert torch.equal(logits[~pad][:, rest], clean[~pad][:, rest]) and not (inds[~pad] == 37).any()
