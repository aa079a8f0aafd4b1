"""The lone and the chained layer-step over the magnitudes of the hidden state and of h, without an adapter: the codes are multiplied
exactly, so what is left is fp32 sums of up to 2048 products and __expf (relative 2^-21 and 2^-22), whatever the magnitude.  The bound is
four times the largest error seen on a B200; fp16 activations without a scale of their own are off by 1e-3 and more at a state of 1e-4."""
import dataclasses

import numpy as np
import pytest
import torch

import paper_2609_18063_b200 as edg
from oracle import moe_oracle as orc
from paper_2609_18063_b200 import layer_io
from workloads import synth

from _gpu_util import x_dev

pytestmark = pytest.mark.gpu

BOUND = 1.2e-5        # seen: 3.1e-6


@pytest.mark.parametrize("H,I,group", [(1024, 256, 32), (2048, 512, 64), (1024, 512, 128), (2048, 256, 32)])
@pytest.mark.parametrize("chaining", [0, 2])
def test_error_against_64_bits_at_every_magnitude(H, I, group, chaining):
    cfg = dataclasses.replace(synth.CONFIGS["cfg1"], name="small", H=H, I=I, group=group, E=16, K=4, rank=0, n_slots=16, pre_dtype="f16", seed=37)
    d = edg.make_desc(cfg, n_slots=16)
    host = layer_io.host_layer(d, lambda e: synth.expert_tensors(cfg, 0, e))
    pool, tables = torch.empty((1, 16, host.shape[1]), dtype=torch.uint8, device="cuda"), torch.empty((1, 16), dtype=torch.int32, device="cuda")
    store = edg.Store(d, [host], pool, tables, None, torch.cuda.Stream())
    store.load_whole_layer(0)
    scales = [2.0 ** e for e in (6, 0, -3, -7, -10, -14, -18, -24, -40, -100)]        # h runs from 1e4 down to far below fp16, and to zero
    base = synth.bf16_bits_to_f32(synth.hidden_states(cfg, 1, stream=5))[0]
    base[:64] *= 2.0 ** -12                                                            # a block far smaller than the others
    X = np.stack([synth.f32_to_bf16_bits(base * s) for s in scales])
    n, W = len(scales), torch.from_numpy(synth.prerouter_weights(cfg)).cuda()
    xd, ws = x_dev(X), layer_io.new_workspace(d)
    inds, gates, y = torch.zeros((n + 1, 4), dtype=torch.int32, device="cuda"), torch.zeros((n + 1, 4), device="cuda"), torch.zeros((n, H), device="cuda")
    edg.prerouter_topk(d, W, xd[:1], 1, inds[0], gates[0])
    store.set_chaining(chaining)
    for t in range(n):
        edg.moe_layer_decode(store, 0, xd[t], inds[t], gates[t], W, inds[t + 1], gates[t + 1], None, y[t], ws)
    assert edg.workspace_status(ws) == 0
    ih, gh, yh = inds.cpu().numpy(), gates.cpu().numpy(), y.cpu().numpy()
    worst = 0.0
    for t in range(n):
        ref = orc.moe_ffn(X[t], ih[t], gh[t].astype(np.float64), lambda e: synth.expert_tensors(cfg, 0, e), None, cfg.lora_scale, group)
        if np.abs(ref).max() < 1e-30:          # (below what fp32 holds as a normal number after the codes' 2^-24)
            assert np.isfinite(yh[t]).all() and np.abs(yh[t]).max() < 1e-29
            continue
        worst = max(worst, orc.rel_l2(yh[t], ref))
        assert orc.rel_l2(yh[t], ref) <= BOUND, (scales[t], orc.rel_l2(yh[t], ref))
    print("largest relative error", worst)
    store.close()
