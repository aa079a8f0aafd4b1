"""The full head's streaming rings and the register form of the sigmoid-group gate at the sizes where they can go wrong: rows of half a
slot, of one, of several and of a broken one, warps and CTAs without rows, fp32 residual rows; every number of entries
per lane, one expert group per lane, ties and NaN.  The checks are those of test_gpu_routing."""
import dataclasses

import numpy as np
import pytest
import torch

import paper_2609_18063_b200 as edg
from oracle import moe_oracle as orc
from workloads import synth

import test_gpu_routing as routing

pytestmark = pytest.mark.gpu


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
