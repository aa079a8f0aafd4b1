"""The full head's streaming rings at the sizes where they can go wrong: rows of half a slot, of one, of several and of a broken one,
warps and CTAs without rows, fp32 residual rows.  The checks are those of test_gpu_routing."""
import dataclasses

import pytest

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
