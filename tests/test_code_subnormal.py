"""The arithmetic behind codes as fp16 subnormals, in numpy against what IEEE fp16 fixes: code k of a 32-bit word sits in bits 4k..4k+3, so
masking both halves with 0x000F gives q * 2^-24 (codes 0 and 4; after a shift by 8: 2 and 6), with 0x00F0 q * 2^-20 (codes 1 and 5; 3
and 7).  Activations at odd positions carry 2^-4, all of them the power of two that brings the largest to 2^13 .. 2^14."""
import numpy as np
import pytest


def _halves(word):
    return np.array([word & 0xFFFF, word >> 16], dtype=np.uint16).view(np.float16).astype(np.float64)


def test_every_code_at_every_position_is_its_own_subnormal():
    for k in range(8):
        for q in range(16):
            w = q << (4 * k)
            words = [w & 0x000F000F, w & 0x00F000F0, (w >> 8) & 0x000F000F, (w >> 8) & 0x00F000F0]
            got = {}
            for r, word in enumerate(words):
                got[r], got[r + 4] = _halves(word)
            for kk in range(8):
                assert got[kk] == (q if kk == k else 0) * 2.0 ** (-24 if kk % 2 == 0 else -20)


def _vector_scale(m):
    """vector_scale of the kernels: from the bits of the largest magnitude"""
    field = min(267 - (int(np.float32(m).view(np.uint32)) >> 23), 253)
    return np.array([field << 23], dtype=np.uint32).view(np.float32).astype(np.float64)[0]


@pytest.mark.parametrize("exponent", [-110, -60, -30, -14, -6, 0, 6, 15, 60, 120])
def test_what_value_and_residual_lose(exponent):
    rng = np.random.default_rng(exponent + 200)
    v = (rng.standard_normal(128) * 2.0 ** exponent).astype(np.float32).astype(np.float64)
    v[5] = 0.0
    s = _vector_scale(np.abs(v).max())
    assert 2.0 ** 13 <= np.abs(v).max() * s < 2.0 ** 14
    odd = np.where(np.arange(128) % 2, 2.0 ** -4, 1.0)
    w = v * s * odd
    hi = w.astype(np.float16).astype(np.float64)
    lo = (w - hi).astype(np.float16).astype(np.float64)
    lost = np.abs((hi + lo) / odd / s - v)
    # 11 bits each, or half of the smallest subnormal of an odd position
    assert (lost <= np.maximum(2.0 ** -22 * np.abs(v), 2.0 ** -25 / 2.0 ** -4 / s)).all()
    assert 2.0 ** -25 / 2.0 ** -4 / s <= 2.0 ** -34 * np.abs(v).max()


def test_the_ends_of_the_scale():
    assert _vector_scale(0.0) == 2.0 ** 126 and _vector_scale(np.float32(3e38)) * 3e38 < 2.0 ** 14
    assert np.isfinite(_vector_scale(np.float32(np.inf))) and _vector_scale(np.float32(np.inf)) > 0
