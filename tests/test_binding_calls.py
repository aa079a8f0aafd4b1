"""The calls that go through the C extension: addresses of every kind of buffer, and the errors of the wrong ones."""
import ctypes
import types

import numpy as np
import pytest
import torch

import paper_2609_18063_b200 as edg


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2609_18063_b200 import build
    build.build()


def _decode(x, store=None, **kw):
    store = store or types.SimpleNamespace(handle=None)
    return edg.moe_layer_decode(store, 0, x, None, None, None, None, None, None, None, None, workspace_bytes=0, stream=0, **kw)


@pytest.mark.parametrize("x", [None, 0, 4096, torch.zeros(4), np.zeros(4, np.float32)])
def test_any_buffer_reaches_the_library(x):
    with pytest.raises(edg.EdgError) as e:          # a null store: EDG_E_INVAL from the library itself
        _decode(x)
    assert e.value.code == -1 and "moe_layer_decode" in str(e.value)


@pytest.mark.parametrize("x,error", [(torch.zeros(4, 4).t(), ValueError), (np.zeros((4, 4)).T, ValueError), ([1.0], TypeError),
                                     ("x", TypeError)])
def test_what_has_no_address_is_an_error(x, error):
    with pytest.raises(error):
        _decode(x)


def test_descriptor_and_stream_arguments():
    d = edg.make_desc(None, H=1024, I=256, E=16, K=2, group=32, rank=8, n_adapters=1, n_slots=16)
    with pytest.raises(edg.EdgError):               # null pointers, checked by the library before any launch
        edg.softmax_topk_rows(d, None, 1, None, None, stream=0)
    with pytest.raises(TypeError):
        edg.softmax_topk_rows(ctypes.c_int32(0), None, 1, None, None, stream=0)
    with pytest.raises(AttributeError):
        edg.softmax_topk_rows(d, None, 1, None, None, stream="s")
    with pytest.raises(edg.EdgError):
        edg.softmax_topk_rows(d, None, 1, None, None, stream=types.SimpleNamespace(cuda_stream=0))


def _gate(T=1, scale=1.0):
    """reaches the library with T rows and no buffers: EDG_E_INVAL"""
    edg.sigmoid_group_topk_rows(None, T, 32, 2, 4, 2, scale, None, None, None, stream=0)


@pytest.mark.parametrize("T", [3, True, np.int32(3), np.int64(3), ctypes.c_int32(3), 2 ** 40 + 3, -1, torch.tensor(3)])
def test_what_ctypes_takes_for_an_integer(T):
    with pytest.raises(edg.EdgError):
        _gate(T)


@pytest.mark.parametrize("T", [3.0, "3", None, ctypes.c_int64(3)])
def test_what_is_no_integer(T):
    with pytest.raises(TypeError):
        _gate(T)


@pytest.mark.parametrize("scale", [2, np.float32(2.5), "2.5", torch.tensor(2.5)])
def test_what_makes_a_float(scale):
    with pytest.raises(edg.EdgError):
        _gate(1, scale)


@pytest.mark.parametrize("n", [0, -1, 2 ** 70, np.int64(4096), ctypes.c_size_t(4096)])
def test_workspace_bytes_of_any_integer_type(n):
    with pytest.raises(edg.EdgError):
        edg.moe_layer_decode(types.SimpleNamespace(handle=None), 0, None, None, None, None, None, None, None, None, None, workspace_bytes=n, stream=0)


def test_a_structure_of_another_type_is_an_error():
    d = edg.make_desc(None, H=1024, I=256, E=16, K=2, group=32, rank=8, n_adapters=1, n_slots=16)
    other = edg.binding.MlpHead()                # as large as a Lora
    assert ctypes.sizeof(other) == ctypes.sizeof(edg.binding.Lora)
    call = lambda desc, lora: edg.moe_expert_ffn_int4_lora(desc, None, None, 1, None, None, None, None, lora, None, None, 0, 0)
    for desc, lora in ((d, other), (bytes(d), None), (edg.binding.Lora(), None)):
        with pytest.raises(TypeError):
            call(desc, lora)

    class Mine(edg.binding.LayerDesc):
        pass
    mine = Mine()
    ctypes.memmove(ctypes.byref(mine), ctypes.byref(d), ctypes.sizeof(d))
    with pytest.raises(edg.EdgError):
        call(mine, edg.binding.Lora())
