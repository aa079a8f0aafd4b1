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
