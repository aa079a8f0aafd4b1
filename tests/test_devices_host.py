"""Kernels that need more than 48 KB of shared memory, on the second device of a process: the host code against a runtime of two devices
in which nothing runs (tests/_fake_cudart.c).  And grids that no device takes."""
import ctypes as C
import os
import shutil
import subprocess

import pytest

import paper_2609_18063_b200 as edg

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(ROOT, "paper_2609_18063_b200", "csrc")


def _host_lib(out, sources):
    fake = out[:-3] + "_rt.o"
    subprocess.run([shutil.which("gcc"), "-c", "-fPIC", "-o", fake, os.path.join(HERE, "_fake_cudart.c")], check=True)
    subprocess.run([shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc", "-gencode", "arch=compute_100a,code=compute_100a", "-std=c++17", "-shared",
                    "-Xcompiler", "-fPIC", "-Xlinker", "-Bsymbolic", "-cudart", "none", "-I", os.path.join(ROOT, "include"), "-o", out,
                    "--threads", "0", *[os.path.join(CSRC, f) for f in sources], fake], check=True)
    return C.CDLL(out, mode=os.RTLD_LAZY)


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    return _host_lib(str(tmp_path_factory.mktemp("fake") / "libhost.so"), ["edg_prerouter.cu", "edg_pack.cu"])


@pytest.fixture(scope="module")
def grouped(tmp_path_factory):
    return _host_lib(str(tmp_path_factory.mktemp("fake") / "libgrouped.so"),
                     ["edg_ffn.cu", "edg_grouped.cu", "edg_grouped_ffn.cu", "edg_grouped_umma.cu", "edg_lora_tokens.cu", "edg_pack.cu"])


def _desc(**kw):
    return edg.make_desc(None, **dict(dict(H=2048, I=512, E=256, K=8, group=64, rank=16, n_adapters=1, n_slots=256), **kw))


P = 1 << 20          # an aligned address; nothing reads it


def _mlp(lib, dtype):
    head = edg.binding.MlpHead(P, None, P, None, P, 512)
    p = C.c_void_p(P)
    return lib.prerouter_mlp_topk(C.byref(_desc(pre_dtype=dtype)), C.byref(head), p, p, p, 40, p, p, None, None)


def _tokens(lib, dtype):
    p = C.c_void_p(P)
    return lib.prerouter_topk_tokens(C.byref(_desc(pre_dtype=dtype)), p, p, 64, p, p, None, None)


@pytest.mark.parametrize("dtype", ["f16", "f32"])
@pytest.mark.parametrize("call", [_mlp, _tokens])
def test_every_device_launches(lib, call, dtype):
    for device in (0, 1, 0, 1):
        lib.fake_set_device(device)
        before = lib.fake_launches()
        assert call(lib, dtype) == 0, device
        assert lib.fake_launches() == before + 1


@pytest.mark.parametrize("slots", [1, 1024, 1025, 21845, 40000, 49152, 49153, 50000, 52427, 60000])
def test_the_largest_calls_fit_a_grid(grouped, slots):
    """65,535 tokens of 32 choices, whatever the pool: every form's tiles stay within what a launch may have."""
    d = _desc(H=256, I=256, E=32, K=32, rank=8, n_slots=slots)
    p = C.c_void_p(P)
    lora = edg.binding.Lora(*[P] * 6)
    n = C.c_size_t()
    for T in (65535, 40 * slots // 32 + 1, 96 * slots // 32 + 1):
        if not 2 <= T <= 65535:
            continue
        assert grouped.edg_ffn_workspace_bytes(C.byref(d), T, C.byref(n)) == 0
        assert grouped.moe_expert_ffn_int4_lora(C.byref(d), p, p, T, p, p, p, p, C.byref(lora), p, p, n, None) == 0, T
