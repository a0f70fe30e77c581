"""The library's host code on a CUDA runtime without a GPU (fake_cudart.cpp): what the prefill's launches
and workspace do on a second device, when an allocation fails and under stream capture."""
import ctypes as C
import dataclasses
import importlib
import os
import shutil
import subprocess

import numpy as np
import pytest

from paper_2609_34045_gb300 import stage as K
from paper_2609_34045_gb300 import workload as wl
from test_gpu_wide import CASES

B = importlib.import_module("paper_2609_34045_gb300.build")  # (the package binds the name to its function)
HERE = os.path.dirname(os.path.abspath(__file__))
# weight tiles of 128 tokens from 129 tokens on (F large enough for every SM), few layers
WIDE = wl.ModelShape(n_layers_total=1, d_model=128, n_heads=2, n_kv_heads=1, head_dim=64, ffn=19456, vocab=300)
SMALL = wl.ModelShape(n_layers_total=1, d_model=128, n_heads=2, n_kv_heads=1, head_dim=64, ffn=256, vocab=300)
QK = dataclasses.replace(SMALL, qk_norm=True)
INT4 = dataclasses.replace(SMALL, weight_fmt="int4_g64")


@pytest.fixture(scope="module")
def fake_lib(tmp_path_factory):
    B.build()
    out = str(tmp_path_factory.mktemp("fake") / "libfake.so")
    cuda = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(B.nvcc()))), "include")
    objs = [os.path.join(B.BUILD, f) for f in sorted(os.listdir(B.BUILD)) if f.endswith(".o")]
    subprocess.run(["g++", "-std=c++17", "-O1", "-fPIC", "-shared", "-Wl,-Bsymbolic", "-I", cuda, "-o", out,
                    os.path.join(HERE, "fake_cudart.cpp"), *objs], check=True)
    return out


@pytest.fixture
def dev(fake_lib, tmp_path, monkeypatch):
    """The library on a fake device of its own, behind the package's binding."""
    path = shutil.copy(fake_lib, tmp_path / "libkafila_fake.so")
    monkeypatch.setattr(K, "LIB_PATH", str(path))
    monkeypatch.setattr(K, "_lib", None)
    monkeypatch.delenv("KFL_PREFILL_DENSE_MIN", raising=False)
    lib = K.lib()
    lib.fake_live.restype = lib.fake_peak.restype = lib.fake_pool_held.restype = C.c_size_t
    lib.fake_launches.restype = lib.fake_mallocs.restype = lib.fake_marked.restype = C.c_long
    lib.fake_budget.argtypes = [C.c_size_t]
    return lib


def _load(st, model):
    d, hd, kv, f = model.d_model, model.head_dim, model.n_kv_heads * model.head_dim, model.ffn
    w = {n: np.zeros(m, dtype=np.uint16) for n, m in (("attn_norm", d), ("ffn_norm", d), ("q_norm", hd), ("k_norm", hd))}
    for n, rows, cols in (("wq", model.n_heads * hd, d), ("wk", kv, d), ("wv", kv, d), ("wo", d, model.n_heads * hd),
                          ("wg", f, d), ("wu", f, d), ("wd", d, f)):
        w[n] = (np.zeros((rows, cols), dtype=np.uint16) if model.weight_fmt == "bf16" else
                (np.zeros((rows, cols // 8), dtype=np.uint32), np.zeros((rows, cols // 64), dtype=np.uint16)))
    K.kfl_stage_load_layer(st, 0, w, on_device=False)
    if st.flags:
        head = {"embed": np.zeros((model.vocab, d), dtype=np.uint16), "final_norm": w["attn_norm"]}
        head["lm_head"] = head["embed"] if model.weight_fmt == "bf16" else (
            np.zeros((model.vocab, d // 8), dtype=np.uint32), np.zeros((model.vocab, d // 64), dtype=np.uint16))
        K.kfl_stage_load_head(st, head, on_device=False)


def _stage(model, max_batch=1, flags=0):
    st = K.kfl_stage_create(K.model_cfg(model, 4096, max_batch), 0, 1, flags)
    _load(st, model)
    return st


def _prefill(st, n):
    """The return code of a prompt of n tokens (no kernel runs: the buffers are never read)."""
    pos = np.arange(n, dtype=np.int32)
    h = np.zeros(1, dtype=np.float32)
    return K.lib().kfl_stage_prefill(st.handle, pos.ctypes.data, h.ctypes.data, pos.ctypes.data, 0, n, h.ctypes.data,
                                     pos.ctypes.data, None)


def _matmul(T, k, n):
    a = np.zeros(4, dtype=np.float32)
    at = (a.ctypes.data + 15) // 16 * 16
    return K.lib().kfl_matmul_bf16w(at, T, k, k, at, n, at, (n + 3) // 4 * 4, None)


@pytest.mark.parametrize("model,n,kernel", [
    (SMALL, 40, "prefill_narrow_kernel"), (SMALL, 9, "prefill_narrow_kernel"), (QK, 40, "prefill_narrow_kernel"),
    (INT4, 40, "prefill_narrow4_kernel"), (WIDE, 200, "prefill_gemm_persistent"),
    (WIDE, 600, "prefill_attn_kernel")])
def test_prompts_on_a_second_device(dev, model, n, kernel):
    """The kernels' shared memory is opted in on each device that launches them."""
    for d in range(2):
        dev.cudaSetDevice(d)
        st = _stage(model)
        before = dev.fake_launches(kernel.encode())
        assert _prefill(st, n) == 0
        assert dev.fake_launches(kernel.encode()) > before
        K.kfl_stage_destroy(st)


@pytest.mark.parametrize("T", [40, 300])
def test_product_on_a_second_device(dev, T):
    for d in range(2):
        dev.cudaSetDevice(d)
        assert _matmul(T, 64, 256) == 0


@pytest.mark.parametrize("model,n", [(SMALL, 40), (INT4, 40), (WIDE, 200)])
def test_a_failed_opt_in_is_tried_again(dev, model, n):
    st = _stage(model)
    dev.fake_fail_optin(1)
    assert _prefill(st, n) < 0
    assert _prefill(st, n) == 0
    K.kfl_stage_destroy(st)


@pytest.mark.parametrize("model,n", [(QK, 40), (SMALL, 9), (SMALL, 40), (INT4, 40)])
def test_a_captured_prompt_keeps_its_workspace(dev, model, n):
    """A longer prompt after the capture leaves the memory that the captured graph uses alone; the
    stage's end gives all of it back."""
    st = _stage(model)
    assert _prefill(st, n) == 0
    dev.fake_capturing(1)
    assert _prefill(st, n) == 0
    dev.fake_capturing(0)
    dev.fake_mark()
    held = dev.fake_marked()
    assert _prefill(st, 700) == 0
    assert dev.fake_marked() == held
    K.kfl_stage_destroy(st)
    assert dev.fake_live() == 0


@pytest.mark.parametrize("captured", [False, True])
@pytest.mark.parametrize("model", [QK, SMALL])
def test_no_memory_for_a_larger_workspace(dev, model, captured):
    """A prompt whose workspace finds no memory leaves the smaller one in use and nothing else behind, does
    not try again while there is no more memory, and runs once there is."""
    st = _stage(model)
    assert _prefill(st, 40) == 0
    if captured:
        dev.fake_capturing(1)
        assert _prefill(st, 40) == 0
        dev.fake_capturing(0)
    held, kernel = dev.fake_live(), b"prefill_narrow_kernel"
    dev.fake_budget(held + (1 << 20))
    # a QK-norm stage's prompt goes as decode steps then, another's is refused
    dense, steps = dev.fake_launches(kernel), dev.fake_launches(b"decode graph")
    assert _prefill(st, 1500) == (0 if model.qk_norm else -3)
    assert dev.fake_launches(kernel) == dense
    assert (dev.fake_launches(b"decode graph") > steps) == model.qk_norm
    assert dev.fake_live() == held
    assert _prefill(st, 40) == 0
    assert dev.fake_launches(kernel) > dense  # densely again, on the workspace it had
    calls = dev.fake_mallocs()
    _prefill(st, 1500)
    assert dev.fake_mallocs() == calls and dev.fake_live() == held
    dev.fake_budget(1 << 40)
    dense = dev.fake_launches(kernel)
    assert _prefill(st, 1500) == 0 and dev.fake_launches(kernel) > dense
    K.kfl_stage_destroy(st)
    assert dev.fake_live() == 0


@pytest.mark.parametrize("call", ["load", "long prompt"])
def test_memory_kept_by_the_product_is_given_back(dev, call):
    """What kfl_matmul_bf16w's pool keeps stands in no other allocation's way: host weights' copies while they
    load, the fp16 copies of an int4 stage's long prompts."""
    model = dataclasses.replace(WIDE, weight_fmt="int4_g64")
    for known in (False, True):
        st = _stage(model)
        run = {"load": lambda: _load(st, model), "long prompt": lambda: _prefill(st, 600)}[call]
        if known:
            assert _matmul(2048, 8192, 8192) == 0 and dev.fake_pool_held() >= 32 << 20
            dev.fake_budget(peak)
        dev.fake_peak()
        assert not run()
        peak = dev.fake_peak()
        K.kfl_stage_destroy(st)


@pytest.mark.parametrize("T,k,n", [(300, 8191, 8191), (2048, 18943, 18943), (40, 18943, 30000), (8192, 18944, 64), (40, 64, 64)])
def test_the_product_keeps_no_more_than_its_threshold(dev, T, k, n):
    """The pool holds 512 MiB at most after a call; copied weights (here up to 1.1 GB) go through it in slabs, and
    what is larger (x's terms of 8192 tokens) stays out of it and is given back."""
    for _ in range(2):
        assert _matmul(T, k, n) == 0
        assert dev.fake_pool_held() <= 512 << 20 and dev.fake_live() == 0
    if n > 8192:
        assert dev.fake_launches(b"tile_rows_kernel") > 2


@pytest.mark.parametrize("d,f,n,decoded", [(128, 256, 128, True), (128, 256, 129, False), (3584, 18944, 300, True),
                                           (3584, 18944, 400, False), (5120, 27648, 512, True), (5120, 27648, 513, False)])
def test_int4_prompts_decode_in_the_product_while_that_is_cheaper(dev, d, f, n, decoded):
    st = _stage(dataclasses.replace(INT4, d_model=d, ffn=f))
    assert _prefill(st, n) == 0
    assert (dev.fake_launches(b"prefill_narrow4_kernel") > 0) == decoded
    assert (dev.fake_launches(b"dequant_int4_f16_kernel") > 0) != decoded
    K.kfl_stage_destroy(st)


def test_int4_prompts_without_memory_for_the_copies(dev):
    """Up to 512 tokens then decode in the products; longer ones are refused until there is memory."""
    st = _stage(dataclasses.replace(INT4, d_model=3584, ffn=18944))
    assert _prefill(st, 300) == 0
    dev.fake_budget(dev.fake_live() + (400 << 20))  # the longer workspace, but no two copies of 272 MB
    assert _prefill(st, 400) == 0 and dev.fake_launches(b"dequant_int4_f16_kernel") == 0
    assert _prefill(st, 520) == -3
    dev.fake_budget(1 << 40)
    assert _prefill(st, 520) == 0 and dev.fake_launches(b"dequant_int4_f16_kernel") > 0
    K.kfl_stage_destroy(st)
    assert dev.fake_live() == 0


@pytest.mark.parametrize("model,n,kernels", [c[1:] for c in CASES], ids=[c[0] for c in CASES])
def test_the_long_prompts_tests_reach_their_kernels(dev, model, n, kernels):
    st = _stage(model, 2, K.KFL_IS_HEAD)
    assert _prefill(st, n) == 0
    missing = [k for k in kernels if dev.fake_launches(k.encode()) == 0]
    assert not missing
    K.kfl_stage_destroy(st)
