"""GPU checks of the long prompts' kernels: the matrix products on 128-token tiles (bf16 and dequantized int4
weights), whole and cut, and the attention without pairs.

CASES are models whose prompts take them: bf16 ones with an FFN wide enough that its tiles reach every SM, int4
ones past the few-token line; test_fake_device.py checks on the CPU that they do.
"""
import dataclasses

import numpy as np
import pytest
import torch

from gpu_helpers import Pair, ensure_built
from paper_2609_34045_gb300 import stage as K
from paper_2609_34045_gb300 import workload as wl
from test_gpu_parity import RAGGED, RAGGED128, RAGGED_INT4
from test_gpu_prefill import _prefill

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    ensure_built()
    torch.cuda.init()


SMALL = wl.ModelShape(n_layers_total=1, d_model=128, n_heads=2, n_kv_heads=1, head_dim=64, ffn=9800, vocab=300)
GEMM = "prefill_gemm_persistentILi%dELb0"  # mode: 1 residual, 2 SwiGLU, 3 Q/K/V, 4 argmax
CUT = "wide_reduce_kernelILi%d"
ALL = [GEMM % m for m in (1, 2, 3, 4)]
# (name, model, tokens, kernels that it reaches); ragged in tokens, in the rows of every matrix and in K
CASES = [
    ("bf16-200", dataclasses.replace(RAGGED, ffn=9800), 200, ALL + [CUT % 1, "prefill_attn_kernelILi64ELb1"]),
    ("bf16-530", dataclasses.replace(RAGGED, ffn=9800), 530, ALL + [CUT % 1, "prefill_attn_kernelILi64ELb0"]),
    ("bf16-hd128-530", dataclasses.replace(RAGGED128, ffn=9800), 530, ALL + [CUT % 1, "prefill_attn_kernelILi128ELb0"]),
    ("bf16-two-passes", SMALL, 2100, ALL + [CUT % 1, "prefill_attn_kernelILi64ELb0"]),
    ("int4-200", RAGGED_INT4, 200, ALL + ["dequant_int4", "prefill_attn_kernelILi64ELb1"]),
    # K long enough that the tiles of every product are cut
    ("int4-cut-200", dataclasses.replace(RAGGED_INT4, d_model=1856, ffn=2048), 200,
     ALL + [CUT % 1, CUT % 2, CUT % 3, CUT % 4, "dequant_int4"]),
    ("int4-530", RAGGED_INT4, 530, ALL + ["dequant_int4", "prefill_attn_kernelILi64ELb0"]),
    ("int4-two-passes", dataclasses.replace(SMALL, ffn=320, weight_fmt="int4_g64"), 2100, ALL + ["dequant_int4"]),
    # decoded in the few-token product, in two token tiles
    ("int4-decoded-150", dataclasses.replace(RAGGED_INT4, ffn=30016), 150, ["prefill_narrow4_kernelILi%d" % m for m in (1, 2, 3, 4)]),
]


@pytest.mark.parametrize("model,n", [c[1:3] for c in CASES], ids=[c[0] for c in CASES])
def test_long_prompt_matches_the_oracle(model, n, monkeypatch):
    """The bar of the other prompts, from hidden states of RMS 1 and not an embedding's of 0.02: without pairs, q and
    the softmax weights are rounded to bf16 (2^-9), and beside an embedding attention is nearly all of the
    residual stream, whose worst element of 530 tokens x 320 was then 1.24e-2 of its token's RMS over three seeds (2-norm
    1.6e-3), the same to 2 % with the kernels of before the tiles were shared.  Here the worst of three seeds is
    7.8e-4 (1.0e-4 where attention has pairs), so a second call is held to 2e-3: a 128-token tile's
    share of a product is 1e-2 and more.  The attention norm's gain is scaled by (320 / d)^(1/2) or so, which
    keeps q and k at the size they have at d_model 320, where the first bar comes from (test_gpu_narrow.py
    says why)."""
    plain, scale = wl.layer_weights, np.float32(2.0 ** -max(0, round(np.log2(model.d_model / 320) / 2)))

    def layer_weights(*a):
        w = plain(*a)
        w["attn_norm"] = wl.f32_to_bf16_bits(wl.bf16_bits_to_f32(w["attn_norm"]) * scale)
        return w

    monkeypatch.setattr(wl, "layer_weights", layer_weights)
    layers = min(2, model.n_layers_total)
    p = Pair(model, 0, layers, K.KFL_LOGITS_OUT, 2, (5, 30), (30 + n + 63) // 64 * 64, seed=61, max_batch=2)
    ref = _prefill(p, 1, 30, n, 61, False)["hidden_out"]
    p.compare_kv()
    hidden = torch.tensor(wl.hidden_in(model, 3, n, 61), dtype=torch.float32, device="cuda")
    out, nxt = torch.zeros(n, model.d_model, device="cuda"), torch.zeros(n, dtype=torch.int32, device="cuda")
    K.kfl_stage_prefill(p.st, None, hidden, torch.arange(30, 30 + n, dtype=torch.int32, device="cuda"), 1, n, out, nxt,
                        torch.cuda.current_stream().cuda_stream)
    err = np.abs(out.cpu().numpy() - ref).max(axis=1) / np.sqrt(np.mean(ref * ref, axis=1))
    assert err.max() <= 2e-3, (int(err.argmax()), err.max())
    p.close()


def _gaussian(g, *shape, std=0.02):
    return torch.randn(shape, generator=g, device="cuda", dtype=torch.bfloat16).mul_(std)


def _codes(g, rows, cols):
    """int4 words of uniform codes with scales of 2^-6 (fp16 holds every weight), and the weights."""
    codes = torch.randint(-8, 8, (rows, cols), generator=g, device="cuda", dtype=torch.int32)
    words = torch.zeros((rows, cols // 8), device="cuda", dtype=torch.int32)
    for j in range(8):
        words |= (codes[:, j::8] & 15) << (4 * j)
    return (words, torch.full((rows, cols // 64), 2.0 ** -6, device="cuda", dtype=torch.bfloat16)), codes


@pytest.mark.parametrize("fmt,d,f,n", [("bf16", 2560, 18944, 2048), ("int4_g64", 5120, 29568, 900),
                                       ("bf16", 16648, 9800, 200)])  # rows longer than the norm's registers
def test_error_of_a_long_mlp(fmt, d, f, n):
    """The MLP of one block (attention adds nothing) whose products have more than a round of tiles, against 64
    bits.  A tensor-core accumulation truncates: 3.2e-8 of the sum per 16 K values.  Gate and up (K = d)
    each lose d / 16 of these, the down projection those of its chunks of 4096 at most; x's and a's terms
    leave 4e-6.  The bar is their sum and a third."""
    bar = 4 / 3 * (3.2e-8 * (2 * d / 16 + min(f, 4096) / 16) + 4e-6)
    g = torch.Generator(device="cuda").manual_seed(d)
    m = wl.ModelShape(n_layers_total=1, d_model=d, n_heads=2, n_kv_heads=1, head_dim=64, ffn=f, vocab=300, weight_fmt=fmt)
    ones = lambda k: torch.ones(k, device="cuda", dtype=torch.bfloat16)
    w, ref = {"attn_norm": ones(d), "ffn_norm": ones(d), "q_norm": ones(64), "k_norm": ones(64)}, {}
    for name, rows, cols in (("wq", 128, d), ("wk", 64, d), ("wv", 64, d), ("wo", d, 128), ("wg", f, d), ("wu", f, d),
                             ("wd", d, f)):
        if fmt == "bf16":
            w[name] = ref[name] = _gaussian(g, rows, cols)
        else:
            w[name], codes = _codes(g, rows, cols)
            ref[name] = codes.to(torch.bfloat16).mul_(2.0 ** -6)
    (w["wo"] if fmt == "bf16" else w["wo"][0]).zero_()
    st = K.kfl_stage_create(K.model_cfg(m, n, 1), 0, 1, 0)
    torch.cuda.synchronize()
    K.kfl_stage_load_layer(st, 0, w, on_device=True)
    h = _gaussian(g, n, d, std=2.0 ** -8).float()
    out = torch.zeros(n, d, device="cuda")
    pos = torch.arange(n, dtype=torch.int32, device="cuda")
    K.kfl_stage_prefill(st, None, h, pos, 0, n, out, None, torch.cuda.current_stream().cuda_stream)
    assert K.kfl_stage_status(st) == 0
    x = h.double()
    x = x / torch.sqrt((x * x).mean(-1, keepdim=True) + m.rms_eps)
    y = torch.zeros(n, d, device="cuda", dtype=torch.float64)
    for r in range(0, f, 2048):
        s = slice(r, r + 2048)
        gate = x @ ref["wg"][s].double().t()
        y += (gate / (1 + torch.exp(-gate)) * (x @ ref["wu"][s].double().t())) @ ref["wd"][:, s].double().t()
    err = float((out.double() - h.double() - y).norm() / y.norm())
    K.kfl_stage_destroy(st)
    assert err <= bar, err


def test_rounding_of_a_long_value_projection():
    """V rows of a product with more than a round of tiles and K = 8192, against 64 bits rounded to bf16: those
    that land beside it.  Truncation of chunks of K = 2048 takes 4.1e-6 of a value's size, of the whole K 1.6e-5;
    a bf16 step is 5.4e-3 (1 / 185) of the value on average, so 0.076 % and 0.30 % would land a step lower.
    Twice that for values that are normal around zero: what they lose goes by their partial sums, of the
    RMS's size, and their steps by their own.  (x's terms, 2^-22, add 0.01 %.)  The bar is between the two."""
    d, n, kv = 8192, 900, 1024
    g = torch.Generator(device="cuda").manual_seed(5)
    m = wl.ModelShape(n_layers_total=1, d_model=d, n_heads=24, n_kv_heads=8, head_dim=128, ffn=256, vocab=300,
                      weight_fmt="int4_g64")
    w = {k: torch.ones(128 if k in ("q_norm", "k_norm") else d, device="cuda", dtype=torch.bfloat16)
         for k in ("attn_norm", "ffn_norm", "q_norm", "k_norm")}
    for name, rows, cols in (("wq", 3072, d), ("wk", kv, d), ("wv", kv, d), ("wo", d, 3072), ("wg", 256, d), ("wu", 256, d),
                             ("wd", d, 256)):
        w[name], codes = _codes(g, rows, cols)
        if name == "wv":
            wv = codes.double().mul_(2.0 ** -6)
    st = K.kfl_stage_create(K.model_cfg(m, 960, 1), 0, 1, 0)
    torch.cuda.synchronize()
    K.kfl_stage_load_layer(st, 0, w, on_device=True)
    h = _gaussian(g, n, d, std=1.0).float()
    out = torch.zeros(n, d, device="cuda")
    K.kfl_stage_prefill(st, None, h, torch.arange(n, dtype=torch.int32, device="cuda"), 0, n, out, None,
                        torch.cuda.current_stream().cuda_stream)
    k, v = (torch.zeros(8, 960, 128, device="cuda", dtype=torch.bfloat16) for _ in range(2))
    K.kfl_kv_read(st, 0, 0, k, v, True)
    x = h.double()
    x = x / torch.sqrt((x * x).mean(-1, keepdim=True) + m.rms_eps)
    ref = (x @ wv.t()).float().bfloat16().view(n, 8, 128).transpose(0, 1)
    K.kfl_stage_destroy(st)
    beside = float((v[:, :n] != ref).double().mean())
    assert beside <= 2.5e-3, beside
