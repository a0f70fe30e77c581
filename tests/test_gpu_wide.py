"""GPU checks of the long prompts' kernels: the matrix products on 128-token tiles (bf16 and dequantized int4
weights) and what stands between them."""
import numpy as np
import pytest
import torch

from gpu_helpers import ensure_built
from paper_2609_34045_gb300 import stage as K
from paper_2609_34045_gb300 import workload as wl

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    ensure_built()
    torch.cuda.init()


def _gaussian(g, *shape, std=0.02):
    return torch.randn(shape, generator=g, device="cuda", dtype=torch.bfloat16).mul_(std)


def _codes(g, rows, cols):
    """int4 words of uniform codes with scales of 2^-6 (fp16 holds every weight), and the weights."""
    codes = torch.randint(-8, 8, (rows, cols), generator=g, device="cuda", dtype=torch.int32)
    words = torch.zeros((rows, cols // 8), device="cuda", dtype=torch.int32)
    for j in range(8):
        words |= (codes[:, j::8] & 15) << (4 * j)
    return (words, torch.full((rows, cols // 64), 2.0 ** -6, device="cuda", dtype=torch.bfloat16)), codes


@pytest.mark.parametrize("fmt,d,f,n,bar", [("bf16", 2560, 18944, 2048, 2.9e-5), ("int4_g64", 5120, 29568, 900, 3.7e-5)])
def test_error_of_a_long_residual_product(fmt, d, f, n, bar):
    """The MLP of one block (attention adds nothing) whose down projection has more than a round of tiles, against
    64 bits.  A tensor-core accumulation truncates: 3.2e-8 of the sum per 16 K values.  Gate and up (K = d)
    each lose d / 16 of these, the down projection the 240 or 232 of its equal chunks; x's and a's terms
    leave 4e-6 at most.  The bar is their sum and a third."""
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
