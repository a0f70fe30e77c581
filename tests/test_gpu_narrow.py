"""GPU parity of the prefill's few-token matrix product (stream-K over the SMs, weight rows as the MMA's
rows) at the edges of its tiles: token groups of 16 up to 128, row tiles of 128 and (a stage's many rows,
more than 64 tokens) 256, one K block of 64 up to several per CTA, with ragged tails; and its int4 form,
which decodes the weights on the way (256-row tiles, K units of 128).

The plain product against fp64: x carried to about 2^-16 relative by its two terms, fp32
accumulation, so each element within 1e-4 of its row's RMS plus 2^-14 relative (the bar of the
128-token tiles).  Through a stage: the prefill's bar against the oracle.
"""
import dataclasses

import numpy as np
import pytest
import torch

import oracle
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


@pytest.mark.parametrize("T,Kd,N", [(1, 64, 1), (16, 72, 129), (17, 128, 300), (48, 1000, 40), (64, 3584, 640),
                                    (65, 200, 29300), (127, 520, 384), (128, 136, 29185), (128, 2048, 1000),
                                    # weight rows that TMA cannot address (K % 8 != 0) are copied to tiles first
                                    (5, 67, 130), (129, 203, 513), (130, 200, 513)])
def test_product_matches_fp64(T, Kd, N):
    rng = np.random.default_rng(T * 31 + Kd * 7 + N)
    x = rng.standard_normal((T, Kd)).astype(np.float32)
    w = torch.from_numpy((rng.standard_normal((N, Kd)) * 0.05).astype(np.float32)).to(torch.bfloat16)
    ldy = (N + 3) // 4 * 4
    y = torch.full((T, ldy), 7.0, dtype=torch.float32, device="cuda")
    wd = w.view(torch.int16).cuda().contiguous()
    # what the call finds in the pool's memory: another shape's terms and partial sums, far from these
    big = torch.full((T + 3, Kd + 64), 3e38, device="cuda")
    K.kfl_matmul_bf16w(big, T + 3, Kd + 64, Kd + 64, torch.full((N + 5, Kd + 64), 0x7F00, dtype=torch.int16, device="cuda"),
                       N + 5, torch.zeros((T + 3, ldy + 8), device="cuda"), ldy + 8, torch.cuda.current_stream().cuda_stream)
    K.kfl_matmul_bf16w(torch.from_numpy(x).cuda(), T, Kd, Kd, wd, N, y, ldy, torch.cuda.current_stream().cuda_stream)
    got = y.cpu().numpy()
    ref = x.astype(np.float64) @ w.to(torch.float64).numpy().T
    rms = np.sqrt(np.mean(ref * ref, axis=1, keepdims=True))
    assert np.all(np.abs(got[:, :N] - ref) <= 1e-4 * rms + 2.0 ** -14 * np.abs(ref))
    assert np.all(got[:, N:] == 7.0)


@pytest.mark.parametrize("T", [1, 64, 128, 129])
def test_product_error_of_a_long_k(T):
    """Both forms of the plain product at K = 18944: x's two terms leave 2^-18 of it (rms 2e-6), and the sums
    are fp32 ones, so 1e-5 of the result (2-norm).  Left in the tensor core's accumulator, which truncates
    (3e-8 per 16 products), they were 1.5e-5 off."""
    k = n = 18944
    g = torch.Generator(device="cuda").manual_seed(T)
    x = torch.randn((T, k), generator=g, device="cuda")
    w = torch.randn((n, k), generator=g, device="cuda", dtype=torch.bfloat16).mul_(0.02)
    y = torch.zeros((T, n), device="cuda")
    K.kfl_matmul_bf16w(x, T, k, k, w.view(torch.int16), n, y, n, torch.cuda.current_stream().cuda_stream)
    ref = torch.cat([x.double() @ w[r:r + 2048].double().t() for r in range(0, n, 2048)], dim=1)
    err = float((y.double() - ref).norm() / ref.norm())
    assert err <= 1e-5, err


@pytest.mark.parametrize("model,n", [(RAGGED, 16), (RAGGED, 65), (RAGGED, 128), (RAGGED128, 33),
                                     (dataclasses.replace(RAGGED, vocab=30000), 70), (RAGGED_INT4, 16),
                                     (RAGGED_INT4, 65), (RAGGED_INT4, 100), (RAGGED_INT4, 129)])
def test_prefill_matches_the_oracle(model, n, monkeypatch):
    # (the bar holds the attention's bf16 q and softmax weights too: at d_model 448, ffn 1024 they alone
    # give 1.02e-2 to 3.3e-2 of the RMS over three seeds, the same to 2e-6 with the 128-token tiles)
    monkeypatch.setenv("KFL_PREFILL_DENSE_MIN", "1")
    p = Pair(model, 0, 2, K.KFL_IS_HEAD, 2, (5, 30), 192, seed=43, max_batch=2)
    for _ in range(2):
        _prefill(p, 1, 30, n, 43, True)
    p.compare_kv()
    p.close()


@pytest.mark.parametrize("model,d,n", [(RAGGED, 8320, 18),  # past what the norm's threads hold in registers
                                       (RAGGED128, 8320, 130), (dataclasses.replace(RAGGED, qk_norm=True), 8264, 100),
                                       (RAGGED_INT4, 16640, 33),
                                       (RAGGED, 16648, 200),
                                       (RAGGED, 32776, 17)])  # too many row tiles for the residual sums' norm
def test_long_rows_match_the_oracle(model, d, n, monkeypatch):
    """Residual sums and RMSNorm of rows at the edges of their kernels' ranges.  The attention norm's gain is
    scaled by about (320 / d)^(1/2), so q and k keep the size they have at d_model 320, where the bar
    comes from.  Unscaled (weights of 0.02), scores at d_model 16648 spread by (0.02^2 d) sqrt(64) / 8 =
    6.7 and a softmax picks single keys: a K element a bf16 step (2^-8 of 2.6) over then moves a
    score by 2.6 * 2^-8 * 2.6 / 8, a weight by 0.3 % of itself, and several of them a row by 1e-2."""
    monkeypatch.setenv("KFL_PREFILL_DENSE_MIN", "1")
    plain, scale = wl.layer_weights, np.float32(2.0 ** -round(np.log2(d / 320) / 2))

    def layer_weights(*a):
        w = plain(*a)
        w["attn_norm"] = wl.f32_to_bf16_bits(wl.bf16_bits_to_f32(w["attn_norm"]) * scale)
        return w

    monkeypatch.setattr(wl, "layer_weights", layer_weights)
    p = Pair(dataclasses.replace(model, d_model=d, vocab=300), 0, 2, K.KFL_IS_HEAD, 2, (5, 30), 256, seed=59, max_batch=2)
    _prefill(p, 1, 30, n, 59, True)
    p.compare_kv()
    p.close()


def test_int4_scales_below_the_fp16_normals():
    """Scales that fp16 cannot hold exactly (2^-14 and below, bf16 significands) take the fp32 product
    of code and scale.  The down projection's are set to 2^-16 and below: fp16 weights of 2^-24
    resolution then carry about 2^-9 relative, averaged over 704 products, so the block's
    contribution stays within 1e-2 of its RMS."""
    m, n, seed = RAGGED_INT4, 40, 47
    w = wl.layer_weights(m, 0, seed)
    words, scales = w["wd"]
    w["wv"] = (np.zeros_like(w["wv"][0]), w["wv"][1])  # attention adds nothing
    w["wd"] = (words, wl.f32_to_bf16_bits(wl.bf16_bits_to_f32(scales) * np.float32(2.0 ** -9)))
    st = K.kfl_stage_create(K.model_cfg(m, 64, 1), 0, 1, 0)
    K.kfl_stage_load_layer(st, 0, w, on_device=False)
    ora = oracle.OracleStage(m, 0, 1, False, False, 1, 64)
    ora.load_layer(0, w)
    hidden = wl.hidden_in(m, 0, n, seed) * np.float32(2.0 ** -8)
    pos = np.arange(n, dtype=np.int32)
    ref = ora.prefill(0, pos, hidden_in=hidden)["hidden_out"]
    out = torch.zeros(n, m.d_model, device="cuda")
    K.kfl_stage_prefill(st, None, torch.tensor(hidden, device="cuda"), torch.tensor(pos, device="cuda"), 0, n, out, None,
                        torch.cuda.current_stream().cuda_stream)
    assert K.kfl_stage_status(st) == 0
    got = out.cpu().numpy()
    # the block's contribution alone (the sum with the hidden states is fp32: exact to 1e-7 of them)
    delta = ref - hidden
    rms = np.sqrt(np.mean(delta * delta, axis=1, keepdims=True))
    assert np.all(np.abs(got - hidden - delta) <= 1e-2 * rms)
    K.kfl_stage_destroy(st)


@pytest.mark.parametrize("model,n,start,max_batch", [
    (RAGGED, 5, 30, 4), (RAGGED, 15, 100, 1), (RAGGED128, 9, 7, 4),
    (dataclasses.replace(RAGGED, qk_norm=True), 17, 30, 2),
    (dataclasses.replace(RAGGED128, qk_norm=True), 165, 300, 4)])  # three token tiles, keys split over a cluster
def test_dense_at_decode_precision(model, n, start, max_batch, monkeypatch):
    """Prompts that run densely in place of decode steps (QK-norm stages; others longer than one step but
    shorter than 16 tokens): the oracle's bar, and the decode steps' results.  Both sides carry
    activations to 2^-22 or better and q and the softmax weights to 2^-17, so they differ where a
    K or V element lands on the other side of a bf16 rounding (2^-8 of it): a few of the elements
    that a row attends to, 1e-3 of its RMS at most (the bar allows ten times that)."""
    monkeypatch.delenv("KFL_PREFILL_DENSE_MIN", raising=False)
    p = Pair(model, 0, 2, 0, 2, (5, start), 512, seed=53, max_batch=max(2, max_batch))
    K.kfl_stage_debug_capture(p.st, None)  # observed stages keep the decode steps
    _prefill(p, 1, start, n, 53, False)
    p.compare_kv()
    hidden = torch.tensor(wl.hidden_in(model, 3, n, 53), dtype=torch.float32, device="cuda")
    pos = torch.arange(start, start + n, dtype=torch.int32, device="cuda")
    out = [torch.zeros(n, model.d_model, device="cuda") for _ in range(2)]
    for o, line in zip(out, (None, str(1 << 30))):
        if line:
            monkeypatch.setenv("KFL_PREFILL_DENSE_MIN", line)
        K.kfl_stage_prefill(p.st, None, hidden, pos, 1, n, o, None, torch.cuda.current_stream().cuda_stream)
    assert K.kfl_stage_status(p.st) == 0
    dense, steps = (o.cpu().numpy().astype(np.float64) for o in out)
    rms = np.sqrt(np.mean(steps * steps, axis=1, keepdims=True))
    assert np.all(np.abs(dense - steps) <= 1e-3 * rms)
    p.close()


@pytest.mark.parametrize("n", [9, 40])
def test_nan_keys_reach_the_output(n):
    """A key block of NaN alone is one CTA's whole share of the split keys: its rows' scores have no largest one,
    and the merge takes them in all the same."""
    m = wl.ModelShape(n_layers_total=1, d_model=128, n_heads=2, n_kv_heads=1, head_dim=64, ffn=256, vocab=300)
    st = K.kfl_stage_create(K.model_cfg(m, 512, 4), 0, 1, 0)
    K.kfl_stage_load_layer(st, 0, wl.layer_weights(m, 0, 3), on_device=False)
    k, v = (torch.randn(1, 200, 64, device="cuda").to(torch.bfloat16) for _ in range(2))
    k[:, 64:128] = float("nan")
    K.kfl_kv_write(st, 0, 0, k, v, 200, True)
    out = torch.zeros(n, m.d_model, device="cuda")
    K.kfl_stage_prefill(st, None, torch.randn(n, m.d_model, device="cuda"),
                        torch.arange(200, 200 + n, dtype=torch.int32, device="cuda"), 0, n, out, None,
                        torch.cuda.current_stream().cuda_stream)
    assert torch.isnan(out).all()
    K.kfl_stage_destroy(st)


@pytest.mark.parametrize("model,n", [(RAGGED, 9), (RAGGED, 40), (dataclasses.replace(RAGGED, qk_norm=True), 40),
                                     (RAGGED_INT4, 40), (RAGGED_INT4, 200)])
def test_captured_prompt_after_a_longer_one(model, n):
    """A captured prompt replayed after a longer prompt has outgrown its workspace gives what it gave."""
    st = K.kfl_stage_create(K.model_cfg(model, 1024, 4), 0, 1, 0)
    K.kfl_stage_load_layer(st, 0, wl.layer_weights(model, 0, 3), on_device=False)
    hidden = torch.randn(700, model.d_model, device="cuda")
    pos = torch.arange(700, dtype=torch.int32, device="cuda")
    out = torch.zeros(700, model.d_model, device="cuda")
    run = lambda t: K.kfl_stage_prefill(st, None, hidden, pos, 1, t, out, None, torch.cuda.current_stream().cuda_stream)
    run(n)
    first = out[:n].clone()
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        run(n)
    run(700)
    # (what the longer prompt would have freed is likely to be given to these)
    filler = [torch.full((1 << 20,), float("nan"), device="cuda") for _ in range(64)]
    out.zero_()
    graph.replay()
    torch.cuda.synchronize()
    assert K.kfl_stage_status(st) == 0
    assert torch.equal(out[:n], first)
    del filler, graph
    K.kfl_stage_destroy(st)
