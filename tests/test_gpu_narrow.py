"""GPU parity of the prefill's few-token matrix product (stream-K over the SMs, weight rows as the MMA's
rows) at the edges of its tiles: token groups of 16 up to 128, row tiles of 128 and (many rows, more
than 64 tokens) 256, one K block of 64 up to several per CTA, with ragged tails.

The plain product against fp64: x carried to about 2^-16 relative by its two terms, fp32
accumulation, so each element within 1e-4 of its row's RMS plus 2^-14 relative (the bar of the
128-token tiles).  Through a stage: the prefill's bar against the oracle.
"""
import dataclasses

import numpy as np
import pytest
import torch

from gpu_helpers import Pair, ensure_built
from paper_2609_34045_gb300 import stage as K
from test_gpu_parity import RAGGED, RAGGED128
from test_gpu_prefill import _prefill

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    ensure_built()
    torch.cuda.init()


@pytest.mark.parametrize("T,Kd,N", [(1, 64, 1), (16, 72, 129), (17, 128, 300), (48, 1000, 40), (64, 3584, 640),
                                    (65, 200, 29300), (127, 520, 384), (128, 136, 29185), (128, 2048, 1000)])
def test_product_matches_fp64(T, Kd, N):
    rng = np.random.default_rng(T * 31 + Kd * 7 + N)
    x = rng.standard_normal((T, Kd)).astype(np.float32)
    w = torch.from_numpy((rng.standard_normal((N, Kd)) * 0.05).astype(np.float32)).to(torch.bfloat16)
    ldy = (N + 3) // 4 * 4
    y = torch.full((T, ldy), 7.0, dtype=torch.float32, device="cuda")
    wd = w.view(torch.int16).cuda().contiguous()
    for _ in range(2):  # the second call finds whatever the first left in the tickets
        K.kfl_matmul_bf16w(torch.from_numpy(x).cuda(), T, Kd, Kd, wd, N, y, ldy,
                           torch.cuda.current_stream().cuda_stream)
    got = y.cpu().numpy()
    ref = x.astype(np.float64) @ w.to(torch.float64).numpy().T
    rms = np.sqrt(np.mean(ref * ref, axis=1, keepdims=True))
    assert np.all(np.abs(got[:, :N] - ref) <= 1e-4 * rms + 2.0 ** -14 * np.abs(ref))
    assert np.all(got[:, N:] == 7.0)


@pytest.mark.parametrize("model,n", [(RAGGED, 16), (RAGGED, 65), (RAGGED, 128), (RAGGED128, 33),
                                     (dataclasses.replace(RAGGED, vocab=30000), 70)])
def test_prefill_matches_the_oracle(model, n, monkeypatch):
    monkeypatch.setenv("KFL_PREFILL_DENSE_MIN", "1")
    p = Pair(model, 0, 2, K.KFL_IS_HEAD, 2, (5, 30), 192, seed=43, max_batch=2)
    for _ in range(2):
        _prefill(p, 1, 30, n, 43, True)
    p.compare_kv()
    p.close()
