"""What a user of the stage engine has it do, as cases that can be timed and compared.

A case is one call of a public entry point on seeded inputs: a decode step of a stage
(``kfl_stage_decode``), a prompt's prefill through a stage (``kfl_stage_prefill``), or the
prefill's matrix product on its own (``kfl_matmul_bf16w``).  ``prepare`` makes what a program holds
before the call (the loaded stage with its filled KV cache, the input and output buffers),
``run`` is the call, and ``exact`` recomputes its outputs in 64 bits with plain torch.

Shapes are those of the workload recipes in ``paper_2609_34045_gb300/workload.py`` and of the GPU
tests, with fewer blocks where the blocks are alike: a stage's time is its blocks' times added up,
and every case's weights (but the tiny model's) are larger than L2, so each pass streams them from HBM.  Weights are normal around zero, int4 ones as a
quantiser would leave them.
"""
from __future__ import annotations

import math

import torch

from paper_2609_34045_gb300 import stage as K
from paper_2609_34045_gb300 import workload as wl

# d_model, query heads, KV heads, head_dim, FFN width, vocabulary
DIMS = {
    "tiny": (512, 8, 2, 64, 1408, 4096),
    "ragged": (320, 6, 2, 64, 704, 1000),
    "7B": (3584, 28, 4, 128, 18944, 152064),
    "32B": (5120, 64, 8, 128, 27648, 152064),
    "72B": (8192, 64, 8, 128, 29568, 152064),
}
EPS, THETA = 1e-6, 1e6
INT4_STD = 2.5  # codes of a quantised normal weight: most of [-8, 7] is used, the ends are rare


def _decode(name, model, blocks, contexts, fmt="bf16", embed=False, logits=False, qk_norm=False):
    return {"name": name, "op": "decode", "model": model, "fmt": fmt, "blocks": blocks, "embed": embed,
            "logits": logits, "qk_norm": qk_norm, "contexts": ",".join(str(c) for c in contexts)}


def _prefill(name, model, blocks, tokens, start=0, fmt="bf16", embed=False, logits=False, qk_norm=False):
    return {"name": name, "op": "prefill", "model": model, "fmt": fmt, "blocks": blocks, "embed": embed,
            "logits": logits, "qk_norm": qk_norm, "tokens": tokens, "start": start}


def listed():
    return [
        # the smallest call: a two-block model whose weights stay in L2, one token; launches and latency
        _decode("tiny-head-decode-b1", "tiny", 2, [128], embed=True, logits=True),
        # one user's token through a ring member's half of a 7B-shaped model
        _decode("7B-body-decode-b1", "7B", 14, [2048]),
        # one user's greedy token through a head stage: embedding, the last blocks, lm_head and argmax
        _decode("32B-head-decode-b1", "32B", 8, [4096], embed=True, logits=True),
        # four users at ragged contexts in one step of a bf16 body stage
        _decode("72B-body-decode-b4-ragged", "72B", 4, [512, 1536, 3072, 4096]),
        # the int4 model at a long context, alone and with every slot taken
        _decode("72B-int4-decode-b1", "72B", 8, [8192], fmt="int4"),
        _decode("72B-int4-head-decode-b4", "72B", 4, [8192, 8192, 8192, 8192], fmt="int4", embed=True, logits=True),
        # a chat turn: a short prompt appended to a filled context
        _prefill("7B-prefill-43-at-700", "7B", 4, 43, start=700),
        # an ordinary prompt through the blocks before the head's return leg, lm_head over its tokens included
        _prefill("7B-tail-prefill-500", "7B", 2, 500, logits=True),
        # the longest prompt of one dense pass
        _prefill("7B-prefill-2048", "7B", 4, 2048),
        # a model with QK-norm (the family that the paper serves): an ordinary prompt
        _prefill("7B-qknorm-prefill-200", "7B", 2, 200, qk_norm=True),
        # the int4 model's prompts: a short one and a long ragged one
        _prefill("72B-int4-prefill-100", "72B", 2, 100, fmt="int4"),
        _prefill("72B-int4-prefill-900", "72B", 2, 900, fmt="int4"),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    """Another case of the same ranges: decode steps of 1 to 4 users at 16 to 8192 positions, prompts
    of 3 to 2048 tokens at any start, both weight formats, head and body stages, QK-norm, every
    model's shapes, and plain products of odd sizes."""
    kind = rng.choice(["decode", "decode", "prefill", "prefill", "prefill", "matmul"])
    if kind == "matmul":
        t = _log_int(rng, 1, 2048)
        return {"op": "matmul", "tokens": t, "k": _log_int(rng, 64, 18944), "n": _log_int(rng, 64, 18944),
                "pad": rng.randrange(0, 9)}
    model = rng.choice(["tiny", "ragged", "7B", "7B", "32B", "72B", "72B"])
    fmt = rng.choice(["bf16", "bf16", "int4"])
    small = model in ("tiny", "ragged")
    qk_norm = rng.random() < 0.2
    if kind == "decode":
        blocks = rng.randint(1, 2) if small else rng.randint(2, 4)
        batch = rng.randint(1, 4)
        c = _decode("", model, blocks, [_log_int(rng, 16, 8192) for _ in range(batch)], fmt=fmt,
                    embed=rng.random() < 0.3, logits=rng.random() < 0.3, qk_norm=qk_norm)
    else:
        blocks = rng.randint(1, 2)
        # prompts of QK-norm stages and of fewer than 16 tokens take decode steps: kept to a pass of
        # some tens of milliseconds
        tokens = _log_int(rng, 3, 300 if qk_norm else 2048 if fmt == "bf16" and model != "72B" else 900)
        logits = model == "7B" and tokens >= 300 and rng.random() < 0.5
        c = _prefill("", model, blocks, tokens, start=_log_int(rng, 1, 4096) - 1, fmt=fmt,
                     embed=not logits and rng.random() < 0.3, logits=logits, qk_norm=qk_norm)
    del c["name"]
    return c


# ------------------------------------------------------------------------------------- inputs

def _gen(seed, *tag):
    key = seed & 0xFFFFFFFF
    for t in tag:
        key = (key * 1000003 + t + 1) & 0x3FFFFFFFFFFFFFF
    return torch.Generator(device="cuda").manual_seed(key)


def _bf16(g, shape, std, mean=0.0):
    x = torch.randn(shape, generator=g, device="cuda", dtype=torch.bfloat16)
    return x.mul_(std).add_(mean) if mean else x.mul_(std)


def _matrix(fmt, g, rows, cols):
    if fmt == "bf16":
        return _bf16(g, (rows, cols), 0.02)
    words = torch.zeros((rows, cols // 8), device="cuda", dtype=torch.int32)
    for j in range(8):
        code = torch.randn(words.shape, generator=g, device="cuda", dtype=torch.bfloat16).mul_(INT4_STD)
        words |= (code.round_().clamp_(-8, 7).int() & 15) << (4 * j)
    scales = 0.02 / INT4_STD * (0.5 + torch.rand((rows, cols // 64), generator=g, device="cuda"))
    scales = scales.to(torch.bfloat16)
    return words, scales


def _layer(case, seed, l):
    d, hq, hkv, hd, f, _ = DIMS[case["model"]]
    g = _gen(seed, 1, l)
    w = {n: _bf16(g, (d,), 0.02, 1.0) for n in ("attn_norm", "ffn_norm")}
    for n in ("q_norm", "k_norm"):
        w[n] = _bf16(g, (hd,), 0.02, 1.0)
    for n, (rows, cols) in {"wq": (hq * hd, d), "wk": (hkv * hd, d), "wv": (hkv * hd, d), "wo": (d, hq * hd),
                            "wg": (f, d), "wu": (f, d), "wd": (d, f)}.items():
        w[n] = _matrix(case["fmt"], g, rows, cols)
    return w


def _head(case, seed):
    d, _, _, _, _, v = DIMS[case["model"]]
    w = {}
    if case["embed"]:
        w["embed"] = _bf16(_gen(seed, 2, 0), (v, d), 0.02)
    if case["logits"]:
        w["final_norm"] = _bf16(_gen(seed, 2, 1), (d,), 0.02, 1.0)
        # a vocabulary's rows differ in norm, as a trained unembedding's do
        spread = torch.exp(0.5 * torch.randn((v, 1), generator=_gen(seed, 2, 3), device="cuda")).to(torch.bfloat16)
        lm = _matrix(case["fmt"], _gen(seed, 2, 2), v, d)
        w["lm_head"] = lm.mul_(spread) if case["fmt"] == "bf16" else (lm[0], lm[1].mul_(spread))
    return w


def _kv(case, seed, l, user, length):
    _, _, hkv, hd, _, _ = DIMS[case["model"]]
    g = _gen(seed, 3, l, user)
    return _bf16(g, (hkv, length, hd), 1.0), _bf16(g, (hkv, length, hd), 1.0)


def _io(case, seed, n):
    """Token ids or hidden states of n rows: bf16 values held as fp32, as a ring member receives them."""
    d, _, _, _, _, v = DIMS[case["model"]]
    g = _gen(seed, 4)
    if case["embed"]:
        return torch.randint(0, v, (n,), generator=g, device="cuda", dtype=torch.int32), None
    return None, _bf16(g, (n, d), 1.0).float()


def _users(case):
    """Filled KV length of each user slot, rows of the call, their positions and their user."""
    if case["op"] == "decode":
        ctx = [int(c) for c in case["contexts"].split(",")]
        return ctx, len(ctx), ctx, list(range(len(ctx)))
    t, s = case["tokens"], case["start"]
    return [s], t, list(range(s, s + t)), [0] * t


def _matmul_inputs(case, seed):
    t, k, n = case["tokens"], case["k"], case["n"]
    g = _gen(seed, 5)
    ldx = k + case["pad"]
    x = torch.randn((t, ldx), generator=g, device="cuda")
    return x, _bf16(g, (n, k), 0.02)


def prepare(case, seed):
    if case["op"] == "matmul":
        x, w = _matmul_inputs(case, seed)
        ldy = (case["n"] + 3) // 4 * 4
        return {"case": case, "x": x, "w": w, "ldx": x.shape[1], "ldy": ldy,
                "y": torch.zeros((case["tokens"], ldy), device="cuda")}
    d, hq, hkv, hd, f, v = DIMS[case["model"]]
    lens, n, pos, _ = _users(case)
    max_ctx = (max(pos) + 1 + 63) // 64 * 64
    shape = wl.ModelShape(n_layers_total=case["blocks"], d_model=d, n_heads=hq, n_kv_heads=hkv, head_dim=hd, ffn=f,
                          vocab=v, rms_eps=EPS, rope_theta=THETA,
                          weight_fmt="bf16" if case["fmt"] == "bf16" else "int4_g64", qk_norm=case["qk_norm"])
    # a prompt arrives at a stage that serves up to four users
    cfg = K.model_cfg(shape, max_ctx, n if case["op"] == "decode" else 4)
    flags = (K.KFL_EMBED_IN if case["embed"] else 0) | (K.KFL_LOGITS_OUT if case["logits"] else 0)
    st = K.kfl_stage_create(cfg, 0, case["blocks"], flags)
    for l in range(case["blocks"]):
        w = _layer(case, seed, l)
        torch.cuda.current_stream().synchronize()
        K.kfl_stage_load_layer(st, l, w, on_device=True)
        for u, length in enumerate(lens):
            if length:
                k, vv = _kv(case, seed, l, u, length)
                K.kfl_kv_write(st, l, u, k, vv, length, True)
        del w
    if flags:
        w = _head(case, seed)
        torch.cuda.current_stream().synchronize()
        K.kfl_stage_load_head(st, w, on_device=True)
        del w
    ids, hidden = _io(case, seed, n)
    return {"case": case, "stage": st, "ids": ids, "hidden": hidden, "n": n,
            "positions": torch.tensor(pos, dtype=torch.int32, device="cuda"),
            "out": torch.zeros((n, d), device="cuda"),
            "next": torch.zeros((n,), dtype=torch.int32, device="cuda") if case["logits"] else None}


def run(state):
    case = state["case"]
    stream = torch.cuda.current_stream().cuda_stream
    if case["op"] == "matmul":
        K.kfl_matmul_bf16w(state["x"], case["tokens"], case["k"], state["ldx"], state["w"], case["n"], state["y"],
                           state["ldy"], stream)
        return {"y": state["y"][:, :case["n"]]}
    if case["op"] == "decode":
        K.kfl_stage_decode(state["stage"], state["ids"], state["hidden"], state["positions"], state["n"],
                           state["out"], state["next"], stream)
    else:
        K.kfl_stage_prefill(state["stage"], state["ids"], state["hidden"], state["positions"], 0, state["n"],
                            state["out"], state["next"], stream)
    out = {"hidden": state["out"]}
    if case["logits"]:
        out["next_ids"] = state["next"]
    return out


# ------------------------------------------------------------------------------------- work

def _matrix_bytes(fmt, rows, cols):
    return rows * cols * 2 if fmt == "bf16" else rows * cols // 2 + rows * (cols // 64) * 2


def work(case):
    if case["op"] == "matmul":
        t, k, n = case["tokens"], case["k"], case["n"]
        return {"bytes": 4 * t * k + 2 * n * k + 4 * t * n, "flops": 2 * t * k * n}
    d, hq, hkv, hd, f, v = DIMS[case["model"]]
    lens, n, pos, _ = _users(case)
    shapes = [((hq + 2 * hkv) * hd, d), (d, hq * hd), (2 * f, d), (d, f)]
    kv_row = 2 * hkv * hd * 2  # one position's K and V
    # cached rows read once per user, the call's own rows written once; a (row, visible key) pair per head
    kv_read = sum(lens) * kv_row
    pairs = sum(p + 1 for p in pos)
    b = case["blocks"] * (sum(_matrix_bytes(case["fmt"], *s) for s in shapes) + 4 * d + kv_read + n * kv_row)
    fl = case["blocks"] * (2 * n * sum(r * c for r, c in shapes) + 4 * hd * hq * pairs)
    b += n * d * 4 + n * (2 * d if case["embed"] else 4 * d)
    if case["logits"]:
        b += _matrix_bytes(case["fmt"], v, d) + 2 * d + 4 * n
        fl += 2 * n * v * d
    return {"bytes": b, "flops": fl}


def tolerance(case):
    """About four times the largest distance from ``exact`` over some sixty cases of each path.

    Every path rounds the new K and V to bf16, as the cache holds them, so a difference in an
    earlier sum moves some of them by 2^-8.  Beyond that: bf16 decode steps keep fp32 activations
    (seen: up to 5e-5); int4 ones round their GEMV inputs to fp16 (up to 1.3e-3); prompts of fewer
    than 16 tokens and of QK-norm stages are decode steps; a dense prefill rounds q and the softmax
    weights to bf16 (up to 6e-3); the plain product carries x to 2^-17 and sums in fp32 (1e-5 at
    K = 17000).  next_ids: a tie within those errors may fall either way in a few of a prompt's 300
    or more rows; a decode step's few ids have to agree."""
    if case["op"] == "matmul":
        return {"rel": 4e-5}
    if case["op"] == "decode" or case["qk_norm"] or case["tokens"] < 16:
        tol = {"rel": 5e-3 if case["fmt"] == "int4" else 2e-4}
    else:
        tol = {"rel": 2e-2}
    if case["logits"]:
        tol["differ"] = 0.01 if case["op"] == "prefill" else 0.0
    return tol


# ------------------------------------------------------------------------------------- 64 bits

def _f64(m):
    if not isinstance(m, tuple):
        return m.double()
    words, scales = m
    rows = words.shape[0]
    code = torch.stack([(words >> (4 * j)) & 15 for j in range(8)], dim=-1)
    code = torch.where(code >= 8, code - 16, code).reshape(rows, -1, 64)
    return (code.double() * scales.double()[:, :, None]).reshape(rows, -1)


def _rms(x, g):
    return x / torch.sqrt((x * x).mean(-1, keepdim=True) + EPS) * g.double()


def _rope(x, pos):
    """x [rows][heads][hd] rotated by pairs (i, i + hd/2) at each row's position."""
    half = x.shape[-1] // 2
    i = torch.arange(half, device="cuda", dtype=torch.float64)
    a = pos.double()[:, None, None] * THETA ** (-i / half)
    c, s = torch.cos(a), torch.sin(a)
    x1, x2 = x[..., :half], x[..., half:]
    return torch.cat([x1 * c - x2 * s, x2 * c + x1 * s], dim=-1)


def _attend(q, k, v, pos):
    """q [rows][Hq][hd] at positions pos over k, v [Hkv][T][hd], causal."""
    rows, hq, hd = q.shape
    hkv, t, _ = k.shape
    o = torch.empty_like(q)
    key = torch.arange(t, device="cuda")
    for h in range(hkv):
        grp = slice(h * (hq // hkv), (h + 1) * (hq // hkv))
        for r in range(0, rows, 256):
            s = torch.einsum("rgd,td->rgt", q[r:r + 256, grp], k[h]) / math.sqrt(hd)
            s = s.masked_fill(key[None, None, :] > pos[r:r + 256, None, None], -math.inf)
            o[r:r + 256, grp] = torch.einsum("rgt,td->rgd", torch.softmax(s, dim=-1), v[h])
    return o


def exact(case, seed):
    if case["op"] == "matmul":
        x, w = _matmul_inputs(case, seed)
        return {"y": x[:, :case["k"]].double() @ w.double().t()}
    d, hq, hkv, hd, f, v = DIMS[case["model"]]
    lens, n, pos, user = _users(case)
    pos_t = torch.tensor(pos, device="cuda")
    ids, hidden = _io(case, seed, n)
    head = _head(case, seed)
    h = head["embed"][ids.long()].double() if case["embed"] else hidden.double()
    for l in range(case["blocks"]):
        w = _layer(case, seed, l)
        y = _rms(h, w["attn_norm"])
        q = (y @ _f64(w["wq"]).t()).view(n, hq, hd)
        k = (y @ _f64(w["wk"]).t()).view(n, hkv, hd)
        vv = (y @ _f64(w["wv"]).t()).view(n, hkv, hd)
        if case["qk_norm"]:
            q, k = _rms(q, w["q_norm"]), _rms(k, w["k_norm"])
        q, k = _rope(q, pos_t), _rope(k, pos_t)
        k, vv = k.float().bfloat16(), vv.float().bfloat16()  # the cache holds bf16
        o = torch.empty((n, hq, hd), device="cuda", dtype=torch.float64)
        for u, length in enumerate(lens):
            at = [i for i in range(n) if user[i] == u]
            kc, vc = _kv(case, seed, l, u, length)
            kc = torch.cat([kc, k[at].transpose(0, 1)], dim=1).double()
            vc = torch.cat([vc, vv[at].transpose(0, 1)], dim=1).double()
            o[at] = _attend(q[at], kc, vc, pos_t[at])
        h = h + o.view(n, hq * hd) @ _f64(w["wo"]).t()
        y = _rms(h, w["ffn_norm"])
        gate = y @ _f64(w["wg"]).t()
        a = gate / (1 + torch.exp(-gate)) * (y @ _f64(w["wu"]).t())
        h = h + a @ _f64(w["wd"]).t()
        del w
    out = {"hidden": h}
    if case["logits"]:
        y, best, idx = _rms(h, head["final_norm"]), None, None
        lm = head["lm_head"]
        for r in range(0, v, 16384):
            part = tuple(m[r:r + 16384] for m in lm) if isinstance(lm, tuple) else lm[r:r + 16384]
            z, i = (y @ _f64(part).t()).max(dim=-1)
            i = i + r
            if best is not None:
                i = torch.where(z > best, i, idx)
                z = torch.maximum(z, best)
            best, idx = z, i
        out["next_ids"] = idx.to(torch.int32)
    return out
