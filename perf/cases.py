"""What is measured of this framework: one pass through its public entry points per case.

A case is a dict of plain values: `op` says which calls a pass makes, the rest are sizes and
options.  Sizes are those of the repository's configurations, tests and benchmark (LLaVA-1.5:
N = 576 visual tokens, LLaVA-NeXT: N = 2880, the high-token regime: N = 7290, ragged
Qwen2.5-VL-like batches padded to 1280), with odd ones among them.  Features, questions and
attention maps are drawn as `paper_2608_06411_gb300.workloads` draws them (clustered visual
tokens, normal question tokens, log-normal attention), here on the GPU.  bf16 arrays are held
as 16-bit integers, as everywhere in this repository.

The predictor's weights are fixed (a deployed model); a context is made once per set of
widths and options and serves every input, as in a serving or training program.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2608_06411_gb300 import binding as mb

DEV = "cuda"
WEIGHTS_SEED = 7


# ----------------------------------------------------------------------------- cases

def listed() -> list:
    return [
        # One LLaVA-1.5 image and a short question: the smallest interactive request.
        dict(name="prune_one_n576", op="prune", B=1, N=576, D=4096, Dh=1024, dp=128, k=32, m_lo=32, m_hi=32,
             lam=1.0, grid=24, br=4, bc=4, dup=0, host=False),
        # One LLaVA-NeXT image (5 crops), 5.56 % of its tokens kept: the interactive request
        # of the paper's headline setting.
        dict(name="prune_one_n2880", op="prune", B=1, N=2880, D=4096, Dh=1024, dp=128, k=160, m_lo=64, m_hi=64,
             lam=1.0, grid=24, br=8, bc=8, dup=0, host=False),
        # Batched serving: 64 LLaVA-NeXT images with ragged questions, every tenth image with
        # near-duplicate crops (the benchmark's own batch).
        dict(name="prune_b64_n2880", op="prune", B=64, N=2880, D=4096, Dh=1024, dp=128, k=160, m_lo=16, m_hi=256,
             lam=1.0, grid=24, br=8, bc=8, dup=10, host=False),
        # High-token regime: 16 images of 10 tiles, long questions (up to 512 tokens), 405 kept.
        dict(name="prune_b16_n7290", op="prune", B=16, N=7290, D=3584, Dh=1024, dp=128, k=405, m_lo=264, m_hi=512,
             lam=1.0, grid=27, br=16, bc=8, dup=0, host=False),
        # Variable-resolution images in a padded batch (Qwen2.5-VL width).
        dict(name="ragged_b16_n1280", op="ragged", B=16, N=1280, D=3584, Dh=1024, dp=128, k=128, m_lo=16, m_hi=128,
             lam=1.0),
        # Features in pinned host memory (the vision tower ran elsewhere), results wanted on
        # the host: the copies are part of the call.
        dict(name="prune_host_b8_n2880", op="prune", B=8, N=2880, D=4096, Dh=1024, dp=128, k=160, m_lo=16, m_hi=256,
             lam=1.0, grid=24, br=8, bc=8, dup=10, host=True),
        # The separate calls, as a program makes them that feeds the language model itself:
        # score, select (with the pick order), assemble kept and question tokens.  Odd sizes.
        dict(name="handoff_b5_n1731", op="handoff", B=5, N=1731, D=2048, Dh=512, dp=64, k=97, m_lo=5, m_hi=77,
             lam=1.0, grid=24, br=8, bc=8, dup=0),
        # Selection alone on given importance scores at the high end of the retention sweep,
        # with a weaker diversity weight.
        dict(name="select_b2_n2880_k640", op="select", B=2, N=2880, D=4096, Dh=1024, dp=128, k=640, lam=0.5, grid=24,
             br=8, bc=8, dup=0),
        # Training the predictor: loss and every weight's gradient (forward and backward) for
        # four LLaVA-NeXT samples, and a small LLaVA-1.5 step.
        dict(name="distill_b4_n2880", op="distill", B=4, N=2880, D=4096, Dh=1024, dp=128, m_lo=16, m_hi=128, grid=24,
             br=8, bc=8),
        dict(name="distill_b2_n576", op="distill", B=2, N=576, D=4096, Dh=1024, dp=128, m_lo=8, m_hi=64, grid=24,
             br=4, bc=4),
        # Teacher selection over a 7B backbone's attention maps (32 layers, 32 heads):
        # LLaVA-1.5 samples and LLaVA-NeXT samples.
        dict(name="qcts_b4_n576", op="qcts", B=4, L=32, H=32, N=576, m_lo=8, m_hi=64, m_ref=7),
        dict(name="qcts_b2_n2880", op="qcts", B=2, L=32, H=32, N=2880, m_lo=16, m_hi=128, m_ref=7),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng) -> dict:
    """One more case: sizes spread over the listed ranges, no costlier than the largest."""
    op = rng.choice(["prune", "prune", "ragged", "handoff", "select", "distill", "qcts"])
    if op == "qcts":
        N = _log(rng, 192, 2880)
        return dict(op=op, B=rng.randint(1, 4), L=rng.choice([16, 28, 32]), H=rng.choice([16, 28, 32]), N=N, m_lo=4,
                    m_hi=rng.randint(8, 96), m_ref=rng.randint(4, 12))
    D, Dh, dp = rng.choice([(4096, 1024, 128), (3584, 1024, 128), (2048, 512, 64), (1536, 512, 128)])
    grid, br, bc = rng.choice([(24, 4, 4), (24, 8, 8), (27, 16, 8)])
    m_hi = _log(rng, 8, 256)
    base = dict(op=op, D=D, Dh=Dh, dp=dp, m_lo=min(4, m_hi), m_hi=m_hi)
    if op == "distill":
        N = _log(rng, 200, 2880)
        return dict(base, B=rng.randint(1, max(1, min(6, 11520 // N))), N=N, m_hi=min(m_hi, 128), grid=grid, br=br, bc=bc)
    lam = rng.choice([1.0, 1.0, 0.5, 2.0])
    N = _log(rng, 300, 7290)
    if op == "ragged":
        N = _log(rng, 400, 1600)
        return dict(base, B=_log(rng, 1, 24), N=N, k=_log(rng, 16, N // 5), lam=lam)
    k = _log(rng, 16, min(640, N // 3))
    B = _log(rng, 1, max(1, min(64, 90000 // N)))
    if op == "select":
        return dict(op=op, B=min(B, 8), N=N, D=D, Dh=Dh, dp=dp, k=k, lam=lam, grid=grid, br=br, bc=bc,
                    dup=rng.choice([0, 3]))
    case = dict(base, B=B, N=N, k=k, lam=lam, grid=grid, br=br, bc=bc, dup=rng.choice([0, 4]))
    return dict(case, host=rng.random() < 0.25) if op == "prune" else case


# ----------------------------------------------------------------------------- inputs

def _gen(seed: int, salt: int = 0) -> torch.Generator:
    return torch.Generator(device=DEV).manual_seed((int(seed) * 1000003 + salt) % (1 << 62))


def _randn(g, *shape):
    return torch.randn(*shape, generator=g, device=DEV, dtype=torch.float32)


def _bits(x) -> torch.Tensor:
    """fp32 -> bf16, as 16-bit integers."""
    return x.to(torch.bfloat16).view(torch.int16)


def _f64(bits) -> torch.Tensor:
    return bits.view(torch.bfloat16).to(torch.float64)


def _lens(case) -> np.ndarray:
    """Question lengths: the case's own, so that output shapes are."""
    rng = np.random.default_rng(case["B"] * 100_003 + case["N"] * 1009 + case["m_hi"])
    return rng.integers(case["m_lo"], case["m_hi"] + 1, size=case["B"]).astype(np.int32)


def _weights(D, Dh, dp) -> dict:
    """He-normal MLP layers, N(0, 1/fan_in) projections, small biases; bf16 bits."""
    g = _gen(WEIGHTS_SEED)
    w = {}
    for m, p in (("T", "Q"), ("V", "K")):
        w[f"w{m}1"] = _bits(_randn(g, Dh, D) * math.sqrt(2.0 / D))
        w[f"b{m}1"] = _bits(_randn(g, Dh) * 0.1)
        w[f"w{m}2"] = _bits(_randn(g, Dh, Dh) * math.sqrt(2.0 / Dh))
        w[f"b{m}2"] = _bits(_randn(g, Dh) * 0.1)
        w[f"w{p}"] = _bits(_randn(g, dp, Dh) * math.sqrt(1.0 / Dh))
    return w


def _images(case, seed) -> torch.Tensor:
    """[B, N, D] bf16 bits: crops of grid x grid tokens, each token its block's centroid plus
    N(0, 0.3^2); every dup-th image repeats its first crop with N(0, 0.05^2) on it."""
    B, N, D, grid = case["B"], case["N"], case["D"], case["grid"]
    per = grid * grid
    crops = -(-N // per)
    r = torch.arange(grid, device=DEV)
    cid = ((r[:, None] * case["br"] // grid) * case["bc"] + (r[None, :] * case["bc"] // grid)).reshape(-1)
    nc = case["br"] * case["bc"]
    ids = (torch.arange(crops, device=DEV)[:, None] * nc + cid[None, :]).reshape(-1)[:N]
    out = torch.empty((B, N, D), dtype=torch.int16, device=DEV)
    dup = case.get("dup", 0)
    for b in range(B):
        g = _gen(seed, b + 1)
        x = _randn(g, crops * nc, D)[ids] + 0.3 * _randn(g, N, D)
        if dup and b % dup == 0 and N > per:
            x[per:] = x[:per].repeat(crops, 1)[per:N] + 0.05 * _randn(g, N - per, D)
        out[b] = _bits(x)
    return out


def _ragged(case, seed):
    """Images on their own rows x cols token grids (8 x 8 blocks of centroids), padded with
    unrelated values to N rows; (bits [B, N, D], valid tokens per image)."""
    B, N, D = case["B"], case["N"], case["D"]
    rng = np.random.default_rng(int(seed) + 5)
    out = torch.empty((B, N, D), dtype=torch.int16, device=DEV)
    nv = np.empty(B, np.int32)
    for b in range(B):
        rows = int(rng.integers(min(20, N // 20), 33))
        rows = min(rows, N // 4)
        target = int(rng.integers(N // 2, N + 1))
        cols = max(1, min(target // rows, N // rows))
        n = nv[b] = rows * cols
        g = _gen(seed, b + 1)
        r = torch.arange(rows, device=DEV)[:, None] * 8 // rows
        c = torch.arange(cols, device=DEV)[None, :] * 8 // cols
        x = 5.0 * _randn(g, N, D)
        x[:n] = _randn(g, 64, D)[(r * 8 + c).reshape(-1)] + 0.3 * _randn(g, int(n), D)
        out[b] = _bits(x)
    return out, nv


def _scores(case, vis, seed) -> torch.Tensor:
    """Importance scores shaped like Eq. 3's: the mean of 48 softmaxes over the image's tokens
    with logits of standard deviation 2 that follow the features."""
    g = _gen(seed, 777_777)
    B, N, D = vis.shape
    p = torch.empty((B, N), dtype=torch.float32, device=DEV)
    for b in range(B):
        v = vis[b].view(torch.bfloat16).to(torch.float32)
        logits = (v @ _randn(g, D, 48)) * (2.0 / math.sqrt(1.09 * D))
        p[b] = torch.softmax(logits, dim=0).mean(dim=1)
    return p


def _teacher(case, seed) -> torch.Tensor:
    g = _gen(seed, 888_888)
    t = torch.softmax(2.0 * _randn(g, case["B"], case["N"]), dim=1)
    t[:, ::7] = 0.0                                   # 0 log 0 = 0
    return t / t.sum(dim=1, keepdim=True)


def _attention(case, lens, seed):
    """Attention maps (packed question blocks [L, H, M_b, N], reference [B, L, H, M_ref, N]):
    log-normal with a saliency per token, a region that the question draws attention to in
    the middle layers, and rows holding 5-50 % of the attention mass."""
    B, L, H, N, mr = case["B"], case["L"], case["H"], case["N"], case["m_ref"]
    attn = torch.empty(int(sum(L * H * int(m) * N for m in lens)), dtype=torch.int16, device=DEV)
    ref = torch.empty((B, L, H, mr, N), dtype=torch.int16, device=DEV)
    rng = np.random.default_rng(int(seed) + 11)
    o = 0
    for b in range(B):
        g = _gen(seed, b + 1)
        sal = 0.5 * _randn(g, N)
        lo = int(rng.integers(0, N - N // 10))
        roi = torch.zeros(N, device=DEV)
        roi[lo:lo + N // 16 + 1] = 1.0
        peak = int(rng.integers(L // 4, 3 * L // 4 + 1))
        head = torch.from_numpy(rng.uniform(0.3, 1.2, H)).to(DEV, torch.float32)[:, None, None]
        for l in range(L):
            gain = 3.0 * math.exp(-0.5 * ((l - peak) / max(L / 8.0, 1.0)) ** 2)
            for M, own in ((int(lens[b]), True), (mr, False)):
                z = torch.exp(0.7 * _randn(g, H, M, N) + sal + (gain * head * roi if own else 0.0))
                z *= (0.05 + 0.45 * torch.rand(H, M, 1, generator=g, device=DEV)) / z.sum(dim=-1, keepdim=True)
                if own:
                    attn[o:o + H * M * N] = _bits(z).reshape(-1)
                    o += H * M * N
                else:
                    ref[b, l] = _bits(z)
    return attn, ref


def _inputs(case, seed) -> dict:
    op, s = case["op"], {}
    if op == "qcts":
        s["lens"] = _lens(case)
        s["attn"], s["ref"] = _attention(case, s["lens"], seed)
        return s
    if op == "ragged":
        s["vis"], s["nv"] = _ragged(case, seed)
    else:
        s["vis"] = _images(case, seed)
    if op == "select":
        s["scores"] = _scores(case, s["vis"], seed)
        return s
    s["lens"] = _lens(case)
    s["text"] = _bits(_randn(_gen(seed, 555_555), int(s["lens"].sum()), case["D"]))
    if op == "distill":
        s["teacher"] = _teacher(case, seed)
    return s


# ----------------------------------------------------------------------------- passes

_contexts = {}


def _context(case) -> mb.Context:
    key = (case["D"], case["Dh"], case["dp"], case.get("lam", 1.0))
    if key not in _contexts:
        _contexts[key] = mb.Context(_weights(*key[:3]), *key[:3], lam=key[3])
    return _contexts[key]


def prepare(case, seed) -> dict:
    s = _inputs(case, seed)
    s["case"], op = case, case["op"]
    if op != "qcts":
        s["ctx"] = _context(case)
    if op in ("prune", "ragged"):
        B, N, D, k = case["B"], case["N"], case["D"], case["k"]
        host = case.get("host", False)
        where = dict(device="cpu", pin_memory=True) if host else dict(device=DEV)
        s["out"] = torch.empty((B, k, D), dtype=torch.int16, **where)
        s["keep"] = torch.empty((B, k), dtype=torch.int32, **where)
        s["scores"] = torch.empty((B, N), dtype=torch.float32, **where)
        if host:
            s["vis"], s["text"] = s["vis"].cpu().pin_memory(), s["text"].cpu().pin_memory()
    return s


def run(s):
    case, op = s["case"], s["case"]["op"]
    if op == "prune":
        s["ctx"].prune(s["text"], s["vis"], s["lens"], case["k"], s["out"], s["keep"], s["scores"])
        return {"scores": s["scores"], "keep": s["keep"], "out": s["out"]}
    if op == "ragged":
        s["ctx"].prune_ragged(s["text"], s["vis"], s["lens"], s["nv"], case["k"], s["out"], s["keep"], s["scores"])
        return {"scores": s["scores"], "keep": s["keep"], "out": s["out"]}
    if op == "handoff":
        scores = s["ctx"].score(s["text"], s["vis"], s["lens"])
        keep, order = s["ctx"].select(scores, s["vis"], case["k"])
        seq, pos = s["ctx"].assemble(s["vis"], keep, s["text"], s["lens"])
        return {"scores": scores, "keep": keep, "order": order, "seq": seq, "pos": pos}
    if op == "select":
        keep, order = s["ctx"].select(s["scores"], s["vis"], case["k"])
        return {"keep": keep, "order": order}
    if op == "distill":
        loss, grads = s["ctx"].distill_grad(s["text"], s["vis"], s["lens"], s["teacher"])
        return {"loss": loss, "grads": grads}
    p, p_ref, js, teacher, teacher_p = mb.qcts(s["attn"], s["lens"], s["ref"], case["L"], case["H"], case["N"])
    return {"p": p, "p_ref": p_ref, "js": js, "teacher": teacher, "teacher_p": teacher_p}


def work(case) -> dict:
    """Bytes: features, questions, weights read once, results written once.  Operations: the
    predictor with its second layer and projection folded (nothing lies between them), Eq. 3's
    logits, and each kept token's basis vector against each candidate; for training the
    unfolded predictor forward and backward (twice its operations, less the unneeded gradient
    with respect to the features)."""
    B, N = case["B"], case["N"]
    M = B * (case["m_lo"] + case["m_hi"]) / 2 if "m_lo" in case else 0
    if case["op"] == "qcts":
        L, H = case["L"], case["H"]
        maps = L * H * N * (M + B * case["m_ref"])
        return {"bytes": 2 * maps + 4 * (2 * B * L * N + B * L + B + B * N), "flops": maps}
    D, Dh, dp = case["D"], case["Dh"], case["dp"]
    feats = 2 * D * (B * N + M)
    if case["op"] == "distill":
        wts = 2 * (D * Dh + Dh * Dh + Dh * dp)
        first, rest = 2 * (B * N + M) * D * Dh, 2 * (B * N + M) * (Dh * Dh + Dh * dp)
        return {"bytes": feats + 2 * wts + 4 * wts + 4 * B * N, "flops": 2 * first + 3 * rest + 3 * 2 * M * N * dp}
    k = case["k"]
    sel = {"bytes": 2 * D * B * N + 4 * B * N + 4 * B * k, "flops": 2 * B * k * N * D}
    if case["op"] == "select":
        return {"bytes": sel["bytes"] + 4 * B * k, "flops": sel["flops"]}
    wts = 2 * 2 * (D * Dh + Dh * dp)
    rows = B * k + (M if case["op"] == "handoff" else 0)
    return {"bytes": feats + wts + 4 * B * N + 4 * B * k + 2 * D * rows,
            "flops": 2 * (B * N + M) * (D * Dh + Dh * dp) + 2 * M * N * dp + sel["flops"]}


def tolerance(case):
    """fp32 sums of bf16 products; scores pass through activations held to 16 bits.  A pick
    whose value ties with another's to fp32 accuracy may go either way (`differ`)."""
    if case["op"] == "distill":
        return {"rel": 1e-4, "max": 1e-3}
    if case["op"] == "qcts":
        return {"rel": 1e-6, "max": 1e-5, "differ": 0.01}
    return {"rel": 1e-4, "max": 1e-3, "differ": 0.01}


# ----------------------------------------------------------------------------- 64 bits

def _gelu(x):
    return 0.5 * x * (1.0 + torch.erf(x / math.sqrt(2.0)))


def _rope(x, pos):
    half = x.shape[1] // 2
    i = torch.arange(half, device=DEV, dtype=torch.float64)
    a = pos.to(torch.float64)[:, None] * (10000.0 ** (-2.0 * i / x.shape[1]))[None, :]
    x1, x2 = x[:, :half], x[:, half:]
    return torch.cat([x1 * a.cos() - x2 * a.sin(), x2 * a.cos() + x1 * a.sin()], dim=1)


def _p_hat(t, v, w):
    """Eq. 3 for one image: t [M, D], v [n, D], weights in 64 bits."""
    n, m = v.shape[0], t.shape[0]
    k = (_gelu(v @ w["wV1"].T + w["bV1"]) @ w["wV2"].T + w["bV2"]) @ w["wK"].T
    q = (_gelu(t @ w["wT1"].T + w["bT1"]) @ w["wT2"].T + w["bT2"]) @ w["wQ"].T
    k = _rope(k, torch.arange(n, device=DEV))
    q = _rope(q, n + torch.arange(m, device=DEV))
    return torch.softmax(q @ k.T / math.sqrt(q.shape[1]), dim=1).mean(dim=0)


def exact(case, seed):
    op = case["op"]
    if op == "select":
        return None                                   # whole numbers only
    s = _inputs(case, seed)
    lens = s["lens"]
    B, N = case["B"], case["N"]
    if op == "qcts":
        L, H, o = case["L"], case["H"], 0
        p = torch.empty((B, L, N), dtype=torch.float64, device=DEV)
        r = torch.empty_like(p)
        for b in range(B):
            for l in range(L):
                n = H * int(lens[b]) * N
                p[b, l] = _f64(s["attn"][o:o + n]).reshape(-1, N).sum(dim=0)
                r[b, l] = _f64(s["ref"][b, l]).reshape(-1, N).sum(dim=0)
                o += n
        p /= p.sum(dim=2, keepdim=True)
        r /= r.sum(dim=2, keepdim=True)
        m = 0.5 * (p + r)
        js = 0.5 * (p * torch.log(p / m)).sum(dim=2) + 0.5 * (r * torch.log(r / m)).sum(dim=2)
        best = js.argmax(dim=1)
        return {"p": p, "p_ref": r, "js": js, "teacher": None, "teacher_p": p[torch.arange(B, device=DEV), best]}
    w = {n: _f64(t) for n, t in _weights(case["D"], case["Dh"], case["dp"]).items()}
    off = np.concatenate([[0], np.cumsum(lens)])
    if op == "distill":
        for t in w.values():
            t.requires_grad_()
        loss = 0.0
        for b in range(B):
            ph = _p_hat(_f64(s["text"][off[b]:off[b + 1]]), _f64(s["vis"][b]), w)
            t = s["teacher"][b].to(torch.float64)
            on = t > 0
            part = (t[on] * torch.log(t[on] / ph[on])).sum() / B
            part.backward()
            loss += part.item()
        return {"loss": torch.tensor([loss], dtype=torch.float64), "grads": {n: t.grad for n, t in w.items()}}
    scores = torch.zeros((B, N), dtype=torch.float64, device=DEV)
    for b in range(B):
        n = int(s["nv"][b]) if op == "ragged" else N
        scores[b, :n] = _p_hat(_f64(s["text"][off[b]:off[b + 1]]), _f64(s["vis"][b, :n]), w)
    none = {"keep": None, "out": None} if op != "handoff" else {"keep": None, "order": None, "seq": None, "pos": None}
    return {"scores": scores, **none}
