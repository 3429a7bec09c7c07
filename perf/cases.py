"""The work that users of this library have it do, as cases that can be timed.

Every case is one call of a public entry point (or one token of a decoder)
on device-resident data:

  gemv   wq4_gemv: one packed projection for 1-32 activation rows
  gemm   wq4_gemm: one packed projection over a prompt's tokens
  attn   wq4_paged_attention: one layer's decode attention over a paged cache
  chain  wq4_decode_chain(_host): one token through every projection
  step   wq4_decode_step: one token with rotary embedding, cache append and
         paged attention in every layer

Sizes are those of the 3B-, 8B- and Phi-3.5-mini-shaped models of
paper_2412_15803_gb300.model and odd sizes in between; codes, scales and
activations have the distributions of the library's synthetic models.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2412_15803_gb300 import wq4
from paper_2412_15803_gb300.attention import PagedAttentionLayer
from paper_2412_15803_gb300.model import SHAPES, DecodeModel, ModelShape, StepCaches

EPS = 1e-5


def listed():
    return [
        # the smallest projection: one token's latency and launch cost
        {"name": "gemv-2048-b1", "kind": "gemv", "N": 2048, "K": 2048, "batch": 1},
        # the largest projection of a 3B layer for one stream
        {"name": "gemv-3b-gate-up-b1", "kind": "gemv", "N": 16384, "K": 3072, "batch": 1},
        # the longest rows of a 3B layer for eight streams decoding together
        {"name": "gemv-3b-down-b8", "kind": "gemv", "N": 3072, "K": 8192, "batch": 8},
        # an odd model: rows of 65 groups (no multiple of 256), an odd row count, five streams
        {"name": "gemv-ragged-b5", "kind": "gemv", "N": 1003, "K": 2080, "batch": 5},
        # the LM head of an 8B model at the largest batch
        {"name": "gemv-8b-head-b32", "kind": "gemv", "N": 128256, "K": 4096, "batch": 32},
        # a short prompt of odd length through the fused QKV projection
        {"name": "gemm-3b-qkv-m77", "kind": "gemm", "N": 5120, "K": 3072, "M": 77},
        # a long prompt (or a chunk of one) through the largest 8B projection
        {"name": "gemm-8b-gate-up-m2048", "kind": "gemm", "N": 28672, "K": 4096, "M": 2048},
        # one stream with a 4096-token conversation, one layer
        {"name": "attn-8b-b1-4096", "kind": "attn", "shape": "8b", "batch": 1, "lo": 4096, "hi": 4096, "page": 16},
        # a serving batch of mixed context lengths, one layer
        {"name": "attn-3b-b32-mixed", "kind": "attn", "shape": "3b", "batch": 32, "lo": 1, "hi": 8192, "page": 16},
        # the whole 3B-shaped model, one token of one stream: the headline
        {"name": "chain-3b-b1", "kind": "chain", "shape": "3b", "layers": 28, "vocab": 128256, "batch": 1, "host": False},
        # the whole 3B-shaped model with attention over 4096 cached tokens
        {"name": "step-3b-b1-4096", "kind": "step", "shape": "3b", "layers": 28, "vocab": 128256, "batch": 1, "ctx": 4096,
         "page": 16},
        # a serving batch through a block of 8B layers, contexts up to 2048
        {"name": "step-8b-b16-2048", "kind": "step", "shape": "8b", "layers": 4, "vocab": 32064, "batch": 16, "ctx": 2048,
         "page": 16},
    ]


def _log(rng, lo, hi):
    """A whole number spread over [lo, hi] by its logarithm."""
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["gemv", "gemv", "gemm", "gemm", "attn", "chain", "step"])
    if kind == "gemv":
        # rows of whole 256-code units as in real models, and now and then any number of groups
        K = 256 * _log(rng, 1, 56) if rng.random() < 0.75 else 32 * _log(rng, 1, 256)
        batch = _log(rng, 1, 32)
        return {"kind": kind, "N": _log(rng, 64, min(128256, 128256 * 4096 // K)), "K": K, "batch": batch}
    if kind == "gemm":
        K = 256 * _log(rng, 1, 56)
        M = _log(rng, 1, 2048)
        return {"kind": kind, "N": 8 * _log(rng, 16, 28672 * 4096 // K // 8 if K > 4096 else 3584), "K": K, "M": M}
    if kind == "attn":
        batch = _log(rng, 1, 64)
        hi = _log(rng, 16, min(16384, 32 * 8192 // batch))
        return {"kind": kind, "shape": rng.choice(["3b", "8b"]), "batch": batch, "lo": rng.randint(1, hi), "hi": hi,
                "page": rng.choice([16, 16, 32, 64])}
    if kind == "chain":
        return {"kind": kind, "shape": rng.choice(["3b", "8b", "phi3.5"]), "layers": rng.randint(1, 4),
                "vocab": _log(rng, 1000, 32064), "batch": _log(rng, 1, 32), "host": rng.random() < 0.25}
    return {"kind": kind, "shape": rng.choice(["3b", "8b"]), "layers": rng.randint(1, 4), "vocab": _log(rng, 1000, 32064),
            "batch": _log(rng, 1, 32), "ctx": _log(rng, 16, 4096), "page": rng.choice([16, 16, 32])}


# ------------------------------------------------------------------ inputs --

def _shape(case):
    s = SHAPES[case["shape"]]
    return ModelShape(s.name, case["layers"], s.hidden, s.ffn, s.n_q_heads, s.n_kv_heads, s.head_dim, case["vocab"])


def _lens(lo, hi, batch):
    """Lengths evenly spread over [lo, hi]."""
    return [hi] if batch == 1 else [lo + (hi - lo) * b // (batch - 1) for b in range(batch)]


def _positions(case):
    """Tokens already cached: contexts from a quarter of ctx to ctx, the new token included."""
    return [n - 1 for n in _lens(max(1, case["ctx"] // 4), case["ctx"], case["batch"])]


def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _activations(rows, K, g):
    return torch.randn((rows, K), generator=g, device="cuda").half().view(torch.int16)


def _as_trained(model):
    """Scales of a trained model's size in place of the synthetic ones, so that rounding in one layer
    is not blown up by all that follow: projections that keep the size of their input, and residual
    branches (O, down) that change the stream by a fifth of it."""
    mats = [(name, m) for layer in model.weights for name, m in layer.items()] + [("lm_head", model.lm_head)]
    for name, (W, scales) in mats:
        # codes 0..14 and scales on [0.005, 0.02] give weights of deviation 0.0563
        gain = 0.2 if name in ("o", "down") else 1.0
        scales.view(torch.float16).mul_(gain / (0.0563 * math.sqrt(8 * W.shape[1])))


def prepare(case, seed):
    g = _generator(seed)
    # the stream handle is kept, as a serving loop keeps it
    s = {"case": case, "stream": torch.cuda.current_stream().cuda_stream}
    kind = case["kind"]
    if kind in ("gemv", "gemm"):
        N, K, rows = case["N"], case["K"], case["batch" if kind == "gemv" else "M"]
        s["W"] = torch.randint(-2 ** 31, 2 ** 31, (N, K // 8), generator=g, device="cuda", dtype=torch.int32)
        s["scales"] = (0.005 + 0.015 * torch.rand((N, K // 32), generator=g, device="cuda")).half().view(torch.int16)
        s["x"] = _activations(rows, K, g)
        s["y"] = torch.empty((rows, N), dtype=torch.int16, device="cuda")
    elif kind == "attn":
        lens = np.random.RandomState(seed % 2 ** 32).permutation(_lens(case["lo"], case["hi"], case["batch"]))
        s["layer"] = PagedAttentionLayer(SHAPES[case["shape"]], lens, page_size=case["page"], seed=seed)
    else:
        shape = _shape(case)
        s["model"] = DecodeModel(shape, batch=case["batch"], seed=seed, eps=EPS, step=kind == "step")
        _as_trained(s["model"])
        s["x"] = _activations(case["batch"], shape.hidden, g)
        if kind == "step":
            s["caches"] = StepCaches(shape, _positions(case), page_size=case["page"], seed=seed)
        if case.get("host"):
            s["x"] = s["x"].cpu().numpy().view(np.uint16)
            s["logits"] = np.empty((case["batch"], shape.vocab), np.uint16)
        else:
            s["logits"] = torch.empty((case["batch"], shape.vocab), dtype=torch.int16, device="cuda")
    return s


# -------------------------------------------------------------------- calls --

def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "gemv":
        wq4.wq4_gemv(s["W"], s["scales"], s["x"], s["y"], case["N"], case["K"], case["batch"], s["stream"])
        return s["y"].view(torch.float16)
    if kind == "gemm":
        wq4.wq4_gemm(s["W"], s["scales"], s["x"], s["y"], case["N"], case["K"], case["M"], s["stream"])
        return s["y"].view(torch.float16)
    if kind == "attn":
        s["layer"].run(s["stream"])
        return s["layer"].out.view(torch.float16)
    if kind == "chain":
        if case["host"]:
            s["model"].decode_host(s["x"], s["logits"], s["stream"])
            return s["logits"].view(np.float16)
        s["model"].decode(s["x"], s["logits"], s["stream"])
        return s["logits"].view(torch.float16)
    s["model"].decode_step(s["caches"], s["x"], s["logits"], s["stream"])
    c = s["caches"]
    return {"logits": s["logits"].view(torch.float16), "k": [k.view(torch.float16) for k in c.k],
            "v": [v.view(torch.float16) for v in c.v]}


# --------------------------------------------------------------------- work --

def work(case):
    kind = case["kind"]
    if kind in ("gemv", "gemm"):
        N, K, rows = case["N"], case["K"], case["batch" if kind == "gemv" else "M"]
        return {"bytes": N * K * 9 // 16 + 2 * rows * (N + K), "flops": 2 * N * K * rows}
    if kind == "attn":
        sh = SHAPES[case["shape"]]
        tokens = sum(_lens(case["lo"], case["hi"], case["batch"]))
        return {"bytes": tokens * sh.n_kv_heads * sh.head_dim * 4 + 4 * case["batch"] * sh.n_q_heads * sh.head_dim,
                "flops": 4 * tokens * sh.n_q_heads * sh.head_dim}
    sh, B = _shape(case), case["batch"]
    nbytes = sh.weight_bytes() + 2 * B * (sh.hidden + sh.vocab)
    flops = 2 * sh.weight_count() * B
    if kind == "step":
        cached = sum(_positions(case))
        nbytes += case["layers"] * (cached + B) * sh.n_kv_heads * sh.head_dim * 4
        flops += case["layers"] * 4 * (cached + B) * sh.n_q_heads * sh.head_dim
    return {"bytes": nbytes, "flops": flops}


def tolerance(case):
    kind = case["kind"]
    if kind == "gemv":
        return {"rel": 1e-3, "max": 4e-3}      # fp32 sums, one rounding of y to fp16
    if kind == "gemm":
        return {"rel": 1.2e-3, "max": 5e-3}    # each weight rounded to fp16 as well
    if kind == "attn":
        return {"rel": 1e-3, "max": 4e-3}      # softmax weights rounded to fp16
    # every stage of every layer rounds to fp16 and passes it on: 0.0008 from the exact token
    # after 4 layers, 0.0021 after 28
    return {"rel": 4e-3, "max": 2.5e-2} if case["layers"] <= 4 else {"rel": 1e-2, "max": 6e-2}


# -------------------------------------------------------- the same in 64 bits --

def _project(W, scales, x):
    """x (q - 7) s^T in fp64 for packed rows W int32 [N][K/8], scales [N][K/32] (fp16 bits), x fp64 [rows][K]."""
    shifts = torch.arange(0, 32, 4, device=W.device, dtype=torch.int32)
    out = []
    for n in range(0, W.shape[0], 8192):
        w = W[n:n + 8192]
        q = ((w[:, :, None] >> shifts) & 15).double().reshape(w.shape[0], -1, 32) - 7
        q *= scales[n:n + 8192].view(torch.float16).double()[:, :, None]
        out.append(x @ q.reshape(w.shape[0], -1).T)
    return torch.cat(out, 1)


def _norm(t):
    return t / torch.sqrt((t * t).mean(1, keepdim=True) + EPS)


def _rope(t, positions, theta):
    """Adjacent pairs of each 128-wide head turned by pos * theta^(-2i / 128)."""
    rows = t.shape[0]
    p = t.reshape(rows, -1, 64, 2)
    i = torch.arange(64, device=t.device, dtype=torch.float64)
    a = positions.double()[:, None] * theta ** (-2 * i / 128)
    c, sn = torch.cos(a)[:, None], torch.sin(a)[:, None]
    return torch.stack([p[..., 0] * c - p[..., 1] * sn, p[..., 0] * sn + p[..., 1] * c], -1).reshape(rows, -1)


def _attend(q, k, v, table, lens, scale, page):
    """Decode attention in fp64: q [batch][Hq * D], k, v [pages][Hkv][page][D], table [batch][n]."""
    Hkv, D = k.shape[1], k.shape[3]
    out = []
    for b, T in enumerate(lens):
        pages = table[b, :(T + page - 1) // page].long()
        kb, vb = (t[pages].double().permute(1, 0, 2, 3).reshape(Hkv, -1, D)[:, :T] for t in (k, v))
        qb = q[b].reshape(Hkv, -1, D)
        out.append((torch.softmax(scale * qb @ kb.transpose(1, 2), -1) @ vb).reshape(-1))
    return torch.stack(out)


def exact(case, seed):
    kind = case["kind"]
    if kind in ("gemv", "gemm"):
        s = prepare(case, seed)
        return _project(s["W"], s["scales"], s["x"].view(torch.float16).double())
    if kind == "attn":
        y = prepare(case, seed)["layer"]
        return _attend(y.q.view(torch.float16).double(), y.k.view(torch.float16), y.v.view(torch.float16), y.table,
                       y.lens.tolist(), y.scale, y.page_size)
    s = prepare(case, seed)
    sh, model = _shape(case), s["model"]
    x = s["x"]
    x = torch.from_numpy(x.view(np.float16)).cuda().double() if case.get("host") else x.view(torch.float16).double()
    H, kv = sh.hidden, sh.n_kv_heads * sh.head_dim
    keys, values = [], []
    for l in range(sh.num_layers):
        w = model.weights[l]
        v = _norm(x)
        qkv = _project(*w["qkv"], v)
        a = qkv[:, :H]
        if kind == "step":
            c = s["caches"]
            pos = c.pos_dev.long()
            k, vv = c.k[l].view(torch.float16).double(), c.v[l].view(torch.float16).double()
            rows = torch.arange(case["batch"], device="cuda")
            pages = c.table[rows, pos // c.page_size].long()
            k[pages, :, pos % c.page_size] = _rope(qkv[:, H:H + kv], pos, c.rope_theta).reshape(-1, sh.n_kv_heads, 128)
            vv[pages, :, pos % c.page_size] = qkv[:, H + kv:].reshape(-1, sh.n_kv_heads, 128)
            keys.append(k)
            values.append(vv)
            a = _attend(_rope(a, pos, c.rope_theta), k, vv, c.table, (pos + 1).tolist(), c.scale, c.page_size)
        x1 = v + _project(*w["o"], _norm(a))
        gu = _project(*w["gate_up"], _norm(x1))
        m = torch.nn.functional.silu(gu[:, :sh.ffn]) * gu[:, sh.ffn:]
        x = x1 + _project(*w["down"], m)
    logits = _project(*model.lm_head, _norm(x))
    if kind == "step":
        return {"logits": logits, "k": keys, "v": values}
    return logits.cpu().numpy() if case["host"] else logits
