"""The library's performance cases: one call (or one training step) each, through the public entry points.

``listed()`` are the sizes of this repository's own workloads (``paper_2106_06899_gb300/workloads.py``),
benchmark and tests; ``draw(rng)`` gives other cases of the same kinds over the whole range that each
kind is used in.  ``prepare`` draws the inputs on the GPU from the seed alone, ``run`` makes one pass,
``work`` counts what a pass cannot do without and ``exact`` restates a pass in 64 bits with plain torch.
"""
import math

import torch

from paper_2106_06899_gb300 import decoder as D
from paper_2106_06899_gb300 import topk as T


def listed():
    return [
        # the smallest attention call: fp32, one head of 512 tokens; launch and latency bound
        dict(name="attn_fp32_small", kind="attn", dtype="f32", B=1, H=1, Lq=512, Lk=512, d=64, topk=32, causal=False),
        # an encoder layer's attention over a batch of 512-token sequences (BERT-base heads)
        dict(name="attn_bert", kind="attn", dtype="bf16", B=8, H=12, Lq=512, Lk=512, d=64, topk=64, causal=False),
        # the same layer under a general attention mask (one bit per query and key, half of them set)
        dict(name="attn_bert_masked", kind="attn_masked", dtype="bf16", B=8, H=12, Lq=512, Lk=512, d=64, topk=64,
             density=0.5),
        # a whole 65,536-token sequence through one layer's heads: the headline workload
        dict(name="attn_long", kind="attn", dtype="bf16", B=1, H=12, Lq=65536, Lk=65536, d=64, topk=64, causal=False,
             dist="lowrank"),
        # a causal decoder layer's prefill with 128-wide heads and a larger kept set
        dict(name="attn_causal", kind="attn", dtype="bf16", B=2, H=16, Lq=16384, Lk=16384, d=128, topk=128,
             causal=True),
        # decoding: the last few positions of each sequence against its long key/value cache
        dict(name="attn_decode", kind="attn", dtype="bf16", B=4, H=12, Lq=128, Lk=65536, d=64, topk=64, causal=True,
             dist="lowrank"),
        # a kept set of several hundred keys
        dict(name="attn_large_k", kind="attn", dtype="bf16", B=1, H=12, Lq=8192, Lk=8192, d=64, topk=256,
             causal=False),
        # training: the forward pass that keeps its (index, score) cache, and the backward pass from it
        dict(name="attn_train", kind="attn_train", dtype="bf16", B=1, H=12, Lq=8192, Lk=8192, d=64, topk=64,
             causal=True),
        # a feed-forward layer of ordinary width over a small, ragged batch of tokens
        dict(name="ffn_small", kind="ffn", N=300, d_model=768, d_ff=3072, topk=64),
        # the wide feed-forward layer (65,536 keys) that the top-k is made for
        dict(name="ffn_large", kind="ffn", N=4096, d_model=1024, d_ff=65536, topk=512),
        # a training step's forward and backward pass through a wide feed-forward layer
        dict(name="ffn_train", kind="ffn_train", N=2048, d_model=1024, d_ff=16384, topk=256),
        # a whole decoder layer's training step: projections, top-k attention, feed-forward, and their gradients
        dict(name="decoder_layer", kind="decoder", L=8192, heads=12, d_ff=3072, topk=64),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["small", "encoder", "masked", "long", "causal", "decode", "large_k", "train", "ffn_small",
                       "ffn_large", "ffn_train", "decoder"])
    if kind == "small":
        L = _log(rng, 64, 1024)
        return dict(kind="attn", dtype="f32", B=rng.randint(1, 2), H=rng.randint(1, 8), Lq=L, Lk=L,
                    d=rng.choice([32, 64, 128]), topk=min(L, _log(rng, 8, 128)), causal=rng.random() < 0.5)
    if kind == "encoder":
        L = _log(rng, 128, 2048)
        B = max(1, min(rng.randint(1, 16), 8192 // L))
        return dict(kind="attn", dtype="bf16", B=B, H=rng.choice([8, 12, 16]), Lq=L, Lk=L, d=64,
                    topk=min(L, _log(rng, 16, 128)), causal=False)
    if kind == "masked":
        L = _log(rng, 100, 1024)
        return dict(kind="attn_masked", dtype=rng.choice(["bf16", "bf16", "f32"]), B=max(1, min(rng.randint(1, 8), 2048 // L)),
                    H=rng.choice([4, 8, 12]), Lq=L, Lk=L, d=64, topk=min(L, _log(rng, 16, 128)),
                    density=rng.uniform(0.2, 0.9))
    if kind == "long":
        L = _log(rng, 4096, 65536)
        return dict(kind="attn", dtype="bf16", B=1, H=rng.randint(1, 12), Lq=L, Lk=L, d=64, topk=_log(rng, 16, 72),
                    causal=False, dist="lowrank")
    if kind == "causal":
        L = _log(rng, 1024, 16384)
        return dict(kind="attn", dtype="bf16", B=rng.randint(1, 2), H=rng.choice([8, 16]), Lq=L, Lk=L,
                    d=rng.choice([64, 128]), topk=_log(rng, 16, 128), causal=True)
    if kind == "decode":
        return dict(kind="attn", dtype="bf16", B=rng.randint(1, 8), H=rng.choice([8, 12, 16]), Lq=_log(rng, 1, 128),
                    Lk=_log(rng, 2048, 65536), d=rng.choice([64, 128]), topk=_log(rng, 16, 128), causal=True,
                    dist="lowrank")
    if kind == "large_k":
        L = _log(rng, 1024, 8192)
        k = rng.randint(130, 512)
        return dict(kind="attn", dtype="bf16", B=1, H=rng.randint(2, 12 if k * L <= 256 * 8192 else 6), Lq=L, Lk=L,
                    d=rng.choice([64, 128]), topk=k, causal=rng.random() < 0.5)
    if kind == "train":
        L = _log(rng, 512, 12288)
        return dict(kind="attn_train", dtype="bf16", B=1, H=rng.choice([8, 12]), Lq=L, Lk=L,
                    d=rng.choice([64, 64, 128]), topk=_log(rng, 16, 96), causal=rng.random() < 0.7)
    if kind == "ffn_small":
        return dict(kind="ffn", N=_log(rng, 8, 512), d_model=64 * rng.randint(4, 16), d_ff=_log(rng, 1024, 8192),
                    topk=_log(rng, 16, 256))
    if kind == "ffn_large":
        return dict(kind="ffn", N=_log(rng, 512, 4096), d_model=64 * rng.randint(8, 16), d_ff=_log(rng, 8192, 65536),
                    topk=_log(rng, 64, 512))
    if kind == "ffn_train":
        return dict(kind="ffn_train", N=_log(rng, 256, 4096), d_model=64 * rng.randint(8, 16),
                    d_ff=_log(rng, 2048, 32768), topk=_log(rng, 32, 256))
    return dict(kind="decoder", L=_log(rng, 512, 8192), heads=rng.choice([8, 12]), d_ff=3072, topk=_log(rng, 32, 64))


_DTYPE = {"f32": torch.float32, "bf16": torch.bfloat16}


def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _randn(g, *shape):
    return torch.randn(*shape, generator=g, device="cuda")


def _attn_inputs(c, g):
    """Q and K of unit-variance entries scaled by d^-1/4 each (Eq. 1's temperature folded in); "lowrank"
    adds a rank-8 part shared by a head's queries and keys, so that score rows have a few heavy entries."""
    B, H, Lq, Lk, d = c["B"], c["H"], c["Lq"], c["Lk"], c["d"]
    q, k, v = _randn(g, B, H, Lq, d), _randn(g, B, H, Lk, d), _randn(g, B, H, Lk, d)
    if c.get("dist") == "lowrank":
        basis = torch.linalg.qr(_randn(g, H, d, 8).cpu()).Q.transpose(1, 2).cuda()[None]
        q += 2.0 * _randn(g, B, H, Lq, 8) @ basis
        k += 2.0 * _randn(g, B, H, Lk, 8) @ basis
    dt = _DTYPE[c["dtype"]]
    return (q * d ** -0.25).to(dt), (k * d ** -0.25).to(dt), v.to(dt)


def _ffn_inputs(c, g):
    s = c["d_model"] ** -0.5
    x = _randn(g, c["N"], c["d_model"]).bfloat16()
    w1 = (_randn(g, c["d_ff"], c["d_model"]) * s).bfloat16()
    w2 = (_randn(g, c["d_ff"], c["d_model"]) * s).bfloat16()
    return x, w1, w2


def _mask(c, g):
    return torch.rand(c["B"], 1, c["Lq"], c["Lk"], generator=g, device="cuda") < c["density"]


def prepare(case, seed):
    c, g = case, _gen(seed)
    st = dict(case=c)
    if c["kind"].startswith("attn"):
        st["q"], st["k"], st["v"] = _attn_inputs(c, g)
        if c["kind"] == "attn_masked":  # a program packs a batch's mask once for all of its layers
            st["words"], st["bs"], st["hs"] = T.pack_mask(_mask(c, g))
        if c["kind"] == "attn_train":
            st["dout"] = _randn(g, *st["q"].shape).to(st["q"].dtype)
    elif c["kind"].startswith("ffn"):
        st["x"], st["w1"], st["w2"] = _ffn_inputs(c, g)
        if c["kind"] == "ffn_train":
            st["dout"] = _randn(g, c["N"], c["d_model"])
    else:
        torch.manual_seed(int(seed))
        st["layer"] = D.DecoderLayer(64 * c["heads"], c["heads"], c["d_ff"], c["topk"], None)
        st["x"] = _randn(g, 1, c["L"], 64 * c["heads"]).bfloat16().requires_grad_()
        st["dout"] = _randn(g, 1, c["L"], 64 * c["heads"]).bfloat16()
    return st


def run(st):
    c = st["case"]
    if c["kind"] == "attn":
        return T.attention(st["q"], st["k"], st["v"], c["topk"], causal=c["causal"])
    if c["kind"] == "attn_masked":
        out = torch.empty_like(st["q"])
        T.topk_attn_fwd_masked(st["q"], st["k"], st["v"], out, c["topk"], mask_words=st["words"],
                               mask_batch_stride=st["bs"], mask_head_stride=st["hs"])
        return out
    if c["kind"] == "attn_train":
        out, idx, score = T.attention(st["q"], st["k"], st["v"], c["topk"], causal=c["causal"], return_indices=True)
        dq, dk, dv = T.attention_bwd(st["q"], st["k"], st["v"], st["dout"], idx, score)
        return dict(out=out, idx=idx, score=score, dq=dq, dk=dk, dv=dv)
    if c["kind"] == "ffn":
        return T.ffn(st["x"], st["w1"], st["w2"], c["topk"])
    if c["kind"] == "ffn_train":
        out, idx, score = T.ffn(st["x"], st["w1"], st["w2"], c["topk"], return_indices=True)
        dx, dw1, dw2 = T.ffn_bwd(st["x"], st["w1"], st["w2"], st["dout"], idx, score)
        return dict(out=out, idx=idx, score=score, dx=dx, dw1=dw1, dw2=dw2)
    layer, x = st["layer"], st["x"]
    y = layer(x)
    grads = torch.autograd.grad(y, [x, *layer.parameters()], st["dout"])
    return [y.detach(), *grads]


def work(case):
    c = case
    if c["kind"].startswith("attn"):
        eb = 4 if c["dtype"] == "f32" else 2
        bh, Lq, Lk, d, k = c["B"] * c["H"], c["Lq"], c["Lk"], c["d"], c["topk"]
        pairs = Lq * (Lk - Lq) + Lq * (Lq + 1) // 2 if c.get("causal") else Lq * Lk
        rows = bh * Lq
        b = (2 * rows + 2 * bh * Lk) * d * eb
        f = 2 * bh * pairs * d + 2 * rows * k * d
        if c["kind"] == "attn_masked":
            b += c["B"] * Lq * ((Lk + 31) // 32) * 4
            f = int(2 * bh * pairs * d * c["density"]) + 2 * rows * k * d
        if c["kind"] == "attn_train":  # the cache out, dout in, fp32 gradients out; four sparse products
            b += rows * k * 8 + rows * d * eb + (rows + 2 * bh * Lk) * d * 4
            f += 8 * rows * k * d
        return dict(bytes=b, flops=f)
    if c["kind"].startswith("ffn"):
        N, dm, dff, k = c["N"], c["d_model"], c["d_ff"], c["topk"]
        b = N * dm * 2 + 2 * dff * dm * 2 + N * dm * 4
        f = 2 * N * dff * dm + 2 * N * k * dm
        if c["kind"] == "ffn_train":
            b += N * k * 8 + N * dm * 4 + N * dm * 4 + 2 * dff * dm * 4
            f += 8 * N * k * dm
        return dict(bytes=b, flops=f)
    L, h, dff, k = c["L"], c["heads"], c["d_ff"], c["topk"]
    dm = 64 * h
    par = 4 * dm * dm + 2 * dff * dm
    # 16-bit weights in, their gradients out; x and dout in, y and dx out; dense products three times (forward
    # and two backward), the causal scores once, the kept keys' products five times
    return dict(bytes=2 * (2 * par + 4 * L * dm), flops=6 * L * par + L * (L + 1) * dm + 10 * L * k * dm)


def _exact_attention(q, k, v, topk, causal, mask):
    """Per (b, h, row chunk): fp64 scores, the k largest, softmax over them, the weighted sum of values."""
    B, H, Lq, d = q.shape
    Lk = k.shape[2]
    out = torch.zeros(B, H, Lq, d, dtype=torch.float64, device=q.device)
    idx = torch.zeros(B, H, Lq, topk, dtype=torch.int64, device=q.device)
    sc = torch.zeros(B, H, Lq, topk, dtype=torch.float64, device=q.device)
    step = max(1, (1 << 27) // Lk)
    keys = torch.arange(Lk, device=q.device)
    for b in range(B):
        for h in range(H):
            kd, vd = k[b, h].double(), v[b, h].double()
            for i in range(0, Lq, step):
                s = q[b, h, i:i + step].double() @ kd.T
                n = s.shape[0]
                if causal:
                    pos = torch.arange(i, i + n, device=q.device)[:, None] + (Lk - Lq)
                    s.masked_fill_(keys[None] > pos, -math.inf)
                if mask is not None:
                    s.masked_fill_(~mask[b, 0, i:i + n], -math.inf)
                top, j = s.topk(topk, dim=1)
                a = torch.softmax(top, dim=1).nan_to_num(0.0)
                out[b, h, i:i + n] = torch.einsum("nt,ntd->nd", a, vd[j])
                idx[b, h, i:i + n], sc[b, h, i:i + n] = j, top
    return out, idx, sc


def _exact_attention_bwd(q, k, v, dout, idx, sc):
    B, H, Lq, d = q.shape
    dq = torch.zeros(B, H, Lq, d, dtype=torch.float64, device=q.device)
    dk = torch.zeros(k.shape, dtype=torch.float64, device=q.device)
    dv = torch.zeros(v.shape, dtype=torch.float64, device=q.device)
    step = max(1, (1 << 25) // (idx.shape[-1] * d))
    for b in range(B):
        for h in range(H):
            qd, kd, vd, gd = (t[b, h].double() for t in (q, k, v, dout))
            for i in range(0, Lq, step):
                j, g = idx[b, h, i:i + step], gd[i:i + step]
                a = torch.softmax(sc[b, h, i:i + step], dim=1)
                da = torch.einsum("nd,ntd->nt", g, vd[j])
                ds = a * (da - (a * da).sum(1, keepdim=True))
                dq[b, h, i:i + step] = torch.einsum("nt,ntd->nd", ds, kd[j])
                flat = j.reshape(-1)
                dk[b, h].index_add_(0, flat, (ds[..., None] * qd[i:i + step, None]).reshape(-1, d))
                dv[b, h].index_add_(0, flat, (a[..., None] * g[:, None]).reshape(-1, d))
    return dq, dk, dv


def _exact_ffn(x, w1, w2, topk):
    N, dm = x.shape
    out = torch.zeros(N, dm, dtype=torch.float64, device=x.device)
    idx = torch.zeros(N, topk, dtype=torch.int64, device=x.device)
    sc = torch.zeros(N, topk, dtype=torch.float64, device=x.device)
    w1d, w2d = w1.double(), w2.double()
    step = max(1, (1 << 28) // max(w1.shape[0], topk * dm))
    for i in range(0, N, step):
        top, j = (x[i:i + step].double() @ w1d.T).topk(topk, dim=1)
        out[i:i + step] = torch.einsum("nt,ntd->nd", torch.relu(top), w2d[j])
        idx[i:i + step], sc[i:i + step] = j, top
    return out, idx, sc


def _exact_ffn_bwd(x, w1, w2, dout, idx, sc):
    dx = torch.zeros(x.shape, dtype=torch.float64, device=x.device)
    dw1 = torch.zeros(w1.shape, dtype=torch.float64, device=x.device)
    dw2 = torch.zeros(w2.shape, dtype=torch.float64, device=x.device)
    w1d, w2d = w1.double(), w2.double()
    dm = x.shape[1]
    step = max(1, (1 << 28) // (idx.shape[1] * dm))
    for i in range(0, x.shape[0], step):
        xd, g, j, s = x[i:i + step].double(), dout[i:i + step].double(), idx[i:i + step], sc[i:i + step]
        ds = torch.einsum("nd,ntd->nt", g, w2d[j]) * (s > 0)
        dx[i:i + step] = torch.einsum("nt,ntd->nd", ds, w1d[j])
        flat = j.reshape(-1)
        dw1.index_add_(0, flat, (ds[..., None] * xd[:, None]).reshape(-1, dm))
        dw2.index_add_(0, flat, (torch.relu(s)[..., None] * g[:, None]).reshape(-1, dm))
    return dx, dw1, dw2


def exact(case, seed):
    c, g = case, _gen(seed)
    if c["kind"] == "decoder":  # which keys a row keeps depends on how the layers before round to 16 bits
        return None
    if c["kind"].startswith("attn"):
        if c["B"] * c["H"] * c["Lq"] * c["Lk"] * c["d"] > 1 << 40:  # minutes of 64-bit arithmetic
            return None
        q, k, v = _attn_inputs(c, g)
        mask = _mask(c, g) if c["kind"] == "attn_masked" else None
        out, idx, sc = _exact_attention(q, k, v, c["topk"], c.get("causal", False), mask)
        if c["kind"] != "attn_train":
            return out
        dout = _randn(g, *q.shape).to(q.dtype)
        dq, dk, dv = _exact_attention_bwd(q, k, v, dout, idx, sc)
        return dict(out=out, idx=None, score=sc, dq=dq, dk=dk, dv=dv)
    x, w1, w2 = _ffn_inputs(c, g)
    out, idx, sc = _exact_ffn(x, w1, w2, c["topk"])
    if c["kind"] == "ffn":
        return out
    dx, dw1, dw2 = _exact_ffn_bwd(x, w1, w2, _randn(g, c["N"], c["d_model"]), idx, sc)
    return dict(out=out, idx=None, score=sc, dx=dx, dw1=dw1, dw2=dw2)
