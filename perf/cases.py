"""The calls whose speed matters to a user of this library, as measurable cases.

A case is one call through the Python binding (``optr``) in a serving
program's terms: a decode over the paged INT2 cache, a decode step (cache
write of the new tokens, then decode), a cache write of a prompt, or the
offline calibration of one KV head.  ``listed()`` names the ones that stand
for everyday use, ``draw()`` gives others of the same ranges, ``prepare()``
builds what a program holds before the call, ``run()`` is the call, ``work()``
its unavoidable bytes and operations, and ``exact()`` the same result in
float64 from plain torch.

The cache a decode reads is filled here with plain torch (rotated, quantized
and packed as include/optr.h lays it out), so that ``exact()`` sees the same
bytes without calling the library.
"""
from __future__ import annotations

import math
import random

import torch

from paper_2608_02691_gb300 import optr

D = 128
PAGE = 16
DEV = "cuda"

# the paper's cache configuration: G = 128, clips, 64 sink and 256 recent
# tokens in BF16
PAPER = {"group": 128, "clip_k": 0.96, "clip_v": 0.92, "sink": 64, "recent": 256}
# min-max groups of 32 and no windows: the benchmark's cache
G32 = {"group": 32, "clip_k": 1.0, "clip_v": 1.0, "sink": 0, "recent": 0}


def _decode(kind, B, lo, hi, opts, h_kv=8, fold=False, host=False, lens=0):
    return {"kind": kind, "B": B, "ctx_lo": lo, "ctx_hi": hi, "lens": lens, "h_kv": h_kv,
            "fold": fold, "host": host, **opts}


def _append(B, lo, hi, pos0, opts, h_kv=8, lens=0):
    return {"kind": "append", "B": B, "ctx_lo": lo, "ctx_hi": hi, "lens": lens, "pos0": pos0,
            "h_kv": h_kv, "fold": False, **opts}


def _calib(T, nt, d_model, steps, opts):
    return {"kind": "calib", "T": T, "nt": nt, "g": 4, "d_model": d_model, "steps": steps, **opts}


def listed():
    return [
        # one short sequence, one layer: the smallest decode, all latency
        {"name": "decode_1x1k", **_decode("decode", 1, 1024, 1024, G32)},
        # a single chat in the paper's configuration, at an odd length
        {"name": "step_1x4k_paper", **_decode("step", 1, 4099, 4099, PAPER)},
        # the serving batch of the benchmark: 16 sequences of 8192 tokens
        {"name": "step_16x8k", **_decode("step", 16, 8192, 8192, G32)},
        # the same with the step's activations in pinned host memory
        {"name": "step_16x8k_host", **_decode("step", 16, 8192, 8192, G32, host=True)},
        # the same batch in the paper's configuration
        {"name": "step_16x8k_paper", **_decode("step", 16, 8192, 8192, PAPER)},
        # long-context retrieval: one sequence of 131072 tokens
        {"name": "decode_1x128k", **_decode("decode", 1, 131072, 131072, G32)},
        # a full ragged serving batch
        {"name": "step_ragged_128", **_decode("step", 128, 1024, 32768, G32, lens=1)},
        # many short requests on half the heads (two-way tensor parallel), value rotation
        # folded into the model, compact records
        {"name": "step_ragged_37_fold", **_decode("step", 37, 100, 6001,
                                                  dict(PAPER, sink=0, recent=0), h_kv=4, fold=True,
                                                  lens=2)},
        # a few new tokens per sequence written outside a step (draft tokens)
        {"name": "append_40x3", **_append(40, 3, 3, 2049, G32)},
        # one chunk of a chunked prefill in the paper's configuration
        {"name": "append_chunk_2000", **_append(1, 2000, 2000, 4096, PAPER)},
        # prefill of four long prompts
        {"name": "append_4x32k", **_append(4, 32768, 32768, 0, G32)},
        # offline: rotations of one KV head at the paper's trace size, one selection period of
        # Adam steps (over the paper's 80 the trajectory amplifies the last bit of a sum until a
        # code flips, so that no two orders of summation can be compared)
        {"name": "calibrate_head", **_calib(2048, 64, 4096, 20, PAPER)},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["decode", "decode", "step", "step", "step", "step", "append", "append",
                       "append", "calib"])
    opts = rng.choice([G32, G32, PAPER, dict(PAPER, sink=0, recent=0), dict(G32, sink=16, recent=100)])
    if kind == "calib":
        return _calib(_log(rng, 256, 2048), rng.choice([16, 33, 64]), rng.choice([1024, 2560, 4096]),
                      _log(rng, 4, 20), opts)
    h_kv = rng.choice([2, 4, 8, 8, 8, 8])
    lens = rng.randrange(1 << 20)
    if kind == "append":
        n = _log(rng, 1, 131072)  # new tokens of the call
        B = min(n, _log(rng, 1, 64))
        per = n // B
        return _append(B, max(1, int(per * rng.uniform(0.3, 1.0))), per, rng.choice([0, 0, _log(rng, 1, 4096)]),
                       opts, h_kv, lens)
    B = _log(rng, 1, 128)
    hi = _log(rng, 64, min(131072, (1 << 20) // B))
    lo = hi if rng.random() < 0.4 else max(1, int(hi * rng.uniform(0.05, 1.0)))
    return _decode(kind, B, lo, hi, opts, h_kv, rng.random() < 0.25,
                   kind == "step" and rng.random() < 0.25, lens)


# ------------------------------------------------------------------ inputs

def _lens(c):
    r = random.Random(c["lens"])
    return [r.randint(c["ctx_lo"], c["ctx_hi"]) for _ in range(c["B"])]


def _gen(seed, stream):
    return torch.Generator(device=DEV).manual_seed(seed * 1000003 + stream)


def _t4(shape, g):
    """Student-t with 4 degrees of freedom, float32."""
    z = torch.randn(shape, generator=g, device=DEV)
    e = torch.rand(shape, generator=g, device=DEV).clamp_min_(1e-12).log_()
    e += torch.rand(shape, generator=g, device=DEV).clamp_min_(1e-12).log_()
    return z.div_(e.mul_(-0.5).sqrt_())


def _model(c, seed):
    """Rotations R_k, R_v, the key mean (four offset channels per head)."""
    h = c["h_kv"]
    g = torch.Generator().manual_seed(seed * 7919 + 17)
    R = []
    for _ in range(2):
        Q, U = torch.linalg.qr(torch.randn(h, D, D, generator=g, dtype=torch.float64))
        R.append((Q * torch.sign(torch.diagonal(U, dim1=1, dim2=2))[:, None, :]).float())
    mu = torch.zeros(h, D)
    for i in range(h):
        ch = torch.randperm(D, generator=g)[:4]
        mu[i, ch] = (6 + 4 * torch.rand(4, generator=g)) * (torch.rand(4, generator=g) - 0.5).sign()
    return R[0], R[1], mu


def _kv(n, mu, g):
    """bf16 keys and values [n][h_kv][128]."""
    h = mu.shape[0]
    k = (_t4((n, h, D), g) + mu.to(DEV)).bfloat16()
    return k, _t4((n, h, D), g).bfloat16()


def _quantize(z, group, clip):
    """float32 z [n][h][128] -> codes [n][h][128], scale and min fp16 [n][h][128 / group]."""
    zg = z.unflatten(2, (D // group, group))
    mn = clip * zg.amin(3, keepdim=True)
    mx = clip * zg.amax(3, keepdim=True)
    r = mx - mn
    code = ((torch.minimum(torch.maximum(zg, mn), mx) - mn) * (3.0 / r)).round_().clamp_(0, 3)
    return code.flatten(2), (r / 3.0).half().squeeze(3), mn.half().squeeze(3)


def _rotated(x, R, sub, dtype=torch.float32):
    z = torch.einsum("nhi,hij->nhj", x.to(dtype), R.to(DEV, dtype))
    if sub is not None:
        z = z - torch.einsum("hi,hij->hj", sub.to(DEV, dtype), R.to(DEV, dtype))
    return z.float()


def _layout(group):
    """Record bytes, value metadata offset, metadata bytes per slot."""
    return (1152, 1088, 4) if group == 128 else (1536, 1280, 16)


def _filled_pool(c, num_pages, R_k, R_v, mu, seed):
    """uint8 [num_pages][h_kv][record]: every slot of every page holds a token's record."""
    rec, vmo, mb = _layout(c["group"])
    h = c["h_kv"]
    pool = torch.empty(num_pages, h, rec, dtype=torch.uint8, device=DEV)
    g = _gen(seed, 1)
    shift = torch.tensor([1, 4, 16, 64], device=DEV, dtype=torch.float32)
    for p0 in range(0, num_pages, 4096):
        P = min(4096, num_pages - p0)
        k, v = _kv(P * PAGE, mu, g)
        for x, R, sub, clip, co, mo in ((k, R_k, mu, c["clip_k"], 0, 1024),
                                        (v, None if c["fold"] else R_v, None, c["clip_v"], 512, vmo)):
            z = x.float() if R is None else _rotated(x, R, sub)
            code, s, m = _quantize(z, c["group"], clip)
            byte = (code.unflatten(2, (4, 8, 4)) * shift).sum(4)            # [n][h][g][w]
            byte = byte.transpose(2, 3).reshape(P, PAGE, h, 32).to(torch.uint8)
            meta = torch.stack([s, m], 3).reshape(P, PAGE, h, -1).view(torch.uint8)
            dst = pool[p0:p0 + P]
            dst[:, :, co:co + 512].unflatten(2, (PAGE, 32)).copy_(byte.transpose(1, 2))
            dst[:, :, mo:mo + PAGE * mb].unflatten(2, (PAGE, mb)).copy_(meta.transpose(1, 2))
    return pool


def _tables(tokens, seed):
    """Shuffled block table int32 [B][max_pages] and the number of pages."""
    n = [(t + PAGE - 1) // PAGE for t in tokens]
    perm = torch.randperm(sum(n), generator=torch.Generator().manual_seed(seed)).int()
    bt = torch.full((len(n), max(n)), -1, dtype=torch.int32)
    o = 0
    for b, x in enumerate(n):
        bt[b, :x] = perm[o:o + x]
        o += x
    return bt, sum(n)


def _decode_inputs(c, seed):
    """Everything a decode or a step reads, on the GPU."""
    ctx = _lens(c)
    B, h = c["B"], c["h_kv"]
    new = 1 if c["kind"] == "step" else 0
    R_k, R_v, mu = _model(c, seed)
    bt, pages = _tables([n + new for n in ctx], seed)
    g = _gen(seed, 2)
    s = {"R_k": R_k, "R_v": R_v, "mu": mu, "ctx": ctx, "bt": bt.to(DEV),
         "pool": _filled_pool(c, pages, R_k, R_v, mu, seed),
         "q": torch.randn(B, 4 * h, D, generator=g, device=DEV).bfloat16(),
         "seq": torch.tensor([n + new for n in ctx], dtype=torch.int32, device=DEV)}
    if new:
        s["k"], s["v"] = _kv(B, mu, g)
        s["cu"] = torch.arange(B + 1, dtype=torch.int32, device=DEV)
        s["pos0"] = torch.tensor(ctx, dtype=torch.int32, device=DEV)
    rows = c["sink"] + c["recent"]
    if rows:  # every row of the window store holds some token's key and value
        wk, wv = _kv(B * rows, mu, g)
        s["win"] = torch.stack([x.view(B, rows, h, D).transpose(1, 2) for x in (wk, wv)], 2).contiguous()
        s["slot"] = torch.randperm(B, generator=torch.Generator().manual_seed(seed)).int().to(DEV)
    return s


def _params(c, s):
    return optr.optr_params_create(s["R_k"], None if c["fold"] else s["R_v"], s["mu"], 4 * c["h_kv"],
                                   clip_k=c["clip_k"], clip_v=c["clip_v"], sink=c["sink"],
                                   recent=c["recent"], group=c["group"])


def prepare(case, seed):
    c = case
    if c["kind"] == "calib":
        return _prepare_calib(c, seed)
    if c["kind"] == "append":
        n = _lens(c)
        R_k, R_v, mu = _model(c, seed)
        bt, pages = _tables([c["pos0"] + x for x in n], seed)
        s = {"R_k": R_k, "R_v": R_v, "mu": mu, "bt": bt.to(DEV)}
        s["k"], s["v"] = _kv(sum(n), mu, _gen(seed, 2))
        cu = [0]
        for x in n:
            cu.append(cu[-1] + x)
        s["cu"] = torch.tensor(cu, dtype=torch.int32, device=DEV)
        s["pos0"] = torch.full((c["B"],), c["pos0"], dtype=torch.int32, device=DEV)
        s["p"] = _params(c, s)
        s["pool"] = optr.new_pool(s["p"], pages)
        if c["sink"] + c["recent"]:
            s["win"] = optr.new_windows(s["p"], c["B"])
            s["slot"] = torch.arange(c["B"], dtype=torch.int32, device=DEV)
    else:
        s = _decode_inputs(c, seed)
        s["p"] = _params(c, s)
        s["out"] = torch.empty(c["B"], 4 * c["h_kv"], D, device=DEV)
        s["ws"] = optr.new_workspace(s["p"], c["B"], s["bt"].shape[1])
        if c["host"]:
            for x in ("q", "k", "v", "out"):
                s[x] = s[x].cpu().pin_memory()
    s["kind"] = c["kind"]
    return s


def run(state):
    s = state
    if s["kind"] == "calib":
        R_K, R_V, mu, hk, hv = optr.optr_calibrate_head(s["cfg"], s["q"], s["K"], s["V"], s["t"],
                                                        s["W"], held=s["held"])
        return {"R_K": R_K, "R_V": R_V, "mu": mu, "hist_k": hk, "hist_v": hv}
    win = "win" in s
    if s["kind"] == "append":
        a = (s["p"], s["k"], s["v"], s["cu"], s["pos0"], s["bt"], s["pool"])
        if win:
            optr.optr_kv_append_win(*a, s["win"], s["slot"])
            return {"pool": s["pool"], "win": s["win"]}
        optr.optr_kv_append(*a)
        return {"pool": s["pool"]}
    if s["kind"] == "decode":
        a = (s["p"], s["q"], s["bt"], s["seq"], s["pool"])
        if win:
            optr.optr_decode_attention_win(*a, s["win"], s["slot"], s["out"], s["ws"])
        else:
            optr.optr_decode_attention(*a, s["out"], s["ws"])
        return {"out": s["out"]}
    a = (s["p"], s["q"], s["k"], s["v"], s["cu"], s["pos0"], s["bt"], s["seq"], s["pool"])
    if win:
        optr.optr_decode_step_win(*a, s["win"], s["slot"], s["out"], s["ws"])
        return {"out": s["out"], "pool": s["pool"], "win": s["win"]}
    optr.optr_decode_step(*a, s["out"], s["ws"])
    return {"out": s["out"], "pool": s["pool"]}


# -------------------------------------------------------------------- work

def work(case):
    c = case
    if c["kind"] == "calib":
        # the contractions of the objectives and their gradients per Adam step: four (keys) and
        # two (values) of [g nt][T][128], five each of [T][128][128]
        att, rot = 2.0 * c["g"] * c["nt"] * c["T"] * D, 2.0 * c["T"] * D * D
        byt = 8 * 2 * (2 * c["T"] * D + c["nt"] * c["g"] * D) + 8 * c["g"] * c["d_model"] * D + 8 * 2 * D * D
        return {"bytes": byt, "flops": c["steps"] * (6 * att + 10 * rot)}
    h, B = c["h_kv"], c["B"]
    rec = 72 if c["group"] == 128 else 96
    rows = c["sink"] + c["recent"]
    n = _lens(c)
    if c["kind"] == "append":
        t = sum(n)
        kept = sum(max(0, min(c["pos0"] + x, c["sink"]) - c["pos0"]) + min(x, c["recent"]) for x in n) if rows else 0
        return {"bytes": t * h * (512 + rec) + kept * h * 512, "flops": t * h * 2 * 2.0 * D * D}
    new = 1 if c["kind"] == "step" else 0
    byt, tok = B * 4 * h * D * (2 + 4) + new * B * h * (512 + rec + (512 if rows else 0)), 0
    for x in n:
        x += new
        w = min(x, c["sink"]) + max(0, x - max(c["sink"], x - c["recent"]))
        byt += h * ((x - w) * rec + w * 512)
        tok += x
    return {"bytes": byt, "flops": tok * h * 4 * 2 * 2.0 * D + B * h * 8 * 2.0 * D * D + new * B * h * 4.0 * D * D}


# ------------------------------------------------------------------- exact

def exact(case, seed):
    c = case
    if c["kind"] == "calib":
        return _exact_calib(c, seed)
    if c["kind"] == "append":
        return None  # bytes
    s = _decode_inputs(c, seed)
    rec, vmo, mb = _layout(c["group"])
    h, f8 = c["h_kv"], torch.float64
    new = c["kind"] == "step"
    R_k, R_v, mu = (s[x].to(DEV, f8) for x in ("R_k", "R_v", "mu"))

    def values(r, co, mo):  # records [P][h][rec] -> dequantized [P * 16][h][128]
        byte = r[:, :, co:co + 512].reshape(-1, h, PAGE, 8, 4)                     # [w][g]
        bits = torch.stack([(byte >> (2 * i)) & 3 for i in range(4)], 5)           # [w][g][r]
        code = bits.permute(0, 2, 1, 4, 3, 5).reshape(-1, h, D).to(f8)
        meta = r[:, :, mo:mo + PAGE * mb].reshape(-1, h, PAGE, mb).contiguous().view(torch.float16)
        meta = meta.transpose(1, 2).reshape(-1, h, mb // 4, 2).to(f8).repeat_interleave(c["group"], 2)
        return code * meta[..., 0] + meta[..., 1]

    def requantized(x, R, sub, clip):
        z = x.float() if R is None else _rotated(x, R, sub, f8)
        code, sc, mn = _quantize(z, c["group"], clip)
        return (code.to(f8) * sc.to(f8).repeat_interleave(c["group"], 2)
                + mn.to(f8).repeat_interleave(c["group"], 2))

    if new:
        nk = requantized(s["k"], s["R_k"], s["mu"], c["clip_k"])
        nv = requantized(s["v"], None if c["fold"] else s["R_v"], None, c["clip_v"])
    out = torch.empty(c["B"], 4 * h, D, dtype=f8, device=DEV)
    for b, n0 in enumerate(s["ctx"]):
        n = n0 + new
        q = s["q"][b].to(f8).view(h, 4, D)
        qr = torch.einsum("hgi,hij->hgj", q, R_k)
        r = s["pool"][s["bt"][b, :(n + PAGE - 1) // PAGE].long()]
        kd, vd = values(r, 0, 1024)[:n], values(r, 512, vmo)[:n]
        if new:
            kd[n - 1], vd[n - 1] = nk[b], nv[b]
        lg = torch.einsum("hgd,nhd->hgn", qr, kd)
        pos = torch.arange(n, device=DEV)
        w = pos[(pos < c["sink"]) | (pos >= n - c["recent"])] if c["sink"] + c["recent"] else pos[:0]
        if w.numel():
            row = torch.where(w < c["sink"], w, c["sink"] + (w - c["sink"]) % max(1, c["recent"]))
            wk, wv = (s["win"][s["slot"][b].long(), :, i][:, row].to(f8) for i in (0, 1))  # [h][w][D]
            if new:
                wk[:, w == n - 1], wv[:, w == n - 1] = s["k"][b].to(f8)[:, None], s["v"][b].to(f8)[:, None]
            lg[:, :, w] = torch.einsum("hgd,hwd->hgw", q, wk - mu[:, None])
        p = torch.softmax(lg / math.sqrt(D), 2)
        pi = p.clone()
        pi[:, :, w] = 0
        o = torch.einsum("hgn,nhd->hgd", pi, vd)
        if not c["fold"]:
            o = torch.einsum("hgj,hij->hgi", o, R_v)
        if w.numel():
            o = o + torch.einsum("hgw,hwd->hgd", p[:, :, w], wv)
        out[b] = o.reshape(4 * h, D)
    r = {"out": out}
    if new:
        r["pool"] = None
        if "win" in s:
            r["win"] = None
    return r


# ------------------------------------------------------------- calibration

def _trace(c, seed, mu, stream):
    g = _gen(seed, stream)
    T, nt = c["T"], min(c["nt"], c["T"])
    K = (_t4((T, D), g) + mu.to(DEV)).double()
    V = _t4((T, D), g).double()
    q = torch.randn(nt, c["g"], D, generator=g, device=DEV, dtype=torch.float64)
    return q, K, V, torch.arange(T - nt, T, dtype=torch.int32, device=DEV)


def _prepare_calib(c, seed):
    mu = _model({"h_kv": 1}, seed)[2][0]
    q, K, V, t = _trace(c, seed, mu, 1)
    W = torch.randn(c["g"], c["d_model"], D, generator=_gen(seed, 3), device=DEV, dtype=torch.float64)
    cfg = optr.calib_config(c["g"], c["d_model"], c["T"], q.shape[0], c["T"], q.shape[0], steps=c["steps"],
                            group=c["group"], sink=c["sink"], recent=c["recent"], clip_k=c["clip_k"],
                            clip_v=c["clip_v"])
    return {"kind": "calib", "cfg": cfg, "q": q, "K": K, "V": V, "t": t, "W": W / math.sqrt(c["g"] * D),
            "held": _trace(c, seed, mu, 2)}


def _exact_calib(c, seed):
    """The calibration written out with autograd: Adam (lr 0.02) on the skew generators, the
    best of every 20th rotation on the held-out trace."""
    s = _prepare_calib(c, seed)
    f8, scale = torch.float64, 1.0 / math.sqrt(D)
    H = torch.ones(1, 1, dtype=f8, device=DEV)
    while H.shape[0] < D:
        H = torch.cat([torch.cat([H, H], 1), torch.cat([H, -H], 1)], 0)
    H = H / math.sqrt(D)
    mu = s["K"].mean(0)
    W = s["W"]

    def q2(z, clip):
        zg = z.detach().unflatten(1, (D // c["group"], c["group"]))
        mn, mx = clip * zg.amin(2, keepdim=True), clip * zg.amax(2, keepdim=True)
        r = mx - mn
        code = ((torch.minimum(torch.maximum(zg, mn), mx) - mn) * (3.0 / r)).round().clamp(0, 3)
        zh = (code * (r / 3.0).float().half().to(f8) + mn.float().half().to(f8)).flatten(1)
        inside = ((zg >= mn) & (zg <= mx)).flatten(1).to(f8)
        return zh + inside * (z - z.detach())

    def probs(q, x, xw, win, t):
        lg = torch.einsum("tgd,sd->gts", q, x)
        if win is not None:
            lg = torch.where(win, torch.einsum("tgd,sd->gts", q, xw), lg)
        causal = torch.arange(x.shape[0], device=DEV)[None] <= t[:, None]
        return torch.softmax(torch.where(causal, lg * scale, -math.inf), 2)

    def window(tr):
        if not c["sink"] + c["recent"]:
            return None
        pos = torch.arange(tr[1].shape[0], device=DEV)[None]
        return (pos < c["sink"]) | (pos > tr[3][:, None] - c["recent"])

    traces = ((s["q"], s["K"], s["V"], s["t"]), s["held"])
    wins = [window(tr) for tr in traces]
    ref = [probs(tr[0], tr[1], None, None, tr[3]) for tr in traces]
    n = c["g"] * s["q"].shape[0]

    def key_probs(R, i):
        q, K, _, t = traces[i]
        kc = K - mu
        return probs(q, q2(kc @ R, c["clip_k"]) @ R.T, kc, wins[i], t)

    def key_loss(R, i):
        p, pk = ref[i], key_probs(R, i)
        kl = (p * (p.clamp_min(1e-300).log() - pk.clamp_min(1e-300).log())).sum()
        e = (pk - p) @ traces[i][2] @ W.transpose(1, 2)
        return (kl + (e * e).sum() / c["d_model"]) / n

    def value_loss(R, i):
        V = traces[i][2]
        p = phat[i] if wins[i] is None else phat[i].masked_fill(wins[i], 0.0)
        e = p @ (q2(V @ R, c["clip_v"]) @ R.T - V) @ W.transpose(1, 2)
        return (e * e).sum() / c["d_model"] / n

    def adam(loss):
        A = torch.zeros(D, D, dtype=f8, device=DEV)
        m, v, hist, best = torch.zeros_like(A), torch.zeros_like(A), [], None
        for i in range(c["steps"] + 1):
            A.requires_grad_(True)
            R = H @ torch.linalg.matrix_exp(A - A.T)
            if i % 20 == 0 or i == c["steps"]:
                with torch.no_grad():
                    score = float(loss(R, 1))
                if best is None or score < best[0]:
                    best = (score, R.detach())
            if i == c["steps"]:
                break
            x = loss(R, 0)
            (g,) = torch.autograd.grad(x, A)
            hist.append(float(x.detach()))
            m, v = 0.9 * m + 0.1 * g, 0.999 * v + 0.001 * g * g
            A = A.detach() - 0.02 * (m / (1 - 0.9 ** (i + 1))) / ((v / (1 - 0.999 ** (i + 1))).sqrt() + 1e-8)
        return best[1], torch.tensor(hist, dtype=f8, device=DEV)

    R_K, hist_k = adam(key_loss)
    with torch.no_grad():
        phat = [key_probs(R_K, i) for i in (0, 1)]
    R_V, hist_v = adam(value_loss)
    return {"R_K": R_K, "R_V": R_V, "mu": mu, "hist_k": hist_k, "hist_v": hist_v}
