"""Timing cases: the calls a program that serves long-video requests makes.

A case is a dict of plain values; ``prepare`` makes what such a program holds
before the call (inputs drawn from a seed, output buffers, workspace, and for
a decode step its captured graph), ``run`` makes the call through
``paper_2608_24063_gb300.viscache`` and returns its outputs, ``work`` counts
what the call cannot do without, and ``exact`` gives the outputs in 64 bits
from plain torch.

Inputs follow the workloads of the repository's benchmark: approximately unit
normal queries, keys and values, keys with 2% outlier channels (x 10), an
attention-sink token, frames of 196 (or 256) tokens that repeat from one to
the next (correlation 0.9) and eight contiguous relevant frames.
"""
import ctypes
import math
import random
from fractions import Fraction

import torch

from paper_2608_24063_gb300 import viscache as vc

DEV = "cuda"
MU, TAU = 0.7, 1.0
RATIOS = (19, 23, 28)                   # retention in percent

_7B = dict(L=28, Hq=28, Hkv=4, d=128, dtype="bf16", frame=196)
_72B = dict(L=80, Hq=64, Hkv=8, d=128, dtype="bf16", frame=256)


def _compress(name, shape, n, W, rr, **more):
    return dict(name=name, kind="compress", **shape,
                **{**dict(n_req=1, n_lo=n, n_hi=n, w_lo=W, w_hi=W, rr=rr, rank="shared", mix=0), **more})


def _after(name, kind, n_req, n, rr, **more):
    return dict(name=name, kind=kind, **_7B,
                **{**dict(n_req=n_req, n_lo=n, n_hi=n, w_lo=64, w_hi=64, rr=rr, mix=0), **more})


def listed():
    return [
        # one layer of a small fp32 model: the shortest pass there is, launches and latency
        _compress("compress_f32_1layer", dict(L=1, Hq=8, Hkv=4, d=64, dtype="f32", frame=0), 1024, 32, 25),
        # a short clip (16 frames) on the 7B shape, right after its prefill
        _compress("compress_7b_n3136", _7B, 3136, 64, 28),
        # the usual long video (64 frames) on the 7B shape
        _compress("compress_7b_n12544", _7B, 12544, 64, 19),
        # the same video where every layer ranks its own tokens
        _compress("compress_7b_layer_rank", _7B, 12544, 64, 19, rank="layer"),
        # a server's batch: eight requests of different lengths, windows and retention in one call
        _compress("compress_7b_ragged8", _7B, 2048, 32, 0, n_req=8, n_hi=16384, w_hi=128, mix=5),
        # the largest request: 128 frames on the 72B shape
        _compress("compress_72b_n32768", _72B, 32768, 128, 22),
        # one token of one request: a decode step of 28 layers over its compressed cache
        _after("decode_7b_1req", "decode", 1, 12544, 19, t_lo=512, t_hi=512),
        # one token of each of 16 requests
        _after("decode_7b_16req", "decode", 16, 12544, 19, t_lo=512, t_hi=512),
        # the same step over the 4-bit form of the cache
        _after("decode_kv4_7b_16req", "decode_kv4", 16, 12544, 19, t_lo=512, t_hi=512),
        # the caches of 16 requests into their 4-bit form, and back
        _after("quantize_7b_16req", "quantize", 16, 12544, 19),
        _after("dequantize_7b_16req", "dequantize", 16, 12544, 19),
        # keyframes of 64 videos of 64 frames, before the prefill
        dict(name="scout_64x64", kind="scout", n_req=64, f_lo=64, f_hi=64, D=512, p_num=3, p_den=4, mix=0),
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["compress", "compress", "compress", "f32", "decode", "decode", "decode_kv4",
                       "quantize", "dequantize", "scout"])
    mix = rng.randrange(1, 1 << 20)
    if kind == "scout":
        lo = _log_int(rng, 12, 128)
        c = dict(kind=kind, n_req=_log_int(rng, 1, 64), f_lo=lo, f_hi=min(128, lo + rng.randrange(0, 48)),
                 D=rng.choice([512, 512, 768]), p_num=rng.choice([1, 2, 3]), p_den=4, mix=mix)
        return c
    if kind == "f32":
        n = _log_int(rng, 300, 4096)
        return {k: v for k, v in _compress("", dict(L=rng.randrange(1, 5), Hq=8, Hkv=rng.choice([2, 4]),
                                                    d=rng.choice([64, 64, 128]), dtype="f32", frame=0),
                                           n, rng.randrange(8, 65), rng.choice(RATIOS), mix=mix).items()
                if k != "name"}
    rr = rng.choice(RATIOS)
    if kind == "compress":
        big = rng.random() < 0.2
        n_req = 1 if big else rng.choice([1, 1, 2, 3, 5])
        lo = _log_int(rng, 512, 6000 if big else 16384)
        hi = lo if n_req == 1 else min(16384, lo + rng.randrange(1, 6000))
        w = rng.randrange(16, 129)
        c = _compress("", _72B if big else _7B, lo, w, rr if n_req == 1 else 0, n_req=n_req, n_hi=hi,
                      w_hi=w if n_req == 1 else 128, rank=rng.choice(["shared", "shared", "shared", "layer"]), mix=mix)
    else:
        n_req = _log_int(rng, 1, 24)
        lo = _log_int(rng, 700, 16384)
        c = _after("", kind, n_req, lo, rr, n_hi=min(16384, lo + rng.randrange(0, 4000)), mix=mix)
        if kind.startswith("decode"):
            t = _log_int(rng, 16, 900)
            c.update(t_lo=t, t_hi=t + rng.randrange(0, 300))
    c.pop("name")
    return c


# ---------------------------------------------------------------------------
# sizes

def _requests(c):
    """(n, W, retention percent) of every request; sizes between bounds come from the case's `mix`."""
    r = random.Random(c["mix"])
    return [(r.randint(c["n_lo"], c["n_hi"]), r.randint(c["w_lo"], c["w_hi"]), c["rr"] or r.choice(RATIOS))
            for _ in range(c["n_req"])]


def _text(c):
    r = random.Random(c["mix"] + 1)
    return [r.randint(c["t_lo"], c["t_hi"]) for _ in range(c["n_req"])]


def _frames(c):
    r = random.Random(c["mix"])
    return [r.randint(c["f_lo"], c["f_hi"]) for _ in range(c["n_req"])]


def _round(x):
    return math.floor(x + Fraction(1, 2))


def _budgets(L, n, rr):
    """Parabolic layer budgets B_l and the survivors Nq, in exact rationals."""
    h = max(min(2, L), min(L, _round(Fraction(3 * L, 4))))
    b = [Fraction(1) if h == 1 else 1 - Fraction(l * l, 2 * (h - 1) ** 2) for l in range(h)]
    T = _round(Fraction(rr, 100) * n * L)
    share = [T * x / sum(b) for x in b]
    B = [math.floor(x) for x in share]
    for l in sorted(range(h), key=lambda l: (B[l] - share[l], l))[:T - sum(B)]:
        B[l] += 1
    Nq = max(B[0], min(n, _round(Fraction(T) / (h * Fraction(3, 4)))))
    return B + [0] * (L - h), Nq


def _batch(c):
    reqs = _requests(c)
    return (vc.Batch([r[0] for r in reqs], [r[1] for r in reqs], [(r[2], 100) for r in reqs]),
            vc.make_params(c["L"], c["Hq"], c["Hkv"], c["d"], vc.VC_BF16 if c["dtype"] == "bf16" else vc.VC_F32,
                           mu=MU, tau=TAU,
                           rank_mode=vc.VC_RANK_PER_LAYER if c.get("rank") == "layer" else vc.VC_RANK_SHARED))


# ---------------------------------------------------------------------------
# inputs

def _dtype(c):
    return torch.bfloat16 if c["dtype"] == "bf16" else torch.float32


def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed))


def _randn(g, *shape):
    return torch.randn(*shape, generator=g, device=DEV)


def _outlier_scale(c, g):
    """[L][Hkv][1][d] key channel scales: 2% of the channels x 10."""
    L, H, d = c["L"], c["Hkv"], c["d"]
    s = torch.ones(L, H, d, device=DEV)
    pick = torch.rand(L, H, d, generator=g, device=DEV).topk(math.ceil(0.02 * d), dim=-1).indices
    return s.scatter_(-1, pick, 10.0).unsqueeze(2)


def _request_inputs(c, r, g):
    """Qw [L][Hq][W][d], K, V [L][Hkv][n][d] of request r."""
    n, W, _ = _requests(c)[r]
    L, Hq, H, d, P = c["L"], c["Hq"], c["Hkv"], c["d"], c["frame"]
    dt = _dtype(c)
    q = _randn(g, L, Hq, W, d).to(dt)
    mean = q.float().view(L, H, -1, d).mean(2)                       # along this the planted keys move
    no = math.ceil(0.02 * d) if P else 0
    sigma = math.sqrt((d - no + 100 * no) / d)
    push = mean * (sigma * math.sqrt(d) / mean.square().sum(-1, keepdim=True))
    if P:
        scale, F = _outlier_scale(c, g), -(-n // P)
        f0 = int(torch.randint(0, max(1, F - 7), (1,), generator=g, device=DEV))
        planted = slice(f0 * P, min(n, (f0 + 8) * P))
    else:                                                             # no frames: 5% relevant tokens
        planted = torch.randperm(n, generator=g, device=DEV)[:max(1, n // 20)]
    K = torch.empty(L, H, n, d, dtype=dt, device=DEV)
    V = torch.empty(L, H, n, d, dtype=dt, device=DEV)
    step = max(1, (1 << 28) // (H * n * d))                           # layers at a time
    for l0 in range(0, L, step):
        l1 = min(L, l0 + step)
        for out in (K, V):
            if P:
                x = _randn(g, l1 - l0, H, F, P, d)
                for f in range(1, F):
                    x[:, :, f].mul_(math.sqrt(1 - 0.81)).add_(x[:, :, f - 1], alpha=0.9)
                x = x.view(l1 - l0, H, F * P, d)[:, :, :n]
            else:
                x = _randn(g, l1 - l0, H, n, d)
            if out is K:
                if P:
                    x = x * scale[l0:l1]
                    x[:, :, 0] += 8 * push[l0:l1]
                x[:, :, planted] += 3 * push[l0:l1].unsqueeze(2)
            out[l0:l1] = x.to(dt)
    return q, K, V


def _pass_inputs(c, seed):
    g = _gen(seed)
    return [_request_inputs(c, r, g) for r in range(c["n_req"])]


def _packed(tensors):
    return tensors[0] if len(tensors) == 1 else torch.cat([t.reshape(-1) for t in tensors])


def _cache(c, seed):
    """A compressed cache: K, V rows (request, layer, KV head, kept row) and the row count of each segment."""
    g = _gen(seed)
    K, V, segs = [], [], []
    for n, _, rr in _requests(c):
        B, _ = _budgets(c["L"], n, rr)
        scale = _outlier_scale(c, g)
        for l, b in enumerate(B):
            segs.append(b)
            if b:
                K.append((_randn(g, c["Hkv"], b, c["d"]) * scale[l]).to(_dtype(c)).view(-1, c["d"]))
                V.append(_randn(g, c["Hkv"], b, c["d"]).to(_dtype(c)).view(-1, c["d"]))
    return torch.cat(K), torch.cat(V), segs


def _step_inputs(c, seed):
    """Query rows [L][n_req][Hq][d] and each layer's text rows [L][sum Hkv T][d]."""
    g = _gen(seed + 7919)
    rows = c["Hkv"] * sum(_text(c))
    dt = _dtype(c)
    return (_randn(g, c["L"], c["n_req"], c["Hq"], c["d"]).to(dt), _randn(g, c["L"], rows, c["d"]).to(dt),
            _randn(g, c["L"], rows, c["d"]).to(dt))


def _embeddings(c, seed):
    """Frame embeddings (scenes of eight near-duplicate frames) and prompts near one scene of each video."""
    g = _gen(seed)
    H, P = [], []
    for F in _frames(c):
        centres = _randn(g, -(-F // 8), c["D"])
        H.append(centres.repeat_interleave(8, 0)[:F] + 0.5 * _randn(g, F, c["D"]))
        at = int(torch.randint(0, centres.shape[0], (1,), generator=g, device=DEV))
        P.append(centres[at] + 0.5 * _randn(g, c["D"]))
    return torch.cat(H), torch.stack(P)


# ---------------------------------------------------------------------------
# the calls

def prepare(case, seed):
    c = case
    s = {"case": c}
    if c["kind"] == "scout":
        F = _frames(c)
        H, P = _embeddings(c, seed)
        k = sum(-(-f * c["p_num"] // c["p_den"]) for f in F)
        out = (torch.empty(k, dtype=torch.int32, device=DEV), torch.empty(k, dtype=torch.int32, device=DEV),
               torch.empty(k, device=DEV))
        need = vc.lib().viscache_scout_workspace_size(len(F), (ctypes.c_int32 * len(F))(*F), c["D"])
        s.update(H=H, P=P, F=F, out=out, ws=torch.empty(need, dtype=torch.uint8, device=DEV))
        return s
    batch, prm = _batch(c)
    s.update(batch=batch, prm=prm)
    if c["kind"] == "compress":
        q, k, v = zip(*_pass_inputs(c, seed))
        s.update(Q=_packed(q), K=_packed(k), V=_packed(v))
        rows = vc.compressed_rows(batch, prm)
        s.update(K_out=torch.empty(rows, c["d"], dtype=_dtype(c), device=DEV),
                 V_out=torch.empty(rows, c["d"], dtype=_dtype(c), device=DEV),
                 idx=torch.empty(rows, dtype=torch.int32, device=DEV),
                 ws=torch.empty(vc.prunekv_workspace_size(batch, prm), dtype=torch.uint8, device=DEV))
        return s
    K, V, _ = _cache(c, seed)
    if c["kind"] == "quantize":
        s.update(K=K, V=V, out=vc.viscache_kv4_quantize(batch, prm, K, V))
    elif c["kind"] == "dequantize":
        s.update(kv4=vc.viscache_kv4_quantize(batch, prm, K, V), out=(torch.empty_like(K), torch.empty_like(V)))
    else:
        s.update(K=K, V=V)
        if c["kind"] == "decode_kv4":
            s["kv4"] = vc.viscache_kv4_quantize(batch, prm, K, V)
        q, kt, vt = _step_inputs(c, seed)
        T = _text(c)
        ws = torch.empty(vc.viscache_decode_workspace_size(batch, prm, T), dtype=torch.uint8, device=DEV)
        s.update(q=q, kt=kt, vt=vt, T=T, ws=ws, out=torch.empty_like(q))
        # the step as a graph, as a server keeps it for a batch
        side = torch.cuda.Stream()
        side.wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(side):
            _decode_step(s)
        torch.cuda.current_stream().wait_stream(side)
        torch.cuda.synchronize()
        s["graph"] = torch.cuda.CUDAGraph()
        with torch.cuda.graph(s["graph"]):
            _decode_step(s)
    return s


def _decode_step(s):
    for l in range(s["case"]["L"]):
        more = dict(K_text=s["kt"][l], V_text=s["vt"][l], n_text=s["T"], out=s["out"][l], ws=s["ws"])
        if "kv4" in s:
            vc.viscache_decode_attention_kv4(s["batch"], s["prm"], l, s["q"][l], s["kv4"], **more)
        else:
            vc.viscache_decode_attention(s["batch"], s["prm"], l, s["q"][l], s["K"], s["V"], **more)


def run(state):
    s, kind = state, state["case"]["kind"]
    if kind == "compress":
        K, V, idx = _call_compress(s)
        return {"K": K, "V": V, "idx": idx}
    if kind == "scout":
        c = s["case"]
        order, keys, gains, _ = vc.viscache_scout_mmr(s["H"], s["P"], s["F"], p=(c["p_num"], c["p_den"]),
                                                      out=s["out"], ws=s["ws"])
        return {"order": order, "keyframes": keys, "gains": gains}
    if kind == "quantize":
        kc, vcodes, kp, vp = vc.viscache_kv4_quantize(s["batch"], s["prm"], s["K"], s["V"], out=s["out"])
        return {"K_codes": kc, "V_codes": vcodes, "K_params": kp, "V_params": vp}
    if kind == "dequantize":
        K, V = vc.viscache_kv4_dequantize(s["batch"], s["prm"], *s["kv4"], out=s["out"])
        return {"K": K, "V": V}
    s["graph"].replay()
    return {"out": s["out"]}


def _call_compress(s):
    return vc.prunekv_compress(s["batch"], s["prm"], s["Q"], s["K"], s["V"], K_out=s["K_out"], V_out=s["V_out"],
                               idx_out=s["idx"], ws=s["ws"])


# ---------------------------------------------------------------------------
# what a call cannot do without

def work(case):
    c = case
    if c["kind"] == "scout":
        F = _frames(c)
        k = [-(-f * c["p_num"] // c["p_den"]) for f in F]
        return {"bytes": 4 * c["D"] * (sum(F) + len(F)) + 12 * sum(k), "flops": sum(f * f for f in F) * c["D"]}
    L, Hq, H, d = c["L"], c["Hq"], c["Hkv"], c["d"]
    e = 2 if c["dtype"] == "bf16" else 4
    nbytes = flops = 0
    text = _text(c) if "t_lo" in c else [0] * c["n_req"]
    for (n, W, rr), T in zip(_requests(c), text):
        B, Nq = _budgets(L, n, rr)
        kept, surv = H * sum(B), H * sum(Nq for b in B if b)
        if c["kind"] == "compress":
            # keys and queries once, the survivors' values once, the outputs
            nbytes += e * d * (H * n * L + Hq * W * L + surv + 2 * kept) + 4 * kept
            flops += 2 * Hq * W * n * d * L + 4 * H * d * sum(b * (Nq - b) for b in B)
            continue
        groups = H * sum(-(-b // 32) for b in B)
        form = 2 * kept * (d // 2) + 8 * groups * d + 8 * kept * (d // 32)     # 4-bit codes and parameters
        if c["kind"] in ("quantize", "dequantize"):
            nbytes += 2 * kept * d * e + form
            flops += 2 * 2 * kept * d
        else:
            nbytes += 2 * L * Hq * d * e + 2 * H * T * L * d * e
            nbytes += form if c["kind"] == "decode_kv4" else 2 * kept * d * e
            flops += 4 * d * (Hq // H) * (kept + H * T * L)
    return {"bytes": nbytes, "flops": flops}


# ---------------------------------------------------------------------------
# the outputs in 64 bits

def exact(case, seed):
    c = case
    if c["kind"] == "compress":
        # fp64 products of this many operations take half a minute and more
        return None if work(c)["flops"] > 4e12 else _exact_compress(c, seed)
    if c["kind"] == "scout":
        return _exact_scout(c, seed)
    if c["kind"] in ("quantize", "dequantize"):
        K, V, segs = _cache(c, seed)
        kc, kp, vcodes, vp = _quantized(c, K, V, segs)
        if c["kind"] == "quantize":
            return {"K_codes": None, "V_codes": None, "K_params": kp[0], "V_params": vp[0]}
        K, V = _expanded(c, kc, kp[1], vcodes, vp[1], segs)
        return {"K": K, "V": V}
    return _exact_decode(c, seed)


def _exact_compress(c, seed):
    Ks, Vs, idxs = [], [], []
    L, H, d = c["L"], c["Hkv"], c["d"]
    gap = math.inf
    for (n, W, rr), (q, k, v) in zip(_requests(c), _pass_inputs(c, seed)):
        B, Nq = _budgets(L, n, rr)
        s = torch.empty(L, H, n, dtype=torch.float64, device=DEV)
        for l in range(L):
            x = q[l].double().view(H, -1, d) @ k[l].double().transpose(1, 2) / math.sqrt(d)
            s[l] = torch.softmax(x, -1).sum(1)
        shared = c["rank"] == "shared"
        ranked, order = torch.sort(s.mean(0) if shared else s, dim=-1, descending=True, stable=True)
        for l in range(L):
            for cut in {B[l], Nq} if B[l] else ():
                a, b = (ranked if shared else ranked[l])[:, cut - 1:cut + 1].split(1, -1) if cut < n else (None, None)
                gap = min(gap, float(((a - b) / a).min())) if cut < n else gap
        for l in range(L):
            for g in range(H if B[l] else 0):
                o = order[g] if shared else order[l, g]
                keep, drop = o[:B[l]].sort().values, o[B[l]:Nq]
                vk, vd = v[l, g, keep].double(), v[l, g, drop].double()
                if len(drop):
                    vk = MU * vk + (1 - MU) * (torch.softmax(vk @ vd.T / TAU, -1) @ vd)
                Ks.append(k[l, g, keep].double())
                Vs.append(vk)
                idxs.append(keep)
    # two tokens at a cut with scores nearer than 32 bits tell apart: either may be kept, and the rows
    # between them move, so the rows have no value to be held to
    if gap < 3e-7:
        return None
    return {"K": torch.cat(Ks), "V": torch.cat(Vs), "idx": torch.cat(idxs).int()}


def _exact_scout(c, seed):
    H, P = _embeddings(c, seed)
    H, P = H.double(), P.double()
    H, P = H / H.norm(dim=1, keepdim=True), P / P.norm(dim=1, keepdim=True)
    order, keys, gains, at = [], [], [], 0
    for r, F in enumerate(_frames(c)):
        h = H[at:at + F]
        at += F
        sim, rel = (h @ h.T).cpu(), (h @ P[r]).cpu()
        red, free = torch.zeros(F, dtype=torch.float64), torch.ones(F, dtype=torch.bool)
        picks = []
        for i in range(-(-F * c["p_num"] // c["p_den"])):
            score = torch.where(free, 0.7 * rel - 0.3 * red, torch.tensor(-math.inf, dtype=torch.float64))
            f = int(score.argmax())
            picks.append(f)
            gains.append(float(score[f]))
            free[f] = False
            red = sim[f] if i == 0 else torch.maximum(red, sim[f])
        order += picks
        keys += sorted(picks)
    return {"order": torch.tensor(order, dtype=torch.int32), "keyframes": torch.tensor(keys, dtype=torch.int32),
            "gains": torch.tensor(gains, dtype=torch.float64)}


def _segments(c, segs):
    """(first row, rows) of every (request, layer, KV head) segment."""
    at = 0
    for b in segs:
        for _ in range(c["Hkv"] if b else 0):
            yield at, b
            at += b


def _group_of_rows(c, segs):
    """The key group of every row: 32 consecutive rows of a segment."""
    out, g = [], 0
    for _, b in _segments(c, segs):
        out.append(g + torch.arange(b, device=DEV) // 32)
        g += -(-b // 32)
    return torch.cat(out), g


def _quantized(c, K, V, segs):
    """Codes, and (scale, min) in 64 bits and as the 32-bit format stores them, of keys and values."""
    d = c["d"]
    rows, groups = _group_of_rows(c, segs)
    rows = rows.unsqueeze(1).expand(-1, d)
    lo = torch.full((groups, d), math.inf, device=DEV).scatter_reduce_(0, rows, K.float(), "amin")
    hi = torch.full((groups, d), -math.inf, device=DEV).scatter_reduce_(0, rows, K.float(), "amax")
    v = V.float().view(-1, d // 32, 32)
    vlo, vhi = v.amin(-1), v.amax(-1)

    def params(a, b):
        # torch multiplies by 1 / 15 in 32 bits, the format divides: rounded from 64 bits it is the same
        wide = torch.stack([(b.double() - a.double()) / 15, a.double()], -1)
        return wide, torch.stack([((b - a).double() / 15).float(), a], -1)

    def codes(x, p):
        t = torch.where(p[..., 0] > 0, (x - p[..., 1]) / p[..., 0], torch.zeros_like(x))
        return torch.round(t).clamp(0, 15)

    kp, vp = params(lo, hi), params(vlo, vhi)
    return codes(K.float(), kp[1][rows[:, 0]]), kp, codes(v, vp[1].unsqueeze(2)).view(-1, d), vp


def _expanded(c, kc, kp, vcodes, vp, segs):
    rows, _ = _group_of_rows(c, segs)
    k = kp[rows].double()
    v = vp.double().repeat_interleave(32, 1)
    return kc.double() * k[..., 0] + k[..., 1], vcodes.double() * v[..., 0] + v[..., 1]


def _exact_decode(c, seed):
    K, V, segs = _cache(c, seed)
    if c["kind"] == "decode_kv4":
        kc, kp, vcodes, vp = _quantized(c, K, V, segs)
        K, V = (x.float().to(_dtype(c)) for x in _expanded(c, kc, kp[1], vcodes, vp[1], segs))
    q, kt, vt = _step_inputs(c, seed)
    L, H, d = c["L"], c["Hkv"], c["d"]
    out = torch.zeros(q.shape, dtype=torch.float64, device=DEV)
    at, t0 = 0, 0
    for r, T in enumerate(_text(c)):
        for l in range(L):
            b = segs[r * L + l]
            rows = slice(at, at + H * b)
            at += H * b
            txt = slice(t0, t0 + H * T)
            k = torch.cat([K[rows].view(H, b, d), kt[l, txt].view(H, T, d)], 1).double()
            v = torch.cat([V[rows].view(H, b, d), vt[l, txt].view(H, T, d)], 1).double()
            x = q[l, r].double().view(H, -1, d) @ k.transpose(1, 2) / math.sqrt(d)
            out[l, r] = (torch.softmax(x, -1) @ v).view(-1, d)
        t0 += H * T
    return {"out": out}
