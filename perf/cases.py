"""The work this framework is used for, as timed cases: attention of a chunk over its quantized cache, and the
quantize-append of a finished chunk, through the public binding.

Shapes, formats and value distributions are those of paper_2605_26266_b200/inputs.py (the workloads bench.py and the
tests run) plus two generic ones: a short query chunk, and heads of 64 channels at an ordinary size.  Tensors are
[batch, heads, tokens, head_dim] BF16.  Fields of a case:

  kind      "attn" (kvq_attn_corrected) or "append" (kvq_quantize_append)
  m         tokens of the chunk: query rows and current keys of an "attn" case, appended tokens of an "append" one
  cached    tokens already in the cache (the attended window)
  begin     first token of the window; a ring cache ("ring") holds `cached` tokens and wraps
  dist      "normal"; "outlier": 4 key channels per head x8; "heads": q, k scaled per head by U[0.5, 2];
            "heavy": Student-t(3) keys with 8 channels x10
  stats     log-sum-exp and cached mass are asked for beside the output
"""
import math

import torch

from paper_2605_26266_b200 import binding as kvq


def _case(name, kind, batch, heads, head_dim, bits, group, m, cached, dist="normal", correction=True, begin=0,
          ring=False, stats=False):
    return dict(name=name, kind=kind, batch=batch, heads=heads, head_dim=head_dim, bits=bits, group=group, m=m,
                cached=cached, dist=dist, correction=correction, begin=begin, ring=ring, stats=stats)


def listed():
    return [
        # the smallest problem: two heads of 64 channels, four cached chunks; launches and latency count
        _case("tiny", "attn", 1, 2, 64, 2, 64, 256, 1024),
        # the same chunk when it is finished: the smallest append
        _case("tiny_append", "append", 1, 2, 64, 2, 64, 256, 1024),
        # a diffusion frame of 1560 tokens (no multiple of any tile) over four cached ones, at either width
        _case("sweep_int4", "attn", 1, 16, 128, 4, 128, 1560, 6240, "outlier"),
        _case("sweep_int2", "attn", 1, 16, 128, 2, 128, 1560, 6240, "outlier"),
        # one layer of a video transformer: chunks of 4680 tokens, eight of them cached
        _case("dit", "attn", 1, 24, 128, 2, 64, 4680, 37440, "heads"),
        # the same at a long horizon, 32 cached chunks: the largest
        _case("long", "attn", 1, 24, 128, 2, 128, 4680, 149760),
        # a rollout of chunks of 2048 tokens: the first chunk (empty cache) and the last (15 cached)
        _case("pipeline_first", "attn", 2, 32, 128, 2, 32, 2048, 0, "heavy"),
        _case("pipeline_last", "attn", 2, 32, 128, 2, 32, 2048, 30720, "heavy"),
        # partial prefill: a short chunk over a long prefix
        _case("prefix", "attn", 1, 32, 128, 2, 128, 256, 65536, "outlier"),
        # a handful of new tokens over a prefix, as when a reply is decoded in small steps
        _case("short", "attn", 1, 32, 128, 4, 128, 16, 16384, "outlier"),
        # heads of 64 channels at an ordinary size, sliding window in a ring cache that wraps, with the statistics
        _case("head64", "attn", 1, 16, 64, 4, 32, 1560, 6144, "outlier", begin=3136, ring=True, stats=True),
        # the finished chunk of the video transformer goes into the cache
        _case("append", "append", 1, 24, 128, 2, 64, 4680, 37440, "heads"),
    ]


def draw(rng):
    def log_int(lo, hi):
        return max(lo, min(hi, round(math.exp(rng.uniform(math.log(lo), math.log(hi + 1))))))

    kind = "append" if rng.random() < 0.25 else "attn"
    head_dim = rng.choice((128, 128, 128, 64))
    batch, heads = rng.choice((1, 1, 2)), rng.choice((2, 8, 16, 24, 32))
    m = log_int(16, 4680)
    ring = rng.random() < 0.25
    cached = rng.choice((0, log_int(64, 65536), log_int(64, 65536), log_int(64, 65536)))
    if kind == "append":
        m, cached = log_int(64, 4680), min(cached, 8192)
    if ring:
        cached = max(128, cached // 128 * 128)
    begin = 16 * rng.randrange(0, 64)
    # the cost of a drawn attention stays well below the largest listed one
    limit = 1.0e12 if head_dim == 128 else 1.0e11
    while kind == "attn" and 4.0 * batch * heads * m * (cached + m) * head_dim > limit:
        if cached > 4 * m and not ring:
            cached //= 2
        elif heads > 2:
            heads //= 2
        else:
            m = m // 2 + 1
    return dict(kind=kind, batch=batch, heads=heads, head_dim=head_dim, bits=rng.choice((2, 2, 4)),
                group=rng.choice([g for g in (32, 64, 128) if g <= head_dim]), m=m, cached=cached,
                dist=rng.choice(("normal", "outlier", "heads")), correction=rng.random() < 0.75, begin=begin, ring=ring,
                stats=rng.random() < 0.5)


# ---- inputs ------------------------------------------------------------------------------------

_CHUNK = 4680      # tokens of the cached past that are drawn and appended at a time


def _generator(seed, tag):
    return torch.Generator(device="cuda").manual_seed((seed * 1000003 + tag) & 0x7FFFFFFF)


def _kv(case, seed, tag, tokens):
    """Keys and values of one run of tokens."""
    b, h, d = case["batch"], case["heads"], case["head_dim"]
    g = _generator(seed, 7 + tag)
    k = torch.randn(b, h, tokens, d, device="cuda", generator=g)
    if case["dist"] == "heavy":
        chi2 = torch.zeros_like(k)
        for _ in range(3):
            chi2 += torch.randn(b, h, tokens, d, device="cuda", generator=g).square_()
        k /= (chi2 / 3.0).sqrt_()
    a = _generator(seed, 1)
    if case["dist"] in ("outlier", "heavy"):
        n, scale = (4, 8.0) if case["dist"] == "outlier" else (8, 10.0)
        idx = torch.rand(h, d, device="cuda", generator=a).argsort(-1)[:, :n]
        k *= torch.ones(h, d, device="cuda").scatter_(1, idx, scale)[None, :, None, :]
    if case["dist"] == "heads":
        k *= (0.5 + 1.5 * torch.rand(h, device="cuda", generator=a))[None, :, None, None]
    v = torch.randn(b, h, tokens, d, device="cuda", generator=g)
    return k.to(torch.bfloat16), v.to(torch.bfloat16)


def _query(case, seed):
    b, h, d = case["batch"], case["heads"], case["head_dim"]
    g = _generator(seed, 2)
    q = torch.randn(b, h, case["m"], d, device="cuda", generator=g)
    if case["dist"] == "heads":
        q *= (0.5 + 1.5 * torch.rand(h, device="cuda", generator=g))[None, :, None, None]
    return q.to(torch.bfloat16)


def _past(case):
    """The cached window as runs of (tag, offset in the window, tokens)."""
    return [(i, t, min(_CHUNK, case["cached"] - t)) for i, t in enumerate(range(0, case["cached"], _CHUNK))]


def _capacity(case):
    if case["ring"]:
        return case["cached"]
    return (case["begin"] + case["cached"] + case["m"] + 127) // 128 * 128


def _make_cache(case):
    if case["kind"] == "append" and case["ring"]:
        cap = (max(case["cached"], case["m"]) + 127) // 128 * 128
    else:
        cap = _capacity(case)
    return kvq.Cache(case["batch"], case["heads"], case["head_dim"], case["bits"], case["group"], cap, ring=case["ring"])


def prepare(case, seed):
    cache = _make_cache(case)
    k, v = _kv(case, seed, 1000, case["m"])
    state = dict(case=case, cache=cache, k=k, v=v)
    if case["kind"] == "append":
        return state
    for tag, at, n in _past(case):
        pk, pv = _kv(case, seed, tag, n)
        kvq.kvq_quantize_append(cache, pk, pv, cache_len=case["begin"] + at)
    state["q"] = _query(case, seed)
    state["scale"] = 1.0 / math.sqrt(case["head_dim"])
    state["flags"] = kvq.KVQ_CORRECTION_ON if case["correction"] else kvq.KVQ_CORRECTION_OFF
    state["out"] = torch.empty_like(state["q"])
    rows = state["q"].shape[:3]
    state["lse"] = torch.empty(rows, dtype=torch.float32, device="cuda") if case["stats"] else None
    state["mass"] = torch.empty(rows, dtype=torch.float32, device="cuda") if case["stats"] else None
    return state


def run(state):
    case = state["case"]
    if case["kind"] == "append":
        kvq.kvq_quantize_append(state["cache"], state["k"], state["v"], cache_len=case["begin"] + case["cached"])
        return state["cache"].buffers
    out = kvq.kvq_attn_corrected(state["cache"], state["q"], state["k"], state["v"], state["scale"], state["flags"],
                                 cache_begin=case["begin"], cache_len=case["cached"], out=state["out"],
                                 lse=state["lse"], cached_mass=state["mass"])
    return [out, state["lse"], state["mass"]] if case["stats"] else [out]


def work(case):
    d, rows = case["head_dim"], case["batch"] * case["heads"] * case["m"]
    token = 2 * (d * case["bits"] // 8 + 3 * (d // case["group"]))          # packed keys and values of one token
    if case["kind"] == "append":
        return {"bytes": rows * (4 * d + token), "flops": 0}
    bytes_ = case["batch"] * case["heads"] * case["cached"] * token + rows * (8 * d + (8 if case["stats"] else 0))
    return {"bytes": bytes_, "flops": 4 * rows * (case["cached"] + case["m"]) * d}


def tolerance(case):
    if case["kind"] == "append":
        return "exact"                                  # stored codes, scales and zero-points are whole numbers
    # weights and outputs are rounded to BF16, rotated queries to FP16: 1.3e-3 to 2.9e-3 from 64 bits over these ranges
    return {"rel": 1e-2}


# ---- the same in 64 bits, without the framework -------------------------------------------------

def _f32(x):
    return x.to(torch.float32).to(torch.float64)


def _rotate(x, rounded):
    """(1/sqrt d) H x in 64 bits; `rounded`: with a 32-bit rounding after every operation, as the cache format has it."""
    d, h = x.shape[-1], 1
    y, shape = x.to(torch.float64), x.shape
    while h < d:
        y = y.reshape(*shape[:-1], d // (2 * h), 2, h)
        a, b = y[..., 0, :], y[..., 1, :]
        y = torch.stack((a + b, a - b), dim=-2).reshape(shape)
        y = _f32(y) if rounded else y
        h *= 2
    return _f32(y * float(torch.tensor(1.0 / math.sqrt(d), dtype=torch.float32))) if rounded else y / math.sqrt(d)


def _quantize(y, bits, group):
    """Codes, step bytes and zero-points of Eq. (1), each operation rounded to 32 bits."""
    levels = float(2 ** bits - 1)
    yg = y.to(torch.float64).unflatten(-1, (-1, group))
    mn, mx = yg.amin(-1), yg.amax(-1)
    step = _f32(_f32(mx - mn) / levels).clamp(max=448.0)
    byte = step.to(torch.float32).to(torch.float8_e4m3fn).view(torch.uint8).clamp(min=1)
    ds = byte.view(torch.float8_e4m3fn).to(torch.float64)
    zero = (0.0 - torch.round(_f32(mn / ds))).to(torch.float32).to(torch.bfloat16)
    code = torch.round(_f32(yg / ds[..., None])) + zero.to(torch.float64)[..., None]
    return code.clamp(0.0, levels).to(torch.uint8).flatten(-2), byte, zero


def _pack(code, bits):
    c = code.unflatten(-1, (-1, 8 // bits))
    out = torch.zeros(c.shape[:-1], dtype=torch.uint8, device=code.device)
    for i in range(8 // bits):
        out |= c[..., i] << (bits * i)
    return out


def _dequant(code, byte, zero, group):
    ds, zs = byte.view(torch.float8_e4m3fn).to(torch.float64), zero.to(torch.float64)
    return ((code.to(torch.float64).unflatten(-1, (-1, group)) - zs[..., None]) * ds[..., None]).flatten(-2)


def _exact_append(case, seed):
    cache = _make_cache(case)
    cap = cache.desc.capacity
    k, v = _kv(case, seed, 1000, case["m"])
    slots = (case["begin"] + case["cached"] + torch.arange(case["m"], device="cuda")) % cap
    parts = {}
    for name, x in (("k", _rotate(k, True)), ("v", v)):
        code, byte, zero = _quantize(x, case["bits"], case["group"])
        parts[name] = (_pack(code, case["bits"]), byte, zero.view(torch.uint8))
    outs = []
    for part in range(3):
        for name in ("k", "v"):
            t = parts[name][part]
            full = torch.zeros(t.shape[0], t.shape[1], cap, t.shape[3], dtype=torch.uint8, device="cuda")
            full[:, :, slots] = t
            outs.append(full.flatten())
    return outs


def exact(case, seed):
    if case["kind"] == "append":
        return _exact_append(case, seed)
    bits, group, d = case["bits"], case["group"], case["head_dim"]
    sigma = 1.0 / math.sqrt(d)
    q, (kc, vc) = _query(case, seed), _kv(case, seed, 1000, case["m"])
    past = []
    for tag, _, n in _past(case):
        k, v = _kv(case, seed, tag, n)
        pk = [_quantize(_rotate(k[:, h:h + 1], True), bits, group) for h in range(case["heads"])]
        past.append(([torch.cat(t, 1) for t in zip(*pk)], _quantize(v, bits, group)))
    out = torch.empty(q.shape, dtype=torch.float64, device="cuda")
    lse = torch.empty(q.shape[:3], dtype=torch.float64, device="cuda")
    mass = torch.zeros_like(lse)
    for b in range(case["batch"]):
        for h in range(case["heads"]):
            qh = q[b, h].to(torch.float64)
            keys, vals = kc[b, h].to(torch.float64), vc[b, h].to(torch.float64)
            if past:
                hat_k = torch.cat([_dequant(*[t[b, h] for t in pk], group) for pk, _ in past])
                hat_v = torch.cat([_dequant(*[t[b, h] for t in pv], group) for _, pv in past])
                step2 = torch.cat([pk[1][b, h].view(torch.float8_e4m3fn).to(torch.float64) for pk, _ in past]).square()
                qr = _rotate(qh, False)
                nu = qr.square().unflatten(-1, (-1, group)).sum(-1)
                vals = torch.cat((hat_v, vals))
            n = case["cached"]
            rows = max(1, min(case["m"], (1 << 28) // (n + case["m"])))
            for r in range(0, case["m"], rows):
                s = sigma * (qh[r:r + rows] @ keys.T)
                if past:
                    sc = sigma * (qr[r:r + rows] @ hat_k.T)
                    if case["correction"]:
                        sc -= (sigma * sigma / 24.0) * (nu[r:r + rows] @ step2.T)
                    s = torch.cat((sc, s), 1)
                top = s.amax(1, keepdim=True)
                s.sub_(top).exp_()
                total = s.sum(1, keepdim=True)
                out[b, h, r:r + rows] = (s @ vals) / total
                lse[b, h, r:r + rows] = (top + total.log())[:, 0]
                mass[b, h, r:r + rows] = s[:, :n].sum(1) / total[:, 0]
    return [out, lse, mass] if case["stats"] else [out]
