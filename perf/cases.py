"""The framework's work, as cases that can be timed and compared.

One case is one call (or the pair of calls that belong together) a server
makes on the paged 4-bit KV cache, through the package's public entry points.
The sizes are those of the benchmark's workloads and of the paper's serving
cadence; ``draw`` spreads more cases over the same ranges: both page formats,
both head dimensions, the three page sizes, ragged contexts.

The pools are built here with plain torch (quantized rows of N(0, 1) values,
four K channels per head scaled by 20 in the affine pools, random physical
page order), so that ``exact`` can work in 64 bits from the same bytes without
the package.
"""
import functools
import math

import numpy as np
import torch

import paper_2609_17475_gb300 as jf

DEV = "cuda"
AFFINE, TQ4 = "affine", "tq4"


# ---------------------------------------------------------------------------
# cases
# ---------------------------------------------------------------------------
def _case(name, kind, fmt=AFFINE, heads=(24, 4, 256), page=256, ctx=(), chunk=(), q_len=1,
          splits=0, pages=0):
    """ctx: positions per request (decode kinds), or positions before the chunk
    (append, prefill), as text; chunk: rows per request; splits 0: the
    package's default."""
    c = dict(kind=kind, fmt=fmt, hq=heads[0], hkv=heads[1], d=heads[2], page=page,
             ctx=",".join(map(str, ctx)), chunk=",".join(map(str, chunk)), q_len=q_len,
             splits=splits, pages=pages)
    return dict(c, name=name) if name else c


def listed():
    mixed = np.random.default_rng(5).integers(1024, 65537, 32).tolist()
    return [
        # the smallest call: one short request on a small model
        _case("decode-4k", "decode", heads=(8, 2, 128), ctx=[4096]),
        # a token of the 32K + 6K conversation: append its row, then attend
        _case("step-36k", "step", ctx=[35841]),
        # a token of a full-window conversation
        _case("step-256k", "step", ctx=[262144]),
        # a token for each of 32 users of unequal history, small pages
        _case("decode-mixed-32", "decode", page=64, ctx=mixed),
        # speculative decoding: four proposed tokens verified in one pass
        _case("verify-256k-q4", "verify", ctx=[262144], q_len=4),
        # a prompt chunk's rows written into their pages
        _case("append-2048", "append", ctx=[30720], chunk=[2048]),
        # the last chunk of a 32K prompt attends its whole prefix
        _case("prefill-2048-at-30720", "prefill", ctx=[30720], chunk=[2048]),
        # the cadence beside active decoders: 64-token chunks of eight prompts
        _case("prefill-batch-8x64", "prefill", ctx=[4096 * i - 64 for i in range(1, 9)],
              chunk=[64] * 8),
        # a full-window request put aside and brought back into other pages
        _case("park-resume-256k", "pages", pages=1024),
        # the TQ4 format: a token of a full-window conversation
        _case("tq4-step-256k", "step", TQ4, ctx=[262144]),
        # ... a prompt chunk encoded
        _case("tq4-append-2048", "append", TQ4, ctx=[30720], chunk=[2048]),
        # ... and a ragged prompt chunk attending its prefix
        _case("tq4-prefill-1500-at-20001", "prefill", TQ4, ctx=[20001], chunk=[1500]),
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["decode", "decode", "step", "step", "verify", "verify", "append", "append",
                       "prefill", "prefill", "pages"])
    fmt = rng.choice([AFFINE, AFFINE, TQ4])
    heads = rng.choice([(8, 2, 128), (24, 4, 256), (24, 4, 256), (32, 8, 128), (16, 4, 256)])
    page = rng.choice([64, 128, 256])
    if kind == "pages":
        return _case(None, kind, fmt, heads, page, pages=_log_int(rng, 16, 1024))
    if kind == "append":
        n = rng.choice([1, 1, 1, 4, 16])
        return _case(None, kind, fmt, heads, page, [_log_int(rng, 1, 32000) for _ in range(n)],
                     [_log_int(rng, 16, 4096 // n) for _ in range(n)])
    if kind == "prefill":
        if rng.random() < 0.5:   # a prompt chunk
            return _case(None, kind, fmt, heads, page, [_log_int(rng, 1, 30000)],
                         [_log_int(rng, 64, 2048)])
        n = rng.randint(2, 12)   # chunks beside active decoders
        return _case(None, kind, fmt, heads, page, [_log_int(rng, 256, 32000) for _ in range(n)],
                     [rng.choice([64, 64, rng.randint(17, 256)]) for _ in range(n)])
    q_len = rng.randint(2, 4) if kind == "verify" else 1
    n = rng.choice([1, 1, 2, rng.randint(3, 24)])
    most = 262144 if n <= 2 else 32768
    return _case(None, kind, fmt, heads, page, [_log_int(rng, 512, most) for _ in range(n)],
                 q_len=q_len)


def _ints(text):
    return [int(x) for x in text.split(",")] if text else []


def _position_bytes(case):
    """Bytes of one position of one layer in a page record."""
    d, side = case["d"], (2 if case["fmt"] == TQ4 else case["d"] // 16)
    return 2 * case["hkv"] * (d // 2 + side)


def work(case):
    pos, ctx, chunk = _position_bytes(case), _ints(case["ctx"]), _ints(case["chunk"])
    hq, hkv, d = case["hq"], case["hkv"], case["d"]
    kind = case["kind"]
    if kind == "pages":   # out of the pool and back: each read once, written once
        return {"bytes": 4 * case["pages"] * case["page"] * pos, "flops": 0}
    if kind == "append":
        rows = sum(chunk)
        log_d = int(math.log2(d))
        return {"bytes": rows * (2 * hkv * d * 2 + pos + 8),
                "flops": rows * 2 * hkv * d * (log_d + 2 if case["fmt"] == TQ4 else 2)}
    if kind == "prefill":
        seen = sum(c * s + c * (c + 1) // 2 for s, c in zip(ctx, chunk))
        kept = sum(s + c for s, c in zip(ctx, chunk))
        return {"bytes": kept * pos + 2 * sum(chunk) * hq * d * 2, "flops": 4 * hq * d * seen}
    rows = len(ctx) * case["q_len"]
    new = len(ctx) * (2 * hkv * d * 2 + pos) if kind == "step" else 0
    table = sum(-(-c // case["page"]) for c in ctx) * 4
    return {"bytes": sum(ctx) * pos + 2 * rows * hq * d * 2 + table + new,
            "flops": 4 * hq * d * sum(ctx) * case["q_len"]}


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _generator(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    return g


def _normal(gen, *shape):
    return torch.randn(*shape, generator=gen, device=DEV, dtype=torch.float32).to(torch.bfloat16)


@functools.lru_cache(maxsize=None)
def _codebook(d):
    """The 16 Lloyd-Max centroids of the density (1 - x^2)^((d-3)/2), fp32."""
    x = np.arange(32768) * ((2.0 - 2e-6) / 32767) + (-1.0 + 1e-6)
    x[-1] = 1.0 - 1e-6
    w = (1.0 - x * x) ** ((d - 3) / 2)
    w /= w.sum()
    c = x[np.searchsorted(np.cumsum(w), (np.arange(16) + 0.5) / 16)]
    for _ in range(100):
        cell = np.searchsorted((c[:-1] + c[1:]) / 2, x, side="left")
        mass = np.bincount(cell, w, 16)
        new = np.where(mass > 0, np.bincount(cell, w * x, 16) / np.where(mass > 0, mass, 1), c)
        moved, c = np.abs(new - c).max(), new
        if moved < 1e-6:
            break
    return c.astype(np.float32)


@functools.lru_cache(maxsize=None)
def _signs(d):
    """The random-sign diagonals of K and V."""
    return [np.random.default_rng(s + 7919 * d).choice(np.array([-1, 1], np.int8), d)
            for s in (0, 1)]


def _hadamard(d, dtype):
    h = torch.ones(1, 1, device=DEV, dtype=dtype)
    while h.shape[0] < d:
        h = torch.cat([torch.cat([h, h], 1), torch.cat([h, -h], 1)], 0)
    return h


def _encode(case, x, which):
    """bf16 [..., d] -> (codes uint8 [..., d/2], side bytes uint8 [..., n]); which 0: K, 1: V."""
    d = case["d"]
    x = x.float()
    if case["fmt"] == AFFINE:
        g = x.unflatten(-1, (d // 64, 64))
        lo = g.amin(-1, keepdim=True) + 0.0
        scale = ((g.amax(-1, keepdim=True) - lo) / 15.0).to(torch.bfloat16)
        s = scale.float()
        code = torch.where(s > 0, torch.ceil((g - lo) / s - 0.5).clamp(0, 15), 0.0)
        code = code.flatten(-2)
        side = torch.cat([scale, lo.to(torch.bfloat16)], -1).flatten(-2).view(torch.uint8)
    else:
        sign = torch.from_numpy(_signs(d)[which]).to(DEV).float()
        c = torch.from_numpy(_codebook(d)).to(DEV)
        rho = x.double().square().sum(-1, keepdim=True).sqrt().float()
        y = (x * sign) @ _hadamard(d, torch.float32) / (math.sqrt(d) * rho.clamp_min(1e-30))
        code = torch.bucketize(y, (c[:-1] + c[1:]) * 0.5)
        side = rho.clamp_max(65504.0).to(torch.float16).view(torch.uint8)
    code = code.to(torch.uint8)
    return code[..., 0::2] | (code[..., 1::2] << 4), side


def _pool(case, gen, lens, spare=0):
    """(data uint8 [pages, page bytes], table int32 [requests, most pages]): every
    page of every request holds encoded rows; ``spare`` more pages are zero."""
    p, hkv, d = case["page"], case["hkv"], case["d"]
    need = [-(-n // p) for n in lens]
    total = sum(need)
    data = torch.zeros(total + spare, p * _position_bytes(case), dtype=torch.uint8, device=DEV)
    order = torch.randperm(total + spare, generator=gen, device=DEV)
    loud = torch.ones(hkv, d, device=DEV)
    if case["fmt"] == AFFINE:
        for h in range(hkv):
            loud[h, torch.randperm(d, generator=gen, device=DEV)[:4]] = 20.0
    step = max(1, 65536 // p)
    for a in range(0, total, step):
        n = min(step, total - a)
        parts = [[], []]
        for which in (0, 1):
            x = torch.randn(n, hkv, p, d, generator=gen, device=DEV)
            if which == 0:
                x *= loud[None, :, None, :]
            code, side = _encode(case, x.to(torch.bfloat16), which)
            parts[0].append(code.reshape(n, -1))
            parts[1].append(side.reshape(n, -1))
        data[order[a:a + n]] = torch.cat(parts[0] + parts[1], 1)
    table = torch.full((len(lens), max(need)), -1, dtype=torch.int32, device=DEV)
    at = 0
    for b, n in enumerate(need):
        table[b, :n] = order[at:at + n].to(torch.int32)
        at += n
    return data, table


def _inputs(case, seed):
    """Everything the case reads, from the seed alone."""
    gen = _generator(seed)
    ctx, chunk = _ints(case["ctx"]), _ints(case["chunk"])
    hq, hkv, d, kind = case["hq"], case["hkv"], case["d"], case["kind"]
    s = {}
    if kind == "pages":
        n = case["pages"]
        s["data"] = torch.randint(0, 256, (2 * n, case["page"] * _position_bytes(case)),
                                  generator=gen, device=DEV, dtype=torch.uint8)
        order = torch.randperm(2 * n, generator=gen, device=DEV).to(torch.int32)
        s["source"], s["target"] = order[:n].contiguous(), order[n:].contiguous()
    elif kind == "append":
        lens = [a + c for a, c in zip(ctx, chunk)]
        need = [-(-n // case["page"]) for n in lens]
        s["data"] = torch.zeros(sum(need), case["page"] * _position_bytes(case),
                                dtype=torch.uint8, device=DEV)
        order = torch.randperm(sum(need), generator=gen, device=DEV).to(torch.int32)
        s["table"] = torch.zeros(len(lens), max(need), dtype=torch.int32, device=DEV)
        at = 0
        for b, n in enumerate(need):
            s["table"][b, :n] = order[at:at + n]
            at += n
        rows = sum(chunk)
        s["k"], s["v"] = _normal(gen, rows, hkv, d), _normal(gen, rows, hkv, d)
        s["req"] = torch.cat([torch.full((c,), b, dtype=torch.int32, device=DEV)
                              for b, c in enumerate(chunk)])
        s["pos"] = torch.cat([torch.arange(a, a + c, dtype=torch.int32, device=DEV)
                              for a, c in zip(ctx, chunk)])
    elif kind == "prefill":
        s["data"], s["table"] = _pool(case, gen, [a + c for a, c in zip(ctx, chunk)])
        s["q"] = _normal(gen, sum(chunk), hq, d)
    else:
        s["data"], s["table"] = _pool(case, gen, ctx)
        shape = (len(ctx), case["q_len"], hq, d) if kind == "verify" else (len(ctx), hq, d)
        s["q"] = _normal(gen, *shape)
        s["lens"] = torch.tensor(ctx, dtype=torch.int32, device=DEV)
        if kind == "step":
            s["k"], s["v"] = _normal(gen, len(ctx), hkv, d), _normal(gen, len(ctx), hkv, d)
    return s


def prepare(case, seed):
    s = _inputs(case, seed)
    s["kind"] = kind = case["kind"]
    hq, hkv, d = case["hq"], case["hkv"], case["d"]
    ctx, chunk = _ints(case["ctx"]), _ints(case["chunk"])
    fmt, codec = jf.JF_FMT_AFFINE4_G64, None
    if case["fmt"] == TQ4:
        fmt, codec = jf.JF_FMT_TQ4, jf.Tq4Codec(d, *_signs(d), centroids=_codebook(d))
    s["pool"] = pool = jf.KVPool(s["data"], case["page"], hkv, d, format=fmt, codec=codec)
    s["scale"] = 1.0 / math.sqrt(d)
    s["err"] = torch.zeros(1, dtype=torch.int32, device=DEV)
    if "q" in s:
        s["out"] = torch.empty_like(s["q"])
    if kind == "pages":
        s["blob"] = torch.empty(case["pages"] * pool.page_bytes, dtype=torch.uint8, device=DEV)
    elif kind == "prefill" and len(ctx) == 1:
        s["start"] = ctx[0]
        s["row"] = s["table"][0]
        s["ws"] = jf.prefill_chunk_workspace(pool, ctx[0], chunk[0], hq)
    elif kind == "prefill":
        s["start"], s["chunk"] = ctx, chunk
        s["splits"] = case["splits"] or jf.default_prefill_splits(ctx, chunk, hq, hkv)
        s["ws"] = jf.prefill_batch_workspace(sum(chunk), hq, d, s["splits"], format=fmt)
    elif kind == "verify":
        n = len(ctx)
        s["splits"] = case["splits"] or jf.default_verify_splits(n, case["q_len"], hq, hkv,
                                                                 format=fmt)
        s["ws"] = jf.verify_workspace(n, case["q_len"], hq, hkv, d, s["splits"])
    elif kind in ("decode", "step"):
        s["splits"] = case["splits"] or jf.default_num_splits(len(ctx), hkv, format=fmt)
        s["ws"] = jf.decode_workspace(len(ctx), hq, hkv, d, s["splits"])
    return s


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------
def run(s):
    kind, pool = s["kind"], s["pool"]
    if kind == "decode":
        jf.jf_paged_decode_attn(pool, s["table"], s["lens"], s["q"], s["scale"], s["out"],
                                s["ws"], s["splits"])
    elif kind == "step":
        jf.jf_paged_decode_append_attn(pool, s["table"], s["lens"], s["k"], s["v"], s["q"],
                                       s["scale"], s["out"], s["ws"], s["splits"])
        return {"out": s["out"], "pool": pool.data}
    elif kind == "verify":
        jf.jf_paged_verify_attn(pool, s["table"], s["lens"], s["q"], s["scale"], s["out"],
                                s["ws"], s["splits"])
    elif kind == "append":
        jf.jf_kv_quantize_append(pool, s["table"], s["req"], s["pos"], s["k"], s["v"], s["err"])
        return {"pool": pool.data}
    elif kind == "prefill" and "row" in s:
        jf.jf_prefill_chunk_attn(pool, s["row"], s["q"], s["start"], s["scale"], True, s["out"],
                                 s["ws"])
    elif kind == "prefill":
        jf.jf_prefill_batch_attn(pool, s["table"], s["start"], s["chunk"], s["q"], s["scale"],
                                 True, s["out"], s["ws"], num_splits=s["splits"])
    else:
        pages = s["source"].numel()
        jf.jf_kv_checkpoint(pool, s["source"], pages, s["blob"], s["err"])
        jf.jf_kv_restore(pool, s["target"], pages, s["blob"], s["err"])
        return {"blob": s["blob"], "pool": pool.data}
    return {"out": s["out"]}


# ---------------------------------------------------------------------------
# the same in 64 bits
# ---------------------------------------------------------------------------
def _decode_rows(case, code, side):
    """codes [n, d/2], side [n, bytes] -> fp64 [n, d]; TQ4 rows stay in the rotated basis."""
    z = torch.stack([code & 15, code >> 4], -1).flatten(-2)
    if case["fmt"] == TQ4:
        c = torch.from_numpy(_codebook(case["d"])).to(DEV).double()
        return c[z.long()] * side.contiguous().view(torch.float16).double()
    sb = side.contiguous().view(torch.bfloat16).double().unflatten(-1, (-1, 2))
    x = z.double().unflatten(-1, (-1, 64))
    return (x * sb[..., :1] + sb[..., 1:]).flatten(-2)


def _history(case, s, b, h, n):
    """K and V of request b, KV head h, positions < n, as the bytes say."""
    p, hkv, d = case["page"], case["hkv"], case["d"]
    rec = s["data"][s["table"][b, :-(-n // p)].long()]
    codes, side = hkv * p * d // 2, rec.shape[1] // 2 - hkv * p * d // 2
    got = []
    for which in (0, 1):
        c = rec[:, which * codes:(which + 1) * codes].reshape(-1, hkv, p, d // 2)
        t = rec[:, 2 * codes + which * side:2 * codes + (which + 1) * side]
        t = t.reshape(len(rec), hkv, p, -1)
        got.append(_decode_rows(case, c[:, h].reshape(-1, d // 2)[:n],
                                t[:, h].reshape(n + (-n) % p, -1)[:n]))
    return got


def _attend(case, q, k, v, seen):
    """softmax(q k^T / sqrt(d)) v in fp64; row i sees the first seen[i] positions."""
    d = case["d"]
    q = q.double()
    if case["fmt"] == TQ4:
        had = _hadamard(d, torch.float64)
        sk, sv = (torch.from_numpy(x).to(DEV).double() for x in _signs(d))
        q = (q * sk) @ had / math.sqrt(d)
    out = torch.empty_like(q)
    for a in range(0, len(q), 2048):
        w = q[a:a + 2048] @ k.T / math.sqrt(d)
        hidden = torch.arange(len(k), device=DEV)[None, :] >= seen[a:a + 2048, None]
        w.masked_fill_(hidden, -math.inf)
        out[a:a + 2048] = torch.softmax(w, -1) @ v
    return (out @ had / math.sqrt(d)) * sv if case["fmt"] == TQ4 else out


def exact(case, seed):
    kind = case["kind"]
    if kind in ("pages", "append"):
        return None   # bytes
    s = _inputs(case, seed)
    ctx, chunk = _ints(case["ctx"]), _ints(case["chunk"])
    hq, hkv, d = case["hq"], case["hkv"], case["d"]
    grp = hq // hkv
    out = torch.zeros(s["q"].shape, dtype=torch.float64, device=DEV)
    at = 0
    for b, n in enumerate(ctx):
        if kind == "prefill":
            rows, first, n = chunk[b], n, n + chunk[b]
            q, o = s["q"][at:at + rows], out[at:at + rows]
            at += rows
        else:
            rows, first = case["q_len"], n - case["q_len"]
            q, o = (t[b].reshape(rows, hq, d) for t in (s["q"], out))
        seen = (torch.arange(rows, device=DEV) + first + 1).repeat_interleave(grp)
        for h in range(hkv):
            k, v = _history(case, s, b, h, n)
            if kind == "step":   # the new row replaces the last position
                for which, (dst, x) in enumerate(((k, s["k"]), (v, s["v"]))):
                    dst[n - 1] = _decode_rows(case, *_encode(case, x[b, h][None], which))[0]
            o[:, h * grp:(h + 1) * grp] = _attend(
                case, q[:, h * grp:(h + 1) * grp].reshape(-1, d), k, v, seen).view(rows, grp, d)
    return {"out": out, "pool": None} if kind == "step" else {"out": out}
