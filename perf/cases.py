"""The work that programs have this library do, one call sequence per case.

Shapes are those of the repository's workloads: 14B-shaped layers (40 query /
8 KV heads of 128), 7B-shaped layers (28 / 4), the head_dim-64 toy layer
(8 / 2) and MLA layers (16 heads of 128, latent 512 + positional key 64).
Keys and values are N(0, 1) with a lognormal(0, 0.5) scale per (head, channel),
latent coordinate k is N(0, 1/(k+1)), queries are N(0, 1).  Pre-fill chunks have
keys and values N(0, 1) and queries N(0, 0.75^2): a row's largest score over the
whole context then lies less than 8 (base 2) above that of its first 64 positions.

Five kinds of case:

* ``step``     one decode step of a layer: append the new token, attend with
               the step's query, and (so that the same step can be repeated)
               roll the token back as a rejected speculative token is.
               Per-channel keys cannot be rolled back and kept lists are fixed
               per step: those attend only.
* ``model``    the same step over every layer of a mixed plan.
* ``ingest``   a prompt's keys and values enter an empty cache (they were
               computed elsewhere, or all at once) and the first token attends.
* ``prefill``  a chunk is appended and its queries attend causally over the
               cache; ``chunk == ctx`` is a whole prompt from an empty cache.
* ``evict``    the window-vote evictor picks the positions that stay.

``ragged`` sequences have between half of and all of ``ctx`` positions.
"""
import math
import random

import torch

from paper_2609_37988_gb300.cache import Cache, Layer
from paper_2609_37988_gb300.workloads import config

# (query heads, KV heads, head_dim); MLA: 16 heads of 128 over latent 512 + 64
MODELS = {"14b": (40, 8, 128), "7b": (28, 4, 128), "toy": (8, 2, 64), "mla": (16, 1, 128)}
LATENT, ROPE = 512, 64

# name -> (bits, scheme, group, key axis)
GQA_FORMATS = {
    "bf16": (16, "grouped", 64, "token"),
    "int8": (8, "grouped", 64, "token"),
    "int4": (4, "grouped", 32, "token"),
    "int8c": (8, "grouped", 64, "channel"),
    "int4c": (4, "grouped", 32, "channel"),
    "sym8": (8, "symmetric", 64, "token"),
    "sym4": (4, "symmetric", 64, "token"),
    "sym2": (2, "symmetric", 64, "token"),
}
MLA_FORMATS = {
    "bf16": (16, "grouped"),
    "int8": (8, "grouped"),
    "int4": (4, "grouped"),
    "sym8": (8, "symmetric"),
    "sym4": (4, "symmetric"),
    "sym2": (2, "symmetric"),
}


def listed():
    return [
        # the smallest call: one fp32 token of a small layer, all launch latency
        _case("step", "toy", "int8", 1, 512, name="step_toy_int8", dtype="f32"),
        # one whole decode step of the mixed 48-layer plan, the flagship load
        dict(name="model_14b", kind="model", model="14b", batch=32, ctx=8192, dtype="bf16"),
        # a single user with a long, odd-sized context: few units, many splits
        _case("step", "14b", "int8", 1, 32769, name="step_14b_int8_b1"),
        # KIVI-style keys at the 7B shape, sequences of different lengths
        _case("step", "7b", "int4c", 16, 8192, name="step_7b_int4c_ragged", ragged=True),
        # the symmetric quantiser on an odd batch of ragged sequences
        _case("step", "14b", "sym4", 13, 5003, name="step_14b_sym4_ragged", ragged=True),
        # eviction composed with compression: a step over 1/8 of a long context
        _case("step", "14b", "int4", 4, 131072, name="step_14b_int4_kept", keep=16384),
        # a step of a full-width MLA layer at serving batch
        _case("step", "mla", "bf16", 64, 4096, name="step_mla_d512", width=512),
        # a step of a truncated and quantised MLA layer, ragged
        _case("step", "mla", "sym8", 24, 3001, name="step_mla_d128_sym8_ragged", width=128, ragged=True),
        # prompts of a batch enter an empty cache
        _case("ingest", "14b", "int4", 32, 2048, name="ingest_14b_int4"),
        # chunked pre-fill over a compressed GQA cache
        _case("prefill", "14b", "int4", 4, 8192, name="prefill_14b_int4", chunk=2048),
        # chunked pre-fill over a full-width MLA latent cache
        _case("prefill", "mla", "bf16", 4, 4096, name="prefill_mla_d512", width=512, chunk=1024),
        # eviction of a long context down to 1/8
        _case("evict", "14b", "int4", 4, 131072, name="evict_14b_int4", window=32, keep=16384),
    ]


def _case(kind, model, fmt, batch, ctx, *, name=None, dtype="bf16", width=0, keep=0, chunk=0, window=0, ragged=False):
    c = dict(kind=kind, model=model, format=fmt, batch=batch, ctx=ctx, dtype=dtype, width=width, keep=keep,
             chunk=chunk, window=window, ragged=ragged)
    if name is not None:
        c["name"] = name
    return c


def _log(rng, lo, hi):
    """A whole number spread over the logarithm of [lo, hi]."""
    return max(lo, min(hi, round(math.exp(rng.uniform(math.log(lo), math.log(max(lo, hi)))))))


def draw(rng):
    kind = rng.choice(["step", "step", "kept", "mla", "mla", "ingest", "prefill", "prefill_mla", "evict"])
    gqa = rng.choice(["14b", "7b"])
    dtype = rng.choice(["bf16", "bf16", "bf16", "f32"])
    width = rng.choice([512, 256, 128, 64])
    mla_fmt = rng.choice(["bf16", "bf16"] + list(MLA_FORMATS))
    if kind == "step":
        if rng.random() < 0.15:
            return _case("step", "toy", rng.choice(["bf16", "int8", "int4"]), _log(rng, 1, 32), _log(rng, 128, 8192),
                         dtype=dtype, ragged=rng.random() < 0.5)
        batch = _log(rng, 1, 64)
        return _case("step", gqa, rng.choice(list(GQA_FORMATS)), batch, _log(rng, 128, min(131072, 262144 // batch)),
                     dtype=dtype, ragged=rng.random() < 0.5)
    if kind == "kept":
        batch = _log(rng, 1, 16)
        ctx = _log(rng, 2048, min(131072, 524288 // batch))
        return _case("step", gqa, rng.choice(["bf16", "int8", "int4", "sym8", "sym4", "sym2"]), batch, ctx,
                     keep=max(64, ctx // rng.choice([2, 4, 8, 16])), dtype=dtype)
    if kind == "mla":
        batch = _log(rng, 1, 64)
        return _case("step", "mla", mla_fmt, batch, _log(rng, 128, min(32768, 262144 // batch)), width=width,
                     ragged=rng.random() < 0.5)
    if kind == "ingest":
        model = rng.choice([gqa, gqa, gqa, "mla"])
        batch = _log(rng, 1, 32)
        ctx = _log(rng, 65, min(32768, 65536 // batch))
        if model == "mla":
            return _case("ingest", "mla", mla_fmt, batch, ctx, width=width)
        return _case("ingest", gqa, rng.choice(list(GQA_FORMATS)), batch, ctx, dtype=dtype)
    if kind == "prefill":
        batch = _log(rng, 1, 8)
        ctx = _log(rng, 256, 32768 // batch)
        chunk = min(ctx - 1, _log(rng, 16, 2048))
        fmt = rng.choice(list(GQA_FORMATS))
        if fmt.endswith("c"):  # whole prompts
            ctx = chunk = min(ctx, 4096)
        return _case("prefill", gqa, fmt, batch, ctx, chunk=chunk, dtype=dtype)
    if kind == "prefill_mla":
        batch = _log(rng, 1, 8)
        ctx = _log(rng, 256, 16384 // batch)
        return _case("prefill", "mla", mla_fmt, batch, ctx, chunk=min(ctx - 1, _log(rng, 16, 1024)), width=width)
    batch = _log(rng, 1, 8)
    ctx = _log(rng, 1024, min(131072, 524288 // batch))
    window = rng.randint(8, 64)
    return _case("evict", gqa, rng.choice(["bf16", "int8", "int4", "sym8", "sym4", "sym2"]), batch, ctx,
                 window=window, keep=max(window + 1, ctx // rng.choice([2, 4, 8])))


# -- inputs --------------------------------------------------------------------

def _lens(case):
    """Positions of each sequence, the step's new token among them."""
    B, T = case["batch"], case["ctx"]
    if not case.get("ragged"):
        return [T] * B
    rng = random.Random(B * 1000003 + T)
    lens = [rng.randint(T - T // 2, T) for _ in range(B)]
    lens[rng.randrange(B)] = T
    return lens


def _gen(seed, layer, what):
    g = torch.Generator(device="cuda")
    g.manual_seed((seed * 1000003 + layer * 101 + what) % (1 << 62))
    return g


def _randn(shape, seed, layer, what, dtype):
    return torch.randn(shape, generator=_gen(seed, layer, what), device="cuda", dtype=dtype)


def _dtype(case):
    return torch.float32 if case["dtype"] == "f32" else torch.bfloat16


def _kv(case, seed, layer=0):
    """What is written: keys and values [B, T, H_kv, D], or for MLA the latent
    [B, T, 512] and the positional key [B, T, 64]."""
    B, T = case["batch"], case["ctx"]
    if case["model"] == "mla":
        decay = torch.arange(1, LATENT + 1, device="cuda", dtype=torch.float32).rsqrt().to(torch.bfloat16)
        return (_randn((B, T, LATENT), seed, layer, 0, torch.bfloat16).mul_(decay),
                _randn((B, T, ROPE), seed, layer, 1, torch.bfloat16))
    _, H, D = MODELS[case["model"]]
    dt = _dtype(case)
    if case["kind"] == "prefill":
        return _randn((B, T, H, D), seed, layer, 0, dt), _randn((B, T, H, D), seed, layer, 1, dt)
    scale = torch.exp(0.5 * _randn((2, H, D), seed, layer, 2, torch.float32)).to(dt)
    return (_randn((B, T, H, D), seed, layer, 0, dt).mul_(scale[0]),
            _randn((B, T, H, D), seed, layer, 1, dt).mul_(scale[1]))


def _queries(case, seed, rows=0, layer=0):
    """[B, H, D] of a step, or [B, rows, H, D] of a chunk or window; MLA: the
    content and the positional part."""
    Hq, _, D = MODELS[case["model"]]
    lead = (case["batch"], rows) if rows else (case["batch"],)
    if case["model"] == "mla":
        return (_randn(lead + (Hq, D), seed, layer, 3, torch.bfloat16),
                _randn(lead + (Hq, ROPE), seed, layer, 4, torch.bfloat16))
    q = _randn(lead + (Hq, D), seed, layer, 3, _dtype(case))
    return (q.mul_(0.75) if case["kind"] == "prefill" else q,)


def _weights(seed, layer=0):
    H, _, D = MODELS["mla"]
    return tuple(_randn((H, D, LATENT), seed, layer, w, torch.bfloat16).mul_(LATENT ** -0.5) for w in (5, 6))


def _kept(case, seed):
    """Sorted uniform samples of the positions that stay, [B, keep]."""
    B, T, n = case["batch"], case["ctx"], case["keep"]
    order = torch.rand((B, T), generator=_gen(seed, 0, 7), device="cuda").argsort(dim=1)[:, :n]
    return order.sort(dim=1).values.to(torch.int32).contiguous(), torch.full((B,), n, dtype=torch.int32, device="cuda")


def _sigma(case):
    D = MODELS[case["model"]][2]
    return 1.0 / math.sqrt(D + ROPE if case["model"] == "mla" else D)


def _layer(case):
    if case["model"] == "mla":
        bits, scheme = MLA_FORMATS[case["format"]]
        return Layer(bits=bits, scheme=scheme, width=case["width"])
    bits, scheme, group, axis = GQA_FORMATS[case["format"]]
    return Layer(bits=bits, group=group, key_axis=axis, scheme=scheme, evict_capacity=case["keep"])


def _cache(case, layers):
    Hq, H, D = MODELS[case["model"]]
    more = dict(kind="mla", latent_dim=LATENT, rope_dim=ROPE) if case["model"] == "mla" else {}
    c = Cache(n_layers=len(layers), n_q_heads=Hq, n_kv_heads=H, head_dim=D, max_batch=case["batch"],
              max_ctx=case["ctx"], layers=layers, **more)
    for a in c.arenas:
        if a is not None:
            a.zero_()
    c.reset()
    return c


def _model_layers():
    """The mixed 14B plan of the benchmark: 12 bf16 and 20 int4 anchors, 16 inheritors."""
    return [Layer(**a) for a in config(3).layers]


def _fill(case, cache, kv, layer=0):
    """Write every position but those that ``run`` appends."""
    k, v = kv
    B, T = case["batch"], case["ctx"]
    new = _appended(case)
    if case.get("ragged"):
        n = torch.tensor([l - new for l in _lens(case)], dtype=torch.int32, device="cuda")
        cache.append(layer, k[:, :T - new].contiguous(), v[:, :T - new].contiguous(), n)
    else:
        cache.append(layer, k[:, :T - new].contiguous(), v[:, :T - new].contiguous())


def _appended(case):
    """Positions per sequence that a pass appends before it attends and rolls back after."""
    if case["kind"] == "model":
        return 1
    if case["kind"] == "step":
        return 0 if case["keep"] or case["format"].endswith("c") else 1
    return case["chunk"] if case["kind"] == "prefill" and case["chunk"] < case["ctx"] else 0


def _new_rows(case, kv):
    """The rows that a pass appends: each sequence's last ones."""
    n = _appended(case)
    if not n:
        return None
    lens = _lens(case)
    if case.get("ragged"):
        at = torch.tensor(lens, device="cuda") - 1
        b = torch.arange(case["batch"], device="cuda")
        return tuple(x[b, at].unsqueeze(1).contiguous() for x in kv)
    return tuple(x[:, -n:].contiguous() for x in kv)


def prepare(case, seed):
    s = {"kind": case["kind"], "scale": _sigma(case), "mla": case["model"] == "mla"}
    if case["kind"] == "model":
        layers = _model_layers()
        s["cache"] = c = _cache(case, layers)
        s["new"], s["q"] = {}, [_queries(case, seed, layer=l)[0] for l in range(len(layers))]
        for l, a in enumerate(layers):
            if not a.inherit:
                kv = _kv(case, seed, l)
                _fill(case, c, kv, l)
                s["new"][l] = _new_rows(case, kv)
        return s
    s["cache"] = c = _cache(case, [_layer(case)])
    kv = _kv(case, seed)
    s["q"] = _queries(case, seed, rows=case["chunk"] or case["window"])
    if s["mla"]:
        s["w"] = _weights(seed)
    s["keep"] = case["keep"]
    whole = case["kind"] == "ingest" or (case["kind"] == "prefill" and case["chunk"] == case["ctx"])
    if whole:
        s["prompt"] = kv
        return s
    _fill(case, c, kv)
    s["new"] = _new_rows(case, kv)
    if case["kind"] == "step" and case["keep"]:
        c.set_kept(0, *_kept(case, seed))
    return s


# -- one pass ------------------------------------------------------------------

def run(s):
    c, kind = s["cache"], s["kind"]
    if kind == "model":
        outs = []
        for l, q in enumerate(s["q"]):
            if l in s["new"]:
                c.append(l, *s["new"][l])
            outs.append(c.decode(l, q, s["scale"]))
        c.rewind(1)
        return outs
    if kind == "evict":
        q, = s["q"]
        votes = c.evict_window(0, q, s["scale"], s["keep"])
        idx, n, _ = c.kept_lists(0)
        T, window = c.desc.max_ctx, q.shape[1]
        # the serving program frees the positions that no head keeps marked
        stays = torch.zeros(idx.shape[:2] + (T,), dtype=torch.bool, device=idx.device)
        stays.scatter_(2, idx.long(), True)
        return {"votes": votes[..., :T - window], "n": n, "stays": stays}
    if "prompt" in s:
        c.reset()
        c.append(0, *s["prompt"])
    elif s["new"] is not None:
        c.append(0, *s["new"])
    if kind == "prefill":
        out = c.prefill_mla(0, *s["q"], *s["w"], s["scale"]) if s["mla"] else c.prefill(0, *s["q"], s["scale"])
    else:
        out = c.decode_mla(0, *s["q"], *s["w"], s["scale"]) if s["mla"] else c.decode(0, *s["q"], s["scale"])
    if "prompt" in s:
        return {"out": out, "cache": c.arenas[0]}
    if s["new"] is not None:
        c.rewind(s["new"][0].shape[1])
    return out


# -- what a pass cannot do without ------------------------------------------------

def _record_bytes(case, layer=None):
    """Stored bytes per (position, KV head), or per position of an MLA layer."""
    if case["model"] == "mla":
        bits, scheme = MLA_FORMATS[case["format"]]
        return (case["width"] + ROPE) * bits // 8 + (0 if bits == 16 else 4 if scheme == "symmetric" else 16)
    D = MODELS[case["model"]][2]
    if layer is not None:
        bits, scheme, group = layer.bits, layer.scheme, layer.group
    else:
        bits, scheme, group, _ = GQA_FORMATS[case["format"]]
    codes = 2 * D * bits // 8
    return codes if bits == 16 else codes + 4 if scheme == "symmetric" else codes + 2 * 8 * (D // group)


def work(case):
    Hq, H, D = MODELS[case["model"]]
    B, T = case["batch"], case["ctx"]
    esz = 4 if case["dtype"] == "f32" else 2
    if case["kind"] == "model":
        layers = _model_layers()
        src = None
        nbytes = flops = 0
        for a in layers:
            src = src if a.inherit else a
            nbytes += B * T * H * _record_bytes(case, src) + B * Hq * D * (esz + 4)
            nbytes += 0 if a.inherit else B * H * (2 * D * esz + _record_bytes(case, a))
            flops += 4 * D * Hq * B * T
        return {"bytes": nbytes, "flops": flops}
    mla = case["model"] == "mla"
    rec = _record_bytes(case) * H
    row_in = (LATENT + ROPE) * 2 if mla else 2 * H * D * esz
    q_row, o_row = Hq * ((D + ROPE) * 2 if mla else D * esz), Hq * D * 4
    w_bytes = 2 * Hq * D * case["width"] * 2 if mla else 0
    lens = _lens(case)
    if case["kind"] == "evict":
        n, keep = case["window"], case["keep"]
        pairs = B * Hq * sum(T - n + i + 1 for i in range(n))
        # the key half of every record is read; votes and lists are written
        return {"bytes": B * T * rec // 2 + B * n * q_row + 4 * B * H * (T + keep), "flops": 2 * D * pairs}
    n_new = T if case["kind"] == "ingest" or case["chunk"] == T else _appended(case)
    nbytes = B * n_new * (row_in + rec) + w_bytes
    if case["kind"] == "prefill":
        n = case["chunk"]
        pairs = B * Hq * sum(T - n + i + 1 for i in range(n))
        nbytes += B * T * rec + B * n * (q_row + o_row)
        if mla:  # absorbed, or with each head's keys and values formed once: the lesser
            d = case["width"]
            absorbed = pairs * 2 * (2 * d + ROPE) + B * n * Hq * 4 * D * d
            formed = pairs * 2 * (2 * D + ROPE) + B * T * Hq * 4 * D * d
            return {"bytes": nbytes, "flops": min(absorbed, formed)}
        return {"bytes": nbytes, "flops": 4 * D * pairs}
    read = sum(min(l, case["keep"]) if case["keep"] else l for l in lens)
    nbytes += read * rec + B * (q_row + o_row)
    flops = Hq * (read * 2 * (2 * case["width"] + ROPE) + B * 4 * D * case["width"] if mla else read * 4 * D)
    return {"bytes": nbytes, "flops": flops}


def tolerance(case):
    """Operands are held to 16 bits or more (bf16 or f16 halves), sums and softmax
    in 32 bits; each bound is about four times the error seen against 64 bits.
    Stored codes and scales are whole bytes and stay the same."""
    if case["kind"] == "evict":
        # a position whose vote ties with the cut's to rounding may change places
        return {"rel": 1e-5, "max": 1e-3, "differ": 1e-3}
    if case["model"] == "mla" or case.get("format") == "bf16":
        return {"rel": 5e-5, "max": 1e-3}
    if case["kind"] == "prefill":
        return {"rel": 1e-4, "max": 2e-3}
    # codes of one sign average to several times the values they stand for, so
    # sums of thousands of them lose two or three digits: 2e-4 seen
    return {"rel": 8e-4, "max": 8e-3}


# -- the same in 64 bits ---------------------------------------------------------

def _grouped(x, bits, dim_group):
    """Dequantised values of groups along the last axis; codes by binary32 steps."""
    g = x.float().unflatten(-1, (-1, dim_group))
    lo, hi = g.amin(-1, keepdim=True), g.amax(-1, keepdim=True)
    lev = torch.full_like(lo, 2 ** bits - 1)  # a tensor: division by a number multiplies by its reciprocal
    s = (hi - lo) / lev
    code = ((g - lo) / torch.where(s == 0, torch.ones_like(s), s)).round().clamp(0, 2 ** bits - 1)
    return torch.where(s == 0, lo.double(), code.double() * s.double() + lo.double()).flatten(-2)


def _symmetric(x, bits):
    x = x.float()
    q = float(2 ** (bits - 1) - 1)
    hi = x.abs().amax(-1, keepdim=True)
    s = (hi / torch.full_like(hi, q)).bfloat16().float()
    code = (x / torch.where(s == 0, torch.ones_like(s), s)).round().clamp(-q, q)
    return torch.where(s == 0, torch.zeros_like(code), code).double() * s.double()


def _stored(x, bits, scheme, group):
    if bits == 16:
        return x.bfloat16().double()
    return _symmetric(x, bits) if scheme == "symmetric" else _grouped(x, bits, group)


def _stored_kv(k, v, fmt):
    """k, v [T, H, D] of one sequence as the cache returns them, [H, T, D] in 64 bits."""
    bits, scheme, group, axis = fmt
    k, v = k.transpose(0, 1), v.transpose(0, 1)
    vh = _stored(v, bits, scheme, group)
    if axis == "token":
        return _stored(k, bits, scheme, group), vh
    k = k.bfloat16()
    full = k.shape[1] // group * group
    kq = _grouped(k[:, :full].transpose(1, 2).contiguous(), bits, group).transpose(1, 2)
    return torch.cat([kq, k[:, full:].double()], 1), vh


def _attend(q, k, v, scale):
    """q [H, R, D] over k, v [H, T, *]; row r of R sees the positions up to T - R + r."""
    x = torch.matmul(q, k.transpose(1, 2)).mul_(scale)
    R, T = x.shape[1:]
    if R > 1:
        x.masked_fill_(torch.ones((R, T), dtype=torch.bool, device=x.device).triu_(T - R + 1), -math.inf)
    return torch.matmul(torch.softmax(x, -1), v)


def _exact_gqa(case, kv, q, lens, fmt, kept=None):
    """[B, Hq, D], or [B, R, Hq, D] for chunks."""
    Hq, H, D = MODELS[case["model"]]
    G = Hq // H
    outs = []
    for b, n in enumerate(lens):
        k, v = _stored_kv(kv[0][b, :n], kv[1][b, :n], fmt)
        if kept is not None:
            k, v = k[:, kept[b].long()], v[:, kept[b].long()]
        qb = q[b].double()
        if qb.dim() == 2:
            outs.append(_attend(qb.view(H, G, D).flatten(0, 1).unsqueeze(1), k.repeat_interleave(G, 0),
                                v.repeat_interleave(G, 0), _sigma(case)).squeeze(1)
                        if n * Hq * D < 1 << 28 else
                        torch.cat([torch.softmax(qb[h * G:(h + 1) * G] @ k[h].T * _sigma(case), -1) @ v[h]
                                   for h in range(H)]))
        else:
            outs.append(torch.stack([_attend(qb[:, h].unsqueeze(0), k[h // G:h // G + 1], v[h // G:h // G + 1],
                                             _sigma(case))[0] for h in range(Hq)], 1))
    return torch.stack(outs)


def _exact_mla(case, kv, q, w, lens):
    bits, scheme = MLA_FORMATS[case["format"]]
    d = case["width"]
    H = MODELS["mla"][0]
    wk, wv = w[0][:, :, :d].double(), w[1][:, :, :d].double()
    outs = []
    for b, n in enumerate(lens):
        c = _stored(kv[0][b, :n, :d], bits, scheme, d)
        r = _stored(kv[1][b, :n], bits, scheme, ROPE)
        qn, qp = q[0][b].double(), q[1][b].double()
        rows = qn.dim() == 3
        qn, qp = (qn, qp) if rows else (qn.unsqueeze(0), qp.unsqueeze(0))
        o = torch.stack([_attend(torch.cat([qn[:, h], qp[:, h]], -1).unsqueeze(0),
                                 torch.cat([c @ wk[h].T, r], -1).unsqueeze(0), (c @ wv[h].T).unsqueeze(0),
                                 _sigma(case))[0] for h in range(H)], 1)
        outs.append(o if rows else o[0])
    return torch.stack(outs)


def _exact_votes(case, kv, q):
    Hq, H, D = MODELS[case["model"]]
    G, T, n = Hq // H, case["ctx"], case["window"]
    votes = torch.zeros((case["batch"], H, T - n), dtype=torch.float64, device="cuda")
    mask = torch.ones((n, T), dtype=torch.bool, device="cuda").triu_(T - n + 1)
    for b in range(case["batch"]):
        k, _ = _stored_kv(kv[0][b], kv[1][b], GQA_FORMATS[case["format"]])
        for h in range(Hq):
            x = (q[b, :, h].double() @ k[h // G].T * _sigma(case)).masked_fill_(mask, -math.inf)
            votes[b, h // G] += torch.softmax(x, -1)[:, :T - n].sum(0)
    return votes


def exact(case, seed):
    lens = _lens(case)
    if case["kind"] == "model":
        outs, kv, fmt = [], None, None
        for l, a in enumerate(_model_layers()):
            if not a.inherit:
                kv, fmt = _kv(case, seed, l), (a.bits, a.scheme, a.group, a.key_axis)
            outs.append(_exact_gqa(case, kv, _queries(case, seed, layer=l)[0], lens, fmt))
        return outs
    kv = _kv(case, seed)
    q = _queries(case, seed, rows=case["chunk"] or case["window"])
    if case["kind"] == "evict":
        return {"votes": _exact_votes(case, kv, q[0]), "n": None, "stays": None}
    if case["model"] == "mla":
        out = _exact_mla(case, kv, q, _weights(seed), lens)
    else:
        kept = _kept(case, seed)[0] if case["keep"] else None
        out = _exact_gqa(case, kv, q[0], lens, GQA_FORMATS[case["format"]], kept)
    whole = case["kind"] == "ingest" or (case["kind"] == "prefill" and case["chunk"] == case["ctx"])
    return {"out": out, "cache": None} if whole else out
