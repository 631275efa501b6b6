"""The work this library is timed on: maintenance rounds, and each step of a round through its own call.

A case is one call (or one whole round) over a population of `chars` characters:

  round    update_round over a stack of layers: removal of superseded records, the replacement tail through every
           layer, cursor advance.  A round removes as many live entries as its tail leaves behind, so rounds chain:
           every pass is the next round of the same characters.
  attn     tail_attn_prefill of one attention layer (RoPE, append, causal GQA attention over cache and tail)
  gdn      gdn_chunk_scan_from_state of one gated-delta-rule layer, with or without its short convolution
  compact  kv_compact_noalloc on caller-owned KV slabs
  probe    attn_probe: the distribution of the last queries over the live entries, with record masses

Tails of one token are decode steps.  With several characters, prefixes and tails are ragged (packed): `prefix` and
`tail` are their upper ends, lengths are spread down to an eighth of them.  Value distributions: q, v ~ N(0, 1), unit
keys, alpha = sigmoid(N(3, 0.5)), beta = sigmoid(N(0, 1)), carried states N(0, 0.2^2).
"""
import math

import numpy as np
import torch

from paper_2609_18935_gb300 import kvm

# the hybrid stack of the library's benchmark, and the small test shape
HYBRID = {"hq": 16, "hkv": 2, "d": 256, "rot": 64, "h": 16, "dk": 128, "dv": 128}
SMALL = {"hq": 8, "hkv": 2, "d": 64, "rot": 64, "h": 8, "dk": 64, "dv": 64}
MID = {"hq": 16, "hkv": 4, "d": 128, "rot": 128, "h": 8, "dk": 128, "dv": 64}
THETA = 1.0e4


def _case(kind, shape, **kw):
    c = {"kind": kind, "chars": 1, "prefix": 0, "tail": 0, "lens": 0}
    if kind in ("round", "attn", "probe"):
        c.update({k: shape[k] for k in ("hq", "hkv", "d", "rot")})
    if kind in ("round", "gdn"):
        c.update({k: shape[k] for k in ("h", "dk", "dv")})
    c.update(kw)
    return c


def listed():
    return [
        # smallest whole round: one delta-rule and one attention layer, a 512-token character
        _case("round", SMALL, name="round_tiny", layers=2, prefix=512, tail=64, spans=2, delim=0, kv=True),
        # a game character's maintenance round: 8K of memory, a few hundred replacement tokens
        _case("round", HYBRID, name="round_npc", layers=4, prefix=8192, tail=256, spans=4, delim=0, kv=True),
        # a long-lived character in a full-depth stack, the benchmark's workload
        _case("round", HYBRID, name="round_long", layers=48, prefix=32768, tail=1024, spans=10, delim=0, kv=False),
        # one decode step of one character: a round of one token, one older entry dropped
        _case("round", HYBRID, name="round_decode", layers=4, prefix=8192, tail=1, spans=1, delim=0, kv=False),
        # attention of a from-scratch prefill
        _case("attn", HYBRID, name="attn_refill", prefix=0, tail=16896),
        # attention of a population's maintenance round, packed and ragged
        _case("attn", HYBRID, name="attn_population", chars=32, prefix=16384, tail=512, lens=3),
        # attention of a population's decode step
        _case("attn", HYBRID, name="attn_decode", chars=32, prefix=16384, tail=1, lens=5),
        # delta rule of a long-lived character's tail
        _case("gdn", HYBRID, name="gdn_long", tail=1024, conv=False),
        # delta rule with its short convolution over a population's ragged tails
        _case("gdn", HYBRID, name="gdn_population", chars=32, tail=512, lens=3, conv=True),
        # the same layer in a population's decode step
        _case("gdn", HYBRID, name="gdn_decode", chars=32, tail=1, lens=5, conv=True),
        # removal of 3 % of 32K entries in twelve layers' slabs owned by the caller
        _case("compact", HYBRID, name="compact_long", slabs=24, d=256, prefix=32768, remove=983, spans=10),
        # which memories the last eight tokens of a character attend to
        _case("probe", HYBRID, name="probe_npc", prefix=8192, nq=8, groups=32),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["round", "round", "attn", "attn", "attn", "gdn", "gdn", "gdn", "compact", "probe"])
    shape = rng.choice([HYBRID, HYBRID, HYBRID, MID, SMALL])
    one = rng.random() < 0.3                      # a decode step
    chars = 1 if rng.random() < 0.5 else _log(rng, 2, 48)
    lens = rng.randrange(1, 1 << 20) if chars > 1 else 0
    if kind == "round":
        chars = min(chars, 8)
        prefix = _log(rng, 512, 16384)
        tail = 1 if one else _log(rng, 2, min(512, prefix // 8))   # no more than any character holds
        delim = 2 if tail >= 64 and rng.random() < 0.3 else 0
        return _case(kind, shape, layers=rng.choice([2, 4, 8]), chars=chars, lens=lens, prefix=prefix, tail=tail,
                     spans=rng.randint(1, 6), delim=delim, kv=chars == 1)
    if kind == "attn":
        prefix = _log(rng, 128, 32768 if chars <= 8 else 12288)
        tail = 1 if one else _log(rng, 2, 1024 if chars == 1 else 512)
        return _case(kind, shape, chars=chars, lens=lens, prefix=prefix, tail=tail)
    if kind == "gdn":
        tail = 1 if one else _log(rng, 2, 4096 if chars == 1 else 512)
        return _case(kind, shape, chars=chars, lens=lens, tail=tail, conv=rng.random() < 0.5)
    if kind == "compact":
        prefix = _log(rng, 512, 32768)
        return _case(kind, shape, slabs=rng.randint(2, 24), d=shape["d"], prefix=prefix,
                     remove=max(8, int(prefix * rng.uniform(0.01, 0.1))), spans=rng.randint(1, 8))
    return _case(kind, shape, prefix=_log(rng, 256, 32768), nq=rng.randint(1, 16), groups=rng.randint(2, 64))


# ---------------------------------------------------------------------------- sizes of a case
def _lengths(case):
    """(prefix, tail) per character."""
    n, hi_l, hi_m = case["chars"], case["prefix"], case["tail"]
    if n == 1:
        return [hi_l], [hi_m]
    r = np.random.default_rng(case["lens"])
    spread = lambda hi: [int(x) for x in r.integers(max(1, hi // 8), hi + 1, size=n)] if hi else [0] * n
    return spread(hi_l), spread(hi_m)


def _kinds(layers):
    """Three delta-rule layers to one attention layer (one to one in a stack of two)."""
    return [kvm.LAYER_ATTN if i % 4 == 3 or (layers == 2 and i == 1) else kvm.LAYER_GDN for i in range(layers)]


def _spread_spans(live, total, n):
    """`total` of `live` entries in at most n runs, evenly placed."""
    n = max(1, min(n, total, live - total + 1))
    begin, end = [], []
    kept = live - total
    for k in range(n):
        size = total // n + (k < total % n)
        at = (kept * (2 * k + 1)) // (2 * n) + sum(e - b for b, e in zip(begin, end))
        begin.append(at)
        end.append(at + size)
    return begin, end


def _round_spans(case):
    """Each character loses as many entries as its tail leaves: (cu, begin, end)."""
    L, M = _lengths(case)
    cu, b, e = [0], [], []
    for l, m in zip(L, M):
        x, y = _spread_spans(l, min(l, m - min(case["delim"], m)), case["spans"])
        b += x
        e += y
        cu.append(len(b))
    return cu, b, e


# ---------------------------------------------------------------------------- inputs
def _gen(seed, k):
    return torch.Generator(device="cuda").manual_seed(int(seed) * 1000003 + k)


def _normal(g, *shape, unit=False):
    x = torch.randn(shape, generator=g, device="cuda", dtype=torch.float32)
    if unit:
        x = x / x.norm(dim=-1, keepdim=True)
    return x.to(torch.bfloat16)


def _attn_inputs(case, g, m):
    return {"q": _normal(g, m, case["hq"], case["d"]), "k": _normal(g, m, case["hkv"], case["d"], unit=True),
            "v": _normal(g, m, case["hkv"], case["d"])}


def _gdn_inputs(case, g, m):
    h, dk, dv = case["h"], case["dk"], case["dv"]
    gate = lambda mean, std: torch.sigmoid(mean + std * torch.randn((m, h), generator=g, device="cuda"))
    return {"q": _normal(g, m, h, dk), "k": _normal(g, m, h, dk, unit=True), "v": _normal(g, m, h, dv),
            "alpha": gate(3.0, 0.5), "beta": gate(0.0, 1.0)}


def _cache(case, g, live):
    return _normal(g, case["hkv"], live, case["d"], unit=True), _normal(g, case["hkv"], live, case["d"])


def _gdn_state(case, g):
    return 0.2 * torch.randn((case["chars"], case["h"], case["dv"], case["dk"]), generator=g, device="cuda")


def _conv(case, g):
    c = case["h"] * (2 * case["dk"] + case["dv"])
    return (0.5 * torch.randn((c, 4), generator=g, device="cuda"), _normal(g, case["chars"], 3, c))


def _context(case, kinds, conv=0):
    L, M = _lengths(case)
    get = lambda k, alt: case.get(k, alt)
    return kvm.Context(kinds, get("hq", 8), get("hkv", 2), get("d", 64), get("rot", 64), THETA, get("h", 8),
                       get("dk", 64), get("dv", 64), [max(1, l + m) for l, m in zip(L, M)], max(1, sum(M)),
                       conv_kernel=conv)


def _parts(case, seed):
    """Every random input of a case, on the GPU."""
    L, M = _lengths(case)
    m = sum(M)
    if case["kind"] == "attn":
        g = _gen(seed, 0)
        return {"x": _attn_inputs(case, g, m), "cache": [_cache(case, g, l) for l in L]}
    if case["kind"] == "gdn":
        g = _gen(seed, 0)
        return {"x": _gdn_inputs(case, g, m), "S": _gdn_state(case, g), "conv": _conv(case, g) if case["conv"] else None}
    if case["kind"] == "compact":
        g = _gen(seed, 0)
        n, l, d = case["slabs"], case["prefix"], case["d"]
        pos = torch.cumsum(torch.randint(1, 4, (l,), generator=g, device="cuda"), 0).to(torch.int32)
        return {"K": _normal(g, n, l, d), "V": _normal(g, n, l, d), "pos": pos}
    if case["kind"] == "probe":
        g = _gen(seed, 0)
        group = torch.sort(torch.randint(0, case["groups"], (L[0],), generator=g, device="cuda")).values
        return {"cache": [_cache(case, g, L[0])], "q": _normal(g, case["nq"], case["hq"], case["d"]),
                "group": group.to(torch.int32)}
    out = {"layers": []}
    for i, kind in enumerate(_kinds(case["layers"])):
        g = _gen(seed, i)
        if kind == kvm.LAYER_ATTN:
            out["layers"].append({"x": _attn_inputs(case, g, m), "cache": [_cache(case, g, l) for l in L]})
        else:
            out["layers"].append({"x": _gdn_inputs(case, g, m), "S": _gdn_state(case, g)})
    return out


def _cu(lengths):
    return np.concatenate([[0], np.cumsum(lengths)]).astype(np.int32)


def _load(ctx, L, layer, cache):
    for b, (k, v) in enumerate(cache):
        if L[b]:
            ctx.set_kv(layer, b, k, v)


def prepare(case, seed):
    L, M = _lengths(case)
    m, p = sum(M), _parts(case, seed)
    s = {"case": case, "cu": _cu(M)}
    if case["kind"] == "compact":
        b, e = _spread_spans(case["prefix"], case["remove"], case["spans"])
        s.update(K=p["K"], V=p["V"], pos=p["pos"], begin=np.array(b, np.int32), end=np.array(e, np.int32))
        return s
    if case["kind"] == "gdn":
        ctx = _context(case, [kvm.LAYER_GDN], 4 if case["conv"] else 0)
        ctx.set_state(0, p["S"])
        if case["conv"]:
            ctx.set_conv_weights(0, p["conv"][0])
            ctx.set_conv_state(0, p["conv"][1])
        s.update(ctx=ctx, x=p["x"], out=torch.empty_like(p["x"]["v"]))
        return s
    kinds = _kinds(case["layers"]) if case["kind"] == "round" else [kvm.LAYER_ATTN]
    ctx = _context(case, kinds)
    for b, l in enumerate(L):
        ctx.load_prefix(b, l, l, np.arange(l, dtype=np.int32))
    s["ctx"] = ctx
    if case["kind"] == "attn":
        _load(ctx, L, 0, p["cache"])
        s.update(x=p["x"], out=torch.empty_like(p["x"]["q"]))
    elif case["kind"] == "probe":
        _load(ctx, L, 0, p["cache"])
        s.update(q=p["q"], group=p["group"])
    else:
        n_attn = kinds.count(kvm.LAYER_ATTN)
        bf = dict(dtype=torch.bfloat16, device="cuda")
        attn = torch.empty((n_attn, m, case["hq"], case["d"]), **bf)
        gdn = torch.empty((len(kinds) - n_attn, m, case["h"], case["dv"]), **bf)
        ins, outs, a, g = {}, {}, 0, 0
        for i, (kind, q) in enumerate(zip(kinds, p["layers"])):
            ins[i] = q["x"]
            if kind == kvm.LAYER_ATTN:
                _load(ctx, L, i, q["cache"])
                outs[i], a = attn[a], a + 1
            else:
                ctx.set_state(i, q["S"])
                outs[i], g = gdn[g], g + 1
        cu, b, e = (np.array(x, np.int32) for x in _round_spans(case))
        delim = None
        if case["delim"]:
            # the tail's first tokens delimit the replacement
            at = [0] * case["chars"]
            n = [min(case["delim"], x) for x in M]
            delim = tuple(np.array(x, np.int32) for x in (range(case["chars"] + 1), at, n))
        s.update(kinds=kinds, ins=ins, outs=outs, attn=attn, gdn=gdn, spans=(cu, b, e), delim=delim)
    torch.cuda.synchronize()                      # set_kv and set_state read the tensors made here
    return s


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "attn":
        x = s["x"]
        s["ctx"].tail_attn_prefill(0, s["cu"], x["q"], x["k"], x["v"], s["out"])
        return {"out": s["out"]}
    if kind == "gdn":
        x = s["x"]
        s["ctx"].gdn_chunk_scan_from_state(0, s["cu"], x["q"], x["k"], x["v"], x["alpha"], x["beta"], s["out"])
        return {"out": s["out"], "state": s["ctx"].get_state(0)}
    if kind == "compact":
        live = kvm.kv_compact_noalloc(s["K"], s["V"], s["pos"], case["prefix"], s["begin"], s["end"])
        # rows from the new live length on are the caller's free space
        return {"live": live, "K": s["K"][:, :live], "V": s["V"][:, :live], "pos": s["pos"][:live]}
    if kind == "probe":
        probs, mass = s["ctx"].attn_probe(0, 0, s["q"], s["group"], case["groups"])
        return {"probs": probs, "mass": mass}
    ctx = s["ctx"]
    ctx.update_round(*s["spans"], s["cu"], s["ins"], s["outs"], delim=s["delim"])
    out = {"attn": s["attn"], "gdn": s["gdn"],
           "state": [ctx.get_state(i) for i, k in enumerate(s["kinds"]) if k == kvm.LAYER_GDN]}
    if case["kv"]:
        out["kv"] = [ctx.get_kv(i, 0) for i, k in enumerate(s["kinds"]) if k == kvm.LAYER_ATTN]
        out["pos"] = ctx.get_positions(0)
    return out


# ---------------------------------------------------------------------------- work of a pass
def _attn_work(case, L, M):
    pairs = sum(m * l + m * (m + 1) / 2 for l, m in zip(L, M))
    m, hq, hkv, d = sum(M), case["hq"], case["hkv"], case["d"]
    # survivors' K and V, the tail's q, k, v in, the output and the appended rows out
    return sum(l for l, t in zip(L, M) if t) * hkv * d * 4 + m * (2 * hq + 4 * hkv) * d * 2, 4 * d * hq * pairs


def _gdn_work(case, M, conv):
    m, h, dk, dv = sum(M), case["h"], case["dk"], case["dv"]
    act = sum(1 for x in M if x)
    b = m * h * ((2 * dk + 2 * dv) * 2 + 8) + act * h * dv * dk * 8
    f = 6 * dk * dv * h * m
    if conv:
        ch = h * (2 * dk + dv)
        b += ch * 16 + act * 3 * ch * 4
        f += 8 * ch * m
    return b, f


def work(case):
    kind = case["kind"]
    L, M = _lengths(case)
    if kind == "attn":
        b, f = _attn_work(case, L, M)
    elif kind == "gdn":
        b, f = _gdn_work(case, M, case["conv"])
    elif kind == "compact":
        x, _ = _spread_spans(case["prefix"], case["remove"], case["spans"])
        moved = case["prefix"] - case["remove"] - x[0]
        b, f = 2 * moved * (2 * case["slabs"] * case["d"] * 2 + 4), 0
    elif kind == "probe":
        b = L[0] * (case["hkv"] * case["d"] * 2 + 8) + case["nq"] * case["hq"] * case["d"] * 2
        f = 2 * case["nq"] * case["hq"] * L[0] * case["d"]
    else:
        cu, x, y = _round_spans(case)
        kinds = _kinds(case["layers"])
        n_attn = kinds.count(kvm.LAYER_ATTN)
        gone = [sum(y[k] - x[k] for k in range(cu[i], cu[i + 1])) for i in range(len(L))]
        moved = sum(l - r - x[cu[i]] for i, (l, r) in enumerate(zip(L, gone)))
        ab, af = _attn_work(case, [l - r for l, r in zip(L, gone)], M)
        gb, gf = _gdn_work(case, M, False)
        b = n_attn * ab + (len(kinds) - n_attn) * gb + 2 * moved * (n_attn * case["hkv"] * case["d"] * 4 + 4)
        f = n_attn * af + (len(kinds) - n_attn) * gf
    return {"bytes": float(b), "flops": float(f)}


def tolerance(case):
    if case["kind"] == "compact":
        return "exact"                            # rows move, bit for bit
    if case["kind"] == "probe":
        return {"rel": 1e-5}                      # 32-bit sums
    return {"rel": 8e-3}                          # bf16 outputs; bf16 keys, probabilities and convolved inputs


# ---------------------------------------------------------------------------- the same in 64 bits
def _rope(x, pos, rot):
    """x [n][heads][d] in 64 bits, rotated at pos [n]: pairs (i, i + rot/2) of the first rot dims."""
    half = rot // 2
    freq = THETA ** (-2.0 * torch.arange(half, device=x.device, dtype=torch.float64) / rot)
    ang = pos.to(torch.float64)[:, None, None] * freq
    a, b = x[..., :half], x[..., half:rot]
    return torch.cat([a * ang.cos() - b * ang.sin(), a * ang.sin() + b * ang.cos(), x[..., rot:]], -1)


def _attn_exact(case, x, cache, L, M, keep=None):
    """(out, per character the cache after it); keep: per character the surviving rows."""
    out, after, at = [], [], 0
    g = case["hq"] // case["hkv"]
    for b, (l, m) in enumerate(zip(L, M)):
        K, V = (t.double() for t in cache[b])
        if keep is not None:
            K, V = K[:, keep[b]], V[:, keep[b]]
        n = K.shape[1]
        pos = l + torch.arange(m, device="cuda")
        q = _rope(x["q"][at:at + m].double(), pos, case["rot"])
        K = torch.cat([K, _rope(x["k"][at:at + m].double(), pos, case["rot"]).transpose(0, 1)], 1)
        V = torch.cat([V, x["v"][at:at + m].double().transpose(0, 1)], 1)
        o = torch.empty_like(q)
        step = max(1, min(m, (1 << 27) // (max(1, n + m) * g)))
        for i in range(0, m, step):
            j = min(m, i + step)
            hidden = torch.arange(n + j, device="cuda")[None, :] > (n + torch.arange(i, j, device="cuda"))[:, None]
            for h in range(case["hkv"]):
                w = torch.einsum("mgd,nd->gmn", q[i:j, h * g:(h + 1) * g], K[h, :n + j]) / math.sqrt(case["d"])
                w = torch.softmax(w.masked_fill_(hidden, -math.inf), -1)
                o[i:j, h * g:(h + 1) * g] = torch.einsum("gmn,nd->mgd", w, V[h, :n + j])
        out.append(o)
        after.append((K, V))
        at += m
    return torch.cat(out), after


def _gdn_exact(case, x, S, M, conv=None):
    """Token by token: (out, state)."""
    x = {k: v.double() for k, v in x.items()}
    S = S.double().clone()
    cu = _cu(M)
    if conv is not None:
        w, old = conv[0].double(), conv[1].double()
        flat = torch.cat([x[k].flatten(1) for k in ("q", "k", "v")], 1)
        rows = []
        for b, m in enumerate(M):
            y = torch.cat([old[b], flat[cu[b]:cu[b + 1]]])
            y = sum(w[:, i] * y[i:i + m] for i in range(4))
            rows.append(y * torch.sigmoid(y))
        q, k, v = torch.cat(rows).split([x[n][0].numel() for n in ("q", "k", "v")], 1)
        x["q"], x["v"] = q.reshape(x["q"].shape), v.reshape(x["v"].shape)
        k = k.reshape(x["k"].shape)
        x["k"] = k / k.norm(dim=-1, keepdim=True)
    out = torch.empty_like(x["v"])
    order = sorted(range(len(M)), key=lambda b: -M[b])     # characters still running come first
    S = S[order]
    start = torch.as_tensor([int(cu[b]) for b in order], device="cuda")
    for t in range(max(M)):
        n = sum(1 for b in order if M[b] > t)
        at = start[:n] + t
        k, q, v = x["k"][at], x["q"][at], x["v"][at]
        al, be = x["alpha"][at][..., None], x["beta"][at][..., None]
        T = S[:n]
        u = be * (v - al * torch.einsum("bhvk,bhk->bhv", T, k))
        T *= al[..., None]
        T += u[..., None] * k[..., None, :]
        out[at] = torch.einsum("bhvk,bhk->bhv", T, q)
    back = torch.empty_like(S)
    back[order] = S
    return out, back


def exact(case, seed):
    L, M = _lengths(case)
    p = _parts(case, seed)
    kind = case["kind"]
    if kind == "attn":
        return {"out": _attn_exact(case, p["x"], p["cache"], L, M)[0]}
    if kind == "gdn":
        out, S = _gdn_exact(case, p["x"], p["S"], M, p["conv"])
        return {"out": out, "state": S}
    if kind == "compact":
        b, e = _spread_spans(case["prefix"], case["remove"], case["spans"])
        keep = torch.ones(case["prefix"], dtype=torch.bool, device="cuda")
        for i, j in zip(b, e):
            keep[i:j] = False
        return {"live": int(keep.sum()), "K": p["K"][:, keep].double(), "V": p["V"][:, keep].double(), "pos": p["pos"][keep]}
    if kind == "probe":
        n, l = case["nq"], L[0]
        K = p["cache"][0][0].double()
        pos = torch.arange(l - n, l, device="cuda")
        q = _rope(p["q"].double(), pos, case["rot"])
        K = K.repeat_interleave(case["hq"] // case["hkv"], 0)
        w = torch.einsum("mhd,hnd->mhn", q, K) / math.sqrt(case["d"])
        w = w.masked_fill(torch.arange(l, device="cuda")[None, None, :] > pos[:, None, None], -math.inf)
        probs = torch.softmax(w, -1).mean((0, 1))
        mass = torch.zeros(case["groups"], dtype=torch.float64, device="cuda").index_add_(0, p["group"].long(), probs)
        return {"probs": probs, "mass": mass}
    cu, x, y = _round_spans(case)
    keep = []
    for b, l in enumerate(L):
        k = torch.ones(l, dtype=torch.bool, device="cuda")
        for i in range(cu[b], cu[b + 1]):
            k[x[i]:y[i]] = False
        keep.append(k)
    r = {"attn": [], "gdn": [], "state": [], "kv": []}
    for kind, q in zip(_kinds(case["layers"]), p["layers"]):
        if kind == kvm.LAYER_ATTN:
            out, after = _attn_exact(case, q["x"], q["cache"], L, M, keep)
            r["attn"].append(out)
            gone = min(case["delim"], M[0])
            n = int(keep[0].sum())
            rest = [i for i in range(n + M[0]) if not n <= i < n + gone] if gone else slice(None)
            r["kv"].append(tuple(t[:, rest] for t in after[0]))
        else:
            out, S = _gdn_exact(case, q["x"], q["S"], M)
            r["gdn"].append(out)
            r["state"].append(S)
    r["attn"], r["gdn"] = torch.stack(r["attn"]), torch.stack(r["gdn"])
    if not case["kv"]:
        del r["kv"]
    return r
