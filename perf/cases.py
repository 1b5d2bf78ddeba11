"""The work that users of this library have it do, as timed cases.

Four kinds of pass, each through the package's public entry points:

``step``       one decode step over a filled paged cache: for each layer the new token is written and the metered decode
               runs over the whole context (one fused call where the cache allows it, else write and decode), then one
               gate over all cells.  ``variant`` picks the plain decode or one of its certificates.  A serving loop captures
               its step once in a CUDA graph (``graph``); a first integration calls it eagerly.
``prefill``    the write path over a prompt (or a chunk of one).
``calibrate``  the grouped scheme's set-up: choose the outlier pairs from the prompt's keys, then write the prompt.
``select``     block-level repair selection for every cell of a step, from per-page terms.

Head shapes, context lengths and options are those of the repository's workloads and tests (28 query / 4 KV heads,
8 / 2, up to 8 query heads per KV head; 4k to 128k tokens; batches of 16 x 4k-8k and 32 x 4k-32k).
"""

import dataclasses
import math

import torch

import paper_2607_28699_gb300 as wc

PAGE, DIM = 16, 128
SCHEMES = {"int8": (wc.SCHEME_DITHER_INT8, 8), "int8-10bit": (wc.SCHEME_DITHER_INT8, 10),
           "fp8": (wc.SCHEME_FP8_E4M3, 8), "g32": (wc.SCHEME_DITHER_INT8_G32, 8)}
DELTA = 1e-2 / 784      # Tier-B budget of one cell: 1e-2 over 28 layers x 28 heads


def _step(name, scheme, layers, batch, lo, hi, hq, hkv, variant="plain", rope="half", m=0, tau=0.1, graph=True):
    return {"name": name, "kind": "step", "scheme": scheme, "layers": layers, "batch": batch, "ctx_lo": lo, "ctx_hi": hi,
            "hq": hq, "hkv": hkv, "variant": variant, "rope": rope, "m": m, "tau": tau, "graph": graph}


def listed():
    return [
        # The first call anybody makes: one layer, one short context, no graph; host work and launches count.
        _step("decode-4k-eager", "int8", 1, 1, 4096, 4096, 8, 2, graph=False),
        # A 7B-class model's decode step at 32k, all 28 layers.
        _step("step-32k", "int8", 28, 1, 32768, 32768, 28, 4),
        # Serving: 16 ragged sequences of 4k to 8k on shuffled pages.
        _step("step-batch16", "int8", 8, 16, 4096, 8192, 28, 4),
        # The longest context.
        _step("step-128k", "int8", 4, 1, 131072, 131072, 28, 4),
        # The raw-cast fp8 cache on the largest batch (32 x 4k to 32k), written and read by separate calls.
        _step("step-fp8-batch32", "fp8", 2, 32, 4096, 32768, 28, 4),
        # The finer dither, interleaved RoPE, a small batch of uneven contexts, four query heads per KV head.
        _step("step-10bit-batch4", "int8-10bit", 8, 4, 1000, 16001, 32, 8, rope="interleaved"),
        # The grouped-scale cache with four bypassed pairs and the Tier-B certificate.
        _step("step-g32-tier-b", "g32", 8, 1, 32768, 32768, 28, 4, variant="tier_b", m=4),
        # Output bounds: the value-side decode and the joint gate; two odd contexts, five query heads per KV head.
        _step("step-value-side", "int8", 8, 2, 9001, 20003, 40, 8, variant="value"),
        # Prompt write of 32k tokens, the shape of the write benchmark.
        {"name": "prefill-32k", "kind": "prefill", "scheme": "int8", "n_tok": 32768, "hkv": 4, "rope": "half",
         "value": False},
        # A chunk of a chunked prefill into the fp8 cache, with the value witness.
        {"name": "prefill-fp8-chunk", "kind": "prefill", "scheme": "fp8", "n_tok": 8191, "hkv": 8, "rope": "interleaved",
         "value": True},
        # Grouped cache set-up on a 16k prompt.
        {"name": "calibrate-16k", "kind": "calibrate", "n_tok": 16384, "hkv": 4, "rope": "half", "m": 4},
        # Which pages to repair, for every cell of a 28-layer step at 32k.
        {"name": "repair-select-32k", "kind": "select", "rows": 28, "hq": 28, "pages": 2048, "tau": 0.1},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step"] * 6 + ["prefill"] * 2 + ["calibrate", "select"])
    rope = rng.choice(["half", "interleaved"])
    if kind == "prefill":
        hkv = rng.choice([1, 2, 4, 8])
        scheme = rng.choice(["int8", "int8", "int8-10bit", "fp8", "g32"])
        return {"kind": kind, "scheme": scheme, "n_tok": _log(rng, 1, 131072 // hkv), "hkv": hkv, "rope": rope,
                "value": scheme != "g32" and rng.random() < 0.3}
    if kind == "calibrate":
        hkv = rng.choice([1, 2, 4, 8])
        return {"kind": kind, "n_tok": _log(rng, 256, 131072 // hkv), "hkv": hkv, "rope": rope, "m": rng.randint(1, 16)}
    if kind == "select":
        pages = _log(rng, 8, 8192)
        return {"kind": kind, "rows": rng.randint(1, max(1, 57344 // pages)), "hq": rng.choice([8, 28, 32]), "pages": pages,
                "tau": rng.choice([0.02, 0.05, 0.1, 0.2])}
    scheme = rng.choice(["int8", "int8", "int8", "int8-10bit", "fp8", "g32"])
    variants = {"int8": ["plain", "plain", "tier_b", "value", "repair"], "int8-10bit": ["plain", "tier_b", "value"],
                "fp8": ["plain", "plain", "value", "repair"], "g32": ["plain", "tier_b"]}[scheme]
    hkv = rng.choice([1, 2, 4, 8])
    hq = hkv * rng.randint(1, 8)
    batch = rng.choice([1, 1, 2, 4, 8, 16, 32])
    hi = _log(rng, 64, 131072 // batch)
    lo = hi if batch == 1 else max(1, hi // rng.choice([1, 2, 8]))
    layers = max(1, min(8, 2_000_000 // (hi * batch * hkv)))
    c = _step("", scheme, layers, batch, lo, hi, hq, hkv, rng.choice(variants), rope, rng.randint(0, 16) if scheme == "g32" else 0,
              rng.choice([0.05, 0.1, 0.2]), rng.random() < 0.8)
    del c["name"]
    return c


# ---------------------------------------------------------------------------------------------------------------------
# inputs: the same draws for prepare() and exact()


def _gen(seed, salt):
    return torch.Generator(device="cuda").manual_seed((seed * 1_000_003 + salt * 7919 + 17) % 2**63)


def _ctx_lens(case, seed):
    g = torch.Generator().manual_seed(seed * 31 + 5)
    lens = torch.randint(case["ctx_lo"], case["ctx_hi"] + 1, (case["batch"],), generator=g).tolist()
    lens[seed % case["batch"]] = case["ctx_hi"]
    return lens


def _rope(x, pos, rope):
    inv = 1e4 ** (-torch.arange(DIM // 2, device=x.device, dtype=torch.float64) * 2.0 / DIM)
    ang = pos.to(torch.float64)[:, None] * inv
    cos, sin = ang.cos().float()[:, None], ang.sin().float()[:, None]
    if rope == "half":
        a, b = x[..., :DIM // 2], x[..., DIM // 2:]
        return torch.cat([a * cos - b * sin, a * sin + b * cos], dim=-1)
    a, b = x[..., 0::2], x[..., 1::2]
    return torch.stack([a * cos - b * sin, a * sin + b * cos], dim=-1).flatten(-2)


def _kv(seed, layer, lens, hkv, rope):
    """Post-RoPE K and V, fp16 [sum(lens), hkv, 128]: log-normal channel scales and a sink token 8 times the others' norm."""
    g = _gen(seed, 2 * layer + 1)
    sk = torch.exp(0.5 * torch.randn(hkv, DIM, generator=g, device="cuda"))
    sv = torch.exp(0.5 * torch.randn(hkv, DIM, generator=g, device="cuda"))
    n = sum(lens)
    pos = torch.cat([torch.arange(s, device="cuda") for s in lens])
    sink = torch.where(pos == 0, 8.0, 1.0)[:, None, None]
    k = _rope(torch.randn(n, hkv, DIM, generator=g, device="cuda") * sk * sink, pos, rope).half()
    v = (torch.randn(n, hkv, DIM, generator=g, device="cuda") * sv * sink).half()
    return k, v


def _queries(case, seed, layer, lens):
    g = _gen(seed, 2 * layer + 2)
    q = torch.randn(len(lens), case["hq"], DIM, generator=g, device="cuda")
    return _rope(q, torch.tensor(lens, device="cuda") - 1, case["rope"]).half()


def _tables(lens, hi, seed):
    """Block tables over shuffled pages of a pool for len(lens) sequences of up to hi tokens, every token's slot, and the
    pool's size."""
    per = [(s + PAGE - 1) // PAGE for s in lens]
    most = (hi + PAGE - 1) // PAGE
    order = torch.randperm(len(lens) * most, generator=torch.Generator().manual_seed(seed * 17 + 3)).int()
    bt = torch.full((len(lens), most), -1, dtype=torch.int32)
    slots, at = [], 0
    for b, (s, n) in enumerate(zip(lens, per)):
        bt[b, :n] = order[at:at + n]
        at += n
        t = torch.arange(s)
        slots.append(bt[b, t // PAGE] * PAGE + (t % PAGE).int())
    return bt.cuda(), torch.cat(slots).int().cuda(), len(order)


def _pairs(seed, layer, hkv, m):
    g = torch.Generator().manual_seed(seed * 13 + layer)
    return torch.stack([torch.randperm(DIM // 2, generator=g)[:m].sort().values for _ in range(hkv)]).int().cuda()


def _desc(case, seed, pages):
    scheme, bits = SCHEMES[case.get("scheme", "g32")]
    return wc.CacheDesc(num_q_heads=case.get("hq", case["hkv"]), num_kv_heads=case["hkv"], num_pages=pages, scheme=scheme,
                        rope_layout=wc.ROPE_HALF if case["rope"] == "half" else wc.ROPE_INTERLEAVED, dither_bits=bits, seed=seed)


def _terms(case, seed):
    """Per-page terms as a decode leaves them: references that follow a running maximum, contributions spread over the
    context with a heavy first page, ragged context lengths."""
    g = _gen(seed, 9)
    rows, hq, pages = case["rows"], case["hq"], case["pages"]
    ref = 2.0 + torch.randn(rows, hq, pages, generator=g, device="cuda").abs()
    d = torch.exp(0.7 * torch.randn(rows, hq, pages, generator=g, device="cuda")) * 0.9
    d[..., 0] *= 40.0
    norm = torch.empty(rows, hq, 2, device="cuda")
    norm[..., 0] = 6.0
    norm[..., 1] = float(pages) * (0.4 + 0.3 * torch.rand(rows, hq, generator=g, device="cuda"))
    lens = torch.randint(max(1, pages * PAGE // 2), pages * PAGE + 1, (rows,), generator=g, device="cuda").int()
    lens[0] = pages * PAGE
    return torch.stack([ref, d], dim=-1).contiguous(), norm, lens


# ---------------------------------------------------------------------------------------------------------------------


def prepare(case, seed):
    return {"step": _prepare_step, "prefill": _prepare_write, "calibrate": _prepare_write, "select": _prepare_select}[case["kind"]](case, seed)


def _prepare_step(case, seed):
    lens = _ctx_lens(case, seed)
    bt, slots, pages = _tables(lens, case["ctx_hi"], seed)
    L, B, hkv, hq, m = case["layers"], case["batch"], case["hkv"], case["hq"], case["m"]
    desc = _desc(case, seed, pages)
    value = case["variant"] == "value"
    ends = torch.tensor(lens).cumsum(0).cuda() - 1          # each sequence's newest token
    old = slots.clone()
    old[ends] = -1                                          # it is written by the step
    s = {"case": case, "desc": desc, "bt": bt, "ctx": torch.tensor(lens, dtype=torch.int32, device="cuda"), "slot_new": slots[ends].contiguous(),
         "ws": wc.Workspace(desc, B, bt.shape[1]), "tau": case["tau"], "layers": []}
    # every layer's cache as a view of arrays stacked over the layers
    one = wc.LayerCache.empty(desc, value_witness=value, num_bypass_pairs=m)
    s["cache"] = {f.name: torch.zeros((L, *getattr(one, f.name).shape), dtype=getattr(one, f.name).dtype, device="cuda")
                  for f in dataclasses.fields(one) if getattr(one, f.name) is not None}
    for layer in range(L):
        cache = wc.LayerCache(**{f.name: s["cache"][f.name][layer] if f.name in s["cache"] else None for f in dataclasses.fields(one)})
        if m:
            cache.bypass_pairs.copy_(_pairs(seed, layer, hkv, m))
        k, v = _kv(seed, layer, lens, hkv, case["rope"])
        wc.kv_quantize_witness(desc, layer, k, v, old, cache)
        s["layers"].append((_queries(case, seed, layer, lens), cache, k[ends].contiguous(), v[ends].contiguous()))
        del k, v
    del one
    if not case["graph"]:
        return s
    cells = (L, B, hq)
    new = lambda *shape: torch.zeros(shape, dtype=torch.float32, device="cuda")   # noqa: E731
    s["buf"] = {"out": new(*cells, DIM), "raw": new(*cells), "meter": new(*cells), "x0": new(*cells), "x1": new(*cells), "x2": new(*cells)}
    if case["variant"] == "repair":
        s["terms"], s["norm"] = new(*cells, bt.shape[1], 2), new(*cells, 2)
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(side):
        _run_step(s)
    torch.cuda.current_stream().wait_stream(side)
    torch.cuda.synchronize()
    s["captured"] = torch.cuda.CUDAGraph()
    with torch.cuda.graph(s["captured"]):
        s["result"] = _run_step(s)
    return s


def _run_step(s):
    case, desc, ws = s["case"], s["desc"], s["ws"]
    variant, buf = case["variant"], s.get("buf")
    got = []
    for i, (q, cache, k_new, v_new) in enumerate(s["layers"]):
        o = {} if buf is None else {"out": buf["out"][i], "meter": buf["meter"][i], "meter_raw": buf["raw"][i]}
        if variant == "plain" and case["scheme"] == "int8":
            got.append(wc.metered_decode_attention_append(desc, i, q, s["bt"], s["ctx"], cache, ws, k_new, v_new, s["slot_new"], **o))
            continue
        wc.kv_quantize_witness(desc, i, k_new, v_new, s["slot_new"], cache)
        if variant == "plain":
            got.append(wc.metered_decode_attention(desc, i, q, s["bt"], s["ctx"], cache, ws, **o))
        elif variant == "tier_b":
            if buf is not None:
                o.update(meter_b=buf["x0"][i], meter_b_raw=buf["x1"][i])
            got.append(wc.metered_decode_attention_tier_b(desc, i, q, s["bt"], s["ctx"], cache, ws, DELTA, **o))
        elif variant == "value":
            if buf is not None:
                o.update(value_term=buf["x0"][i], v_max=buf["x1"][i], out_bound=buf["x2"][i])
            got.append(wc.metered_decode_attention_v(desc, i, q, s["bt"], s["ctx"], cache, ws, **o))
        else:
            if buf is not None:
                o.update(page_terms=s["terms"][i], softmax_norm=s["norm"][i])
            got.append(wc.metered_decode_attention_repair(desc, i, q, s["bt"], s["ctx"], cache, ws, **o))
    if buf is None:
        r = [torch.stack(x) for x in zip(*got)] if len(got) > 1 else [x[None] for x in got[0]]
    else:
        r = [buf["out"], buf["meter"], buf["raw"]]
        r += {"plain": [], "tier_b": [buf["x0"], buf["x1"]], "value": [buf["x0"], buf["x1"], buf["x2"]], "repair": [s.get("terms"), s.get("norm")]}[variant]
    res = {"out": r[0], "meter": r[1], "meter_raw": r[2]}
    # the certificate that the step gates on
    if variant == "value":
        res.update(value_term=r[3], v_max=r[4], out_bound=r[5])
        gated = wc.gate_joint(r[2].reshape(-1), r[3].reshape(-1), r[4].reshape(-1), desc.group, s["tau"], 0.01)
    else:
        if variant == "tier_b":
            res.update(meter_b=r[3], meter_b_raw=r[4])
        gated = wc.gate((r[4] if variant == "tier_b" else r[2]).reshape(-1), desc.group, s["tau"])
    res["keep_q"], res["keep_kv"], res["n_kept"] = gated
    if variant == "repair":
        # The terms' references are the decode's own choice: what they say is the contribution of each page.  The lists
        # that follow from the last bits of these are compared by the select cases, on terms that both sides share.
        n = len(s["layers"])
        contrib, _, _, _ = wc.repair_select(r[3].flatten(0, 1), r[4].flatten(0, 1), s["ctx"].repeat(n), s["tau"], keep_q=gated[0])
        res["contrib"] = contrib
    res.update((n, t) for n, t in s["cache"].items() if t.numel())      # the step's updated caches
    return res


def _prepare_write(case, seed):
    lens = [case["n_tok"]]
    _, slots, pages = _tables(lens, case["n_tok"], seed)
    k, v = _kv(seed, 0, lens, case["hkv"], case["rope"])
    desc = _desc(case, seed, pages)
    m = case.get("m", 4 if case.get("scheme") == "g32" else 0)
    cache = wc.LayerCache.empty(desc, value_witness=case.get("value", False), num_bypass_pairs=m)
    if case["kind"] == "prefill" and m:
        cache.bypass_pairs.copy_(_pairs(seed, 0, case["hkv"], m))
    return {"case": case, "desc": desc, "k": k, "v": v, "slots": slots, "cache": cache}


def _prepare_select(case, seed):
    terms, norm, lens = _terms(case, seed)
    shape = terms.shape[:3]
    return {"case": case, "terms": terms, "norm": norm, "ctx": lens, "contrib": torch.zeros(shape, device="cuda"),
            "pages": torch.full(shape, -1, dtype=torch.int32, device="cuda")}


def run(state):
    case = state["case"]
    if case["kind"] == "step":
        if "captured" in state:
            state["captured"].replay()
            return state["result"]
        return _run_step(state)
    if case["kind"] == "select":
        contrib, pages, n, after = wc.repair_select(state["terms"], state["norm"], state["ctx"], case["tau"], contrib=state["contrib"], repair_pages=state["pages"])
        return {"contrib": contrib, "pages": pages, "n_repair": n, "d_after": after}
    cache = state["cache"]
    if case["kind"] == "calibrate":
        wc.select_bypass_pairs(state["k"], case["m"], state["desc"].rope_layout, pairs=cache.bypass_pairs)
    wc.kv_quantize_witness(state["desc"], 0, state["k"], state["v"], state["slots"], cache)
    names = ("k_codes", "v_codes", "k_scale", "v_scale", "k_witness", "v_witness", "k_bypass", "bypass_pairs")
    return {n: getattr(cache, n) for n in names if getattr(cache, n) is not None and getattr(cache, n).numel()}


def _row_bytes(scheme, value, m):
    """Cache bytes of one token and KV head."""
    return 256 + {"int8": 4, "int8-10bit": 4, "fp8": 0, "g32": 16 + 4 * m}[scheme] + 16 + (4 if value else 0)


def work(case):
    if case["kind"] == "select":
        cells = case["rows"] * case["hq"]
        n = cells * case["pages"] * 0.75                     # contexts are half to all of the table
        return {"bytes": n * 12 + cells * 16, "flops": n * 4}
    if case["kind"] in ("prefill", "calibrate"):
        scheme = case.get("scheme", "g32")
        m = case.get("m", 4 if scheme == "g32" else 0)
        rows = case["n_tok"] * case["hkv"]
        return {"bytes": rows * (512 + _row_bytes(scheme, case.get("value", False), m)) + 4 * case["n_tok"], "flops": rows * DIM * 2 * 12}
    tokens = case["layers"] * (case["ctx_hi"] + (case["batch"] - 1) * (case["ctx_lo"] + case["ctx_hi"]) / 2)
    cells = case["layers"] * case["batch"] * case["hq"]
    b = tokens * case["hkv"] * _row_bytes(case["scheme"], case["variant"] == "value", case["m"])
    b += cells * (DIM * 6 + 12) + case["layers"] * case["batch"] * case["hkv"] * 512
    if case["variant"] == "repair":
        b += tokens / PAGE * case["hq"] * 4
    return {"bytes": b, "flops": tokens * case["hq"] * (4 * DIM + 16)}


# ---------------------------------------------------------------------------------------------------------------------
# what run() returns, in 64 bits


def _philox(c0, c1, c2, c3, seed):
    k0, k1, low = seed & 0xFFFFFFFF, seed >> 32, 0xFFFFFFFF
    for _ in range(10):
        p0, p1 = 0xD2511F53 * c0, 0xCD9E8D57 * c2          # 64-bit products, wrapping
        c0, c1, c2, c3 = ((p1 >> 32) & low) ^ c1 ^ k0, p1 & low, ((p0 >> 32) & low) ^ c3 ^ k1, p0 & low
        k0, k1 = (k0 + 0x9E3779B9) & low, (k1 + 0xBB67AE85) & low
    return torch.stack([c0, c1, c2, c3], dim=-1)


def _xi(slots, layer, hkv, row, scheme, seed):
    """The dither of every token's row, [n, hkv, 128] in channel order."""
    bits = SCHEMES[scheme][1]
    groups = 8 if bits == 8 else 16
    slot, head, grp = (slots.long().view(-1, 1, 1), torch.arange(hkv, device="cuda").view(1, -1, 1), torch.arange(groups, device="cuda").view(1, 1, -1))
    zero = torch.zeros_like(slot + head + grp)
    w = _philox(slot + zero, layer * 65536 + head + zero, grp + zero, row + zero, seed)
    n, mask = (4, 0xFF) if bits == 8 else (2, 0x3FF)
    step = 8 if bits == 8 else 16
    j = torch.stack([(w >> (step * i)) & mask for i in range(n)], dim=-1).flatten(-3)
    if scheme == "g32":      # drawn by storage position
        p = torch.arange(DIM, device="cuda")
        at = 16 * ((p >> 2) & 7) + 4 * (p >> 5) + (p & 3) if row == 0 else 16 * ((p >> 1) & 7) + 8 * (p & 1) + (p >> 4)
        j = torch.empty_like(j).index_copy_(-1, at, j)
    return (j.double() + 0.5) / 2**bits - 0.5


def _up(x):
    """x >= 0 rounded up to fp16."""
    h = x.half()
    h = torch.where(h.double() < x, (h.view(torch.int16) + 1).view(torch.float16), h)
    less = (h.view(torch.int16) - 1).clamp(min=0).view(torch.float16)
    return torch.where(less.double() >= x, less, h)


def _quantize(x, slots, layer, row, scheme, seed, bypass=None):
    """(reconstruction, scales) of rows x fp16 [n, hkv, 128]; bypass [hkv, 128]: channels stored exactly."""
    xd = x.double()
    if scheme == "fp8":
        return x.float().clamp(-448, 448).to(torch.float8_e4m3fn).double(), None
    keep = torch.ones(x.shape[1], DIM, device="cuda", dtype=torch.bool) if bypass is None else ~bypass
    a = torch.where(keep, x.abs(), 0)
    groups = 4 if scheme == "g32" else 1
    amax = a.view(*x.shape[:2], groups, DIM // groups).amax(-1).float()
    s = (amax / 126.5).half()
    s = torch.where((s == 0) & (amax > 0), torch.full_like(s, 2.0**-24), s)
    sd = s.double().repeat_interleave(DIM // groups, -1)
    xi = _xi(slots, layer, x.shape[1], row, scheme, seed)
    code = torch.where(sd > 0, xd / sd + xi, xi).round().clamp(-127, 127)
    return torch.where(keep, sd * (code - xi), xd), s


def _bands(r, rope):
    """Norms over the 8 bands of 8 RoPE pairs, [..., 8]."""
    sq = r.square()
    pair = sq[..., :64] + sq[..., 64:] if rope == "half" else sq.view(*sq.shape[:-1], 64, 2).sum(-1)
    return pair.view(*pair.shape[:-1], 8, 8).sum(-1).sqrt()


def _mask(pairs, rope):
    """[hkv, 128]: the bypassed channels."""
    b = torch.zeros(pairs.shape[0], DIM, dtype=torch.bool, device="cuda")
    a, c = (pairs, pairs + 64) if rope == "half" else (2 * pairs, 2 * pairs + 1)
    return b.scatter_(1, a.long(), True).scatter_(1, c.long(), True)


def _layout(case, pages, rows, slots, width):
    """rows [n, hkv, width] in a cache array [pages, hkv, 16, width]."""
    t = torch.zeros(pages, case["hkv"], PAGE, width, dtype=rows.dtype, device="cuda")
    t[(slots // PAGE).long(), :, (slots % PAGE).long()] = rows
    return t


def _cpu(x):
    return x.double().cpu()


def exact(case, seed):
    if case["kind"] == "select":
        return _exact_select(case, seed)
    return _exact_step(case, seed) if case["kind"] == "step" else _exact_write(case, seed)


def _exact_write(case, seed):
    scheme, rope, m = case.get("scheme", "g32"), case["rope"], case.get("m", 4 if case.get("scheme") == "g32" else 0)
    _, slots, pages = _tables([case["n_tok"]], case["n_tok"], seed)
    k, v = _kv(seed, 0, [case["n_tok"]], case["hkv"], rope)
    bypass = None
    if scheme == "g32":
        if case["kind"] == "calibrate":
            e = k.double().square().sum(0)
            e = e[:, :64] + e[:, 64:] if rope == "half" else e.view(-1, 64, 2).sum(-1)
            pairs = e.sort(dim=-1, descending=True, stable=True).indices[:, :m].sort(dim=-1).values
        else:
            pairs = _pairs(seed, 0, case["hkv"], m)
        bypass = _mask(pairs, rope)
    kr, ks = _quantize(k, slots, 0, 0, scheme, seed, bypass)
    w = _bands(kr - k.double(), rope)
    res = {"k_codes": None, "v_codes": None, "k_witness": _cpu(_layout(case, pages, w, slots, 8))}
    del kr, w
    vr, vs = _quantize(v, slots, 0, 1, scheme, seed)
    if ks is not None:
        width = ks.shape[-1]
        for name, s in (("k_scale", ks), ("v_scale", vs)):
            t = _layout(case, pages, s.double(), slots, width)
            res[name] = _cpu(t if scheme == "g32" else t[..., 0])
    if case.get("value"):
        vw = torch.stack([(vr - v.double()).norm(dim=-1), v.double().norm(dim=-1)], dim=-1)
        res["v_witness"] = _cpu(_layout(case, pages, vw, slots, 2))
    return res


def _exact_step(case, seed):
    lens = _ctx_lens(case, seed)
    bt, slots, _ = _tables(lens, case["ctx_hi"], seed)
    scheme, rope, hkv, hq, m = case["scheme"], case["rope"], case["hkv"], case["hq"], case["m"]
    G, variant = hq // hkv, case["variant"]
    rows = {n: [] for n in ("out", "raw", "b_raw", "vt", "vmax", "contrib")}
    for layer in range(case["layers"]):
        K, V = _kv(seed, layer, lens, hkv, rope)
        q_all = _queries(case, seed, layer, lens)
        pairs = _pairs(seed, layer, hkv, m) if scheme == "g32" and m else None
        bypass = _mask(pairs, rope) if pairs is not None else None
        at = 0
        for b, S in enumerate(lens):
            k, v, sl = K[at:at + S], V[at:at + S], slots[at:at + S]
            at += S
            kr, ks = _quantize(k, sl, layer, 0, scheme, seed, bypass)
            vr, _ = _quantize(v, sl, layer, 1, scheme, seed)
            w = _up(_bands(kr - k.double(), rope)).double()
            q = q_all[b].double().view(hkv, G, DIM)
            y = torch.einsum("hgd,thd->hgt", q, kr) / math.sqrt(DIM)
            p = torch.softmax(y, dim=-1)
            c = torch.einsum("hgb,thb->hgt", _bands(q, rope), w) / math.sqrt(DIM)
            t = p * torch.expm1(c)
            D = t.sum(-1)
            rows["out"].append(torch.einsum("hgt,thd->hgd", p, vr).reshape(hq, DIM))
            rows["raw"].append((0.5 * D * (D + 2)).reshape(hq))
            if variant == "tier_b":
                lg = 2.0 * math.log(2.0 * S / DELTA) / (12 * DIM)
                qz = q if bypass is None else torch.where(bypass[:, None], 0.0, q)
                ng = ks.shape[-1]
                q2 = qz.square().view(hkv, G, ng, DIM // ng).sum(-1)
                u = torch.sqrt(lg * torch.einsum("hgn,thn->hgt", q2, ks.double().square()))
                D = (p * torch.expm1(u)).sum(-1)
                rows["b_raw"].append((0.5 * D * (D + 2)).reshape(hq))
            if variant == "value":
                rho, nv = _up((vr - v.double()).norm(dim=-1)).double(), _up(v.double().norm(dim=-1)).double()
                rows["vt"].append(torch.einsum("hgt,th->hg", p, rho).reshape(hq))
                rows["vmax"].append(nv.amax(0).repeat_interleave(G))
            if variant == "repair":
                pad = torch.zeros(hkv, G, bt.shape[1] * PAGE, dtype=torch.float64, device="cuda")
                pad[..., :S] = t
                rows["contrib"].append(pad.view(hq, bt.shape[1], PAGE).sum(-1))
                del pad
    shape = (case["layers"], case["batch"], hq)
    got = {n: torch.stack(x).view(*shape, *x[0].shape[1:]) for n, x in rows.items() if x}
    res = {"out": _cpu(got["out"]), "meter_raw": _cpu(got["raw"]), "meter": _cpu(got["raw"].clamp(max=1.0))}
    if variant == "tier_b":
        res["meter_b_raw"], res["meter_b"] = _cpu(got["b_raw"]), _cpu(got["b_raw"].clamp(max=1.0))
    if variant == "value":
        res["value_term"], res["v_max"] = _cpu(got["vt"]), _cpu(got["vmax"])
        res["out_bound"] = _cpu(2 * got["raw"].clamp(max=1.0) * got["vmax"] + got["vt"])
    if variant == "repair":
        res["contrib"] = _cpu(got["contrib"].flatten(0, 1))
    return res


def _exact_select(case, seed):
    terms, norm, lens = _terms(case, seed)
    c = terms[..., 1].double() * torch.exp2(terms[..., 0].double() - norm[..., :1].double()) / norm[..., 1:].double()
    n = (lens.long() + PAGE - 1) // PAGE
    c = torch.where(torch.arange(case["pages"], device="cuda") < n[:, None, None], c, 0.0)
    ranked = c.sort(-1, descending=True).values
    rest = torch.cat([ranked.flip(-1).cumsum(-1).flip(-1), torch.zeros_like(ranked[..., :1])], dim=-1)   # R_k
    ok = 0.5 * rest * (rest + 2) <= case["tau"]
    k = ok.int().argmax(-1, keepdim=True)
    return {"contrib": _cpu(c), "d_after": _cpu(rest.gather(-1, k)[..., 0]), "pages": None, "n_repair": None}
