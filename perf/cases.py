"""The work a user of this framework has it do, as measurable cases.

A serving program uses the library in three ways.  Prefill: every attention layer of a prompt is
scored, its token set selected, attention run over the set and the kept keys / values compacted
(three calls per layer, or their batched forms for several prompts of one shape).  Decode: one
token per request goes through the layers, each layer's step appending to and reading that layer's
kept cache (contiguous, paged or mixed-precision).  Host: a layer and its first decode step from
and to pinned host buffers in one call.

Every buffer such a program keeps between calls (outputs, caches, workspaces, the descriptor, the
status word) is made once in prepare().  A decode pass appends one row per request; the lengths are
put back at the start of the pass (one small copy on the device), so that every pass does the same
work and the caches never run full.
"""
import ctypes
import math

import torch

import paper_2410_08584_b200 as z

DTYPES = {"bf16": torch.bfloat16, "f16": torch.float16, "f32": torch.float32}
CODES = {"bf16": z.ZIPVL_BF16, "f16": z.ZIPVL_F16, "f32": z.ZIPVL_F32}


def _prefill(L, Hq, Hkv, d, dtype, tau, recipe="heavy", frac=0.10, scale=3.0, probes=128, n_seq=1):
    return dict(kind="prefill", L=L, Hq=Hq, Hkv=Hkv, d=d, dtype=dtype, tau=tau, recipe=recipe, frac=frac,
                scale=scale, probes=probes, n_seq=n_seq)


def _decode(batch, lo, hi, Hq, Hkv, d, dtype, layers, page_rows=0):
    return dict(kind="decode", batch=batch, lo=lo, hi=hi, Hq=Hq, Hkv=Hkv, d=d, dtype=dtype, layers=layers,
                page_rows=page_rows)


def listed():
    cases = [
        # The smallest prefill call: the tiny single layer (1024 tokens, 4 heads of 64, fp32, the last
        # 64 rows as probes, 32 sinks).  Launches, host work and latency count.
        ("tiny_layer_fp32", _prefill(1024, 4, 4, 64, "f32", 0.95, "sinks", 32 / 1024, 4.0, probes=64)),
        # Four short image prompts of one (odd) length prefilled together in half precision: one
        # image tile of 576 tokens and some text, through the batched calls.
        ("short_prompts_batch_fp16", _prefill(709, 32, 32, 128, "f16", 0.97, n_seq=4)),
        # Grouped-query layer of a small model (14 query heads on 2 kv heads of 64 channels), a
        # prompt of a few images whose length is a multiple of nothing.
        ("gqa_d64_layer", _prefill(5003, 14, 2, 64, "bf16", 0.97, frac=0.2, scale=2.5)),
        # The ordinary layer: LLaVA-Next-7B-shaped any-resolution prompt (the default workload of bench.py).
        ("llava_next_7b_layer", _prefill(2944, 32, 32, 128, "bf16", 0.97)),
        # Long video, grouped queries: 128 frames of 144 tokens, frame-correlated keys.
        ("long_video_layer", _prefill(18432, 28, 4, 128, "bf16", 0.95, "video", 0.0, 0.2)),
        # The largest: a 13B-shaped layer at 32K tokens.
        ("long_context_layer", _prefill(32768, 40, 40, 128, "bf16", 0.97)),
        # Interactive decoding: one request on the cache kept of the ordinary prompt, one token
        # through eight layers.
        ("decode_one_request", _decode(1, 2307, 2307, 32, 32, 128, "bf16", 8)),
        # Batched decoding on compacted caches (contexts of 4K to 32K tokens before compaction).
        ("decode_batch", _decode(16, 3011, 24317, 32, 32, 128, "bf16", 1)),
        # Batched decoding of the grouped-query video model over a paged cache in half precision.
        ("decode_gqa_paged_fp16", _decode(16, 6001, 29989, 28, 4, 128, "f16", 4, page_rows=64)),
        # Mixed-precision cache, encode: the ordinary layer's keys / values to 4 and 2 bits.
        ("quantize_cache", dict(kind="quantize", L=2944, H=32, d=128, dtype="bf16", keep=0.77)),
        # Mixed-precision cache, decode: six requests, one token through four layers.
        ("decode_quantized", dict(kind="decode_quant", batch=6, lo=1409, hi=5903, Hq=32, Hkv=32, d=128,
                                  dtype="bf16", layers=4, keep=0.77)),
        # The ordinary layer and its first decode step from and to pinned host memory (the
        # end-to-end call that bench.py times).
        ("host_layer_step", dict(kind="host", L=2944, Hq=32, Hkv=32, d=128, dtype="bf16", tau=0.97)),
    ]
    return [dict(c, name=n) for n, c in cases]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["tiny", "prefill", "prefill", "prefill", "batch", "decode", "decode", "paged", "quantize",
                       "decode_quant", "host"])
    # head shapes of the configurations, the tests and the benchmark: (query heads, kv heads, channels)
    Hq, Hkv, d = rng.choice([(32, 32, 128), (40, 40, 128), (28, 4, 128), (14, 2, 64), (12, 4, 96), (16, 16, 64)])
    dtype = rng.choice(["bf16", "bf16", "f16"])
    tau = rng.choice([0.95, 0.97, 0.99])
    frac, scale = round(rng.uniform(0.02, 0.3), 3), round(rng.uniform(2.0, 3.5), 2)
    if kind == "tiny":
        H, dd = rng.choice([(2, 64), (4, 64), (4, 128)])
        L = _logint(rng, 200, 1400)
        return _prefill(L, H, H, dd, "f32", tau, "sinks", max(1, L // 32) / L, 4.0, probes=64)
    if kind == "prefill":
        L = _logint(rng, 500, 23500)
        if Hkv == 4 and d == 128 and rng.random() < 0.5:
            return _prefill(L // 144 * 144 + 144, Hq, Hkv, d, dtype, tau, "video", 0.0, 0.2)
        return _prefill(L, Hq, Hkv, d, dtype, tau, "heavy", frac, scale)
    if kind == "batch":
        return _prefill(_logint(rng, 250, 3000), Hq, Hkv, d, dtype, tau, "heavy", frac, scale, n_seq=rng.randint(2, 8))
    if kind in ("decode", "paged"):
        batch = _logint(rng, 1, 64)
        hi = _logint(rng, 500, 30000)
        lo = max(1, int(hi * rng.uniform(0.1, 1.0)))
        # no more rows than the listed batch holds
        rows = min(batch * (lo + hi) // 2, 450_000 * 4096 // (Hkv * d) // 2)
        batch = max(1, min(batch, rows * 2 // (lo + hi)))
        layers = rng.randint(1, max(1, min(8, 900_000_000 // (rows * Hkv * d))))
        return _decode(batch, lo, hi, Hq, Hkv, d, dtype, layers, rng.choice([16, 64, 256]) if kind == "paged" else 0)
    H, d = rng.choice([(32, 128), (40, 128), (16, 64)])
    if kind == "quantize":
        return dict(kind="quantize", L=_logint(rng, 500, 20000), H=H, d=d, dtype=dtype, keep=round(rng.uniform(0.3, 0.9), 3))
    if kind == "decode_quant":
        hi = _logint(rng, 500, 12000)
        return dict(kind="decode_quant", batch=_logint(rng, 1, 24), lo=max(1, int(hi * rng.uniform(0.2, 1.0))), hi=hi,
                    Hq=H, Hkv=H // rng.choice([1, 1, 2, 4]), d=d, dtype=dtype, layers=rng.randint(1, 4),
                    keep=round(rng.uniform(0.3, 0.9), 3))
    return dict(kind="host", L=_logint(rng, 500, 5000), Hq=H, Hkv=H, d=d, dtype=dtype, tau=tau)


# ---- inputs ------------------------------------------------------------------------------------

def _lens(case):
    """Rows per request: evenly spread over [lo, hi], in an order that is not sorted."""
    n, lo, hi = case["batch"], case["lo"], case["hi"]
    order = [(i * 7 + 3) % n if n % 7 else i for i in range(n)]
    return [hi if n == 1 else lo + (hi - lo) * o // (n - 1) for o in order]


def _randn(shape, g, dtype):
    """N(0,1) in fp32, rounded once to the storage type; in pieces, so that large caches do not need
    four times their memory for a moment."""
    out = torch.empty(shape, dtype=dtype, device="cuda")
    for piece in out.view(-1).split(1 << 28):
        piece.copy_(torch.randn(piece.shape, generator=g, device="cuda"))
    return out


def _probe_positions(L, n_recent, n_random, g):
    if L <= n_recent + n_random:
        return torch.arange(L, dtype=torch.int32, device="cuda")
    recent = torch.arange(L - n_recent, L, device="cuda")
    if n_random:
        recent = torch.cat([torch.randperm(L - n_recent, generator=g, device="cuda")[:n_random], recent])
    return torch.sort(recent).values.to(torch.int32)


def _layer_inputs(case, g):
    """Q, K, V of one sequence by the recipes of paper_2410_08584_b200/workloads.py, on the device."""
    L, Hq, Hkv, d, dt = case["L"], case["Hq"], case["Hkv"], case["d"], DTYPES[case["dtype"]]
    r = lambda *s: torch.randn(s, generator=g, device="cuda")
    recipe = case.get("recipe", "heavy")
    q = r(L, Hq, d).to(dt)
    if recipe == "video":
        def frames():
            x = r(L // 144, 144, Hkv, d)
            x[1:] *= case["scale"]
            return torch.cumsum(x, dim=0).reshape(L, Hkv, d).to(dt)
        return q, frames(), frames()
    k, v = r(L, Hkv, d), r(L, Hkv, d).to(dt)
    frac, scale = case.get("frac", 0.10), case.get("scale", 3.0)
    if recipe == "sinks":
        big = torch.zeros(L, dtype=torch.bool, device="cuda")
        n = max(1, round(frac * L))
        big[torch.randperm(L - 1, generator=g, device="cuda")[:n - 1] + 1] = True
        big[0] = True
    else:
        big = torch.rand(L, generator=g, device="cuda") < frac
        big[L - min(64, L // 2):] = False
    k[big] *= scale
    return q, k.to(dt), v


def _status():
    return torch.zeros(1, dtype=torch.int32, device="cuda")


def _decode_ws(case, max_len):
    lay = z.zipvl_layer(max_len, case["Hq"], case["Hkv"], case["d"], CODES[case["dtype"]], 0, 0, 0, 0.0, 0)
    return z.workspace(z.zipvl_workspace_bytes(z.OP_DECODE, lay, 0, case["batch"]), "cuda")


def _new_tokens(case, g):
    dt, n, B, d = DTYPES[case["dtype"]], case["layers"], case["batch"], case["d"]
    return _randn((n, B, case["Hq"], d), g, dt), _randn((n, B, case["Hkv"], d), g, dt), _randn((n, B, case["Hkv"], d), g, dt)


def _prepare_prefill(case, g):
    n, L, P = case["n_seq"], case["L"], case["probes"]
    seqs = [_layer_inputs(case, g) for _ in range(n)]
    probe = [_probe_positions(L, 64, P - 64, g) for _ in range(n)]
    s = dict(tau=case["tau"], L=L, status=_status())
    s["q"], s["k"], s["v"] = (torch.stack(t) if n > 1 else t[0] for t in zip(*seqs))
    s["probe"] = torch.stack(probe) if n > 1 else probe[0]
    lead = (n, L) if n > 1 else (L,)
    s["acc"] = torch.empty(lead, dtype=torch.float32, device="cuda")
    s["norm"], s["idx"] = torch.empty_like(s["acc"]), torch.empty(lead, dtype=torch.int32, device="cuda")
    s["count"], s["len"] = (torch.zeros(n, dtype=torch.int32, device="cuda") for _ in range(2))
    s["out"], s["kc"], s["vc"] = torch.empty_like(s["q"]), torch.zeros_like(s["k"]), torch.zeros_like(s["v"])
    lay = z.zipvl_layer(L, case["Hq"], case["Hkv"], case["d"], CODES[case["dtype"]], 0, 0, 0, 0.0, 0)
    s["desc"] = lay
    score_ws = z.load().zipvl_workspace_bytes_batch(z.OP_SCORE, ctypes.byref(lay), s["probe"].shape[-1], n)
    s["ws_score"] = z.workspace(score_ws, "cuda")
    s["ws_select"] = z.workspace(z.zipvl_workspace_bytes(z.OP_SELECT, lay), "cuda")
    s["ws_prefill"] = z.workspace(z.zipvl_workspace_bytes(z.OP_SPARSE_PREFILL, lay), "cuda")
    return s


def _run_prefill(s):
    if s["q"].dim() == 4:
        z.zipvl_score_batch(s["q"], s["k"], s["probe"], acc=s["acc"], norm=s["norm"], ws=s["ws_score"], status=s["status"])
        z.zipvl_select_batch(s["acc"], s["norm"], s["tau"], k_out=s["count"], idx=s["idx"], ws=s["ws_select"],
                             status=s["status"])
        z.zipvl_sparse_prefill_batch(s["q"], s["k"], s["v"], s["idx"], s["count"], s["L"], s["kc"], s["vc"], s["L"],
                                     out=s["out"], len_out=s["len"], ws=s["ws_prefill"], status=s["status"])
    else:
        z.zipvl_score(s["desc"], s["q"], s["k"], s["probe"], acc=s["acc"], norm=s["norm"], ws=s["ws_score"],
                      status=s["status"])
        z.zipvl_select(s["acc"], s["norm"], s["tau"], k_out=s["count"], idx=s["idx"], ws=s["ws_select"],
                       status=s["status"])
        z.zipvl_sparse_prefill_compact(s["desc"], s["q"], s["k"], s["v"], s["idx"], s["count"], s["L"], s["kc"], s["vc"],
                                       s["L"], out=s["out"], len_out=s["len"], ws=s["ws_prefill"], status=s["status"])
    return {m: s[m] for m in ("acc", "norm", "count", "idx", "out", "kc", "vc", "len", "status")}


def _prepare_decode(case, g):
    n, B, Hkv, d, dt = case["layers"], case["batch"], case["Hkv"], case["d"], DTYPES[case["dtype"]]
    lens, page = _lens(case), case["page_rows"]
    s = dict(desc=z.zipvl_decode_desc(B, case["Hq"], Hkv, d, CODES[case["dtype"]], 0.0), max_len=max(lens) + 1, status=_status())
    # room for the tokens still to come, in whole pages where the cache is paged
    caps = [(m + 16 + page - 1) // page * page if page else m + 16 for m in lens]
    if page:
        pages = [c // page for c in caps]
        width, total = max(pages), sum(pages)
        perm = torch.randperm(total, generator=g, device="cuda").to(torch.int32)
        s["table"] = torch.zeros(B, width, dtype=torch.int32, device="cuda")
        at = 0
        for b, p in enumerate(pages):
            s["table"][b, :p] = perm[at:at + p]
            at += p
        s["kc"], s["vc"] = (_randn((n, total, page, Hkv, d), g, dt) for _ in range(2))
    else:
        off = [sum(caps[:b]) * Hkv * d for b in range(B)]
        s["off"] = torch.tensor(off, dtype=torch.int64, device="cuda")
        s["kc"], s["vc"] = (_randn((n, sum(caps), Hkv, d), g, dt) for _ in range(2))
    s["cap"] = torch.tensor(caps, dtype=torch.int32, device="cuda")
    s["lens0"] = torch.tensor([lens] * n, dtype=torch.int32, device="cuda")
    s["lens"] = s["lens0"].clone()
    s["q"], s["kn"], s["vn"] = _new_tokens(case, g)
    s["out"] = torch.empty_like(s["q"])
    s["ws"] = _decode_ws(case, s["max_len"])
    # what the layers of such a program hold: their own slices
    s["layers"] = [tuple(s[m][i] for m in ("q", "kn", "vn", "kc", "vc", "lens", "out")) for i in range(n)]
    return s


def _run_decode(s):
    s["lens"].copy_(s["lens0"])
    for q, kn, vn, kc, vc, lens, out in s["layers"]:
        if "table" in s:
            z.zipvl_decode_paged(s["desc"], q, kn, vn, kc, vc, s["table"], s["cap"], lens, s["max_len"], out=out, ws=s["ws"],
                                 status=s["status"])
        else:
            z.zipvl_decode(s["desc"], q, kn, vn, kc, vc, s["off"], s["cap"], lens, s["max_len"], out=out, ws=s["ws"],
                           status=s["status"])
    return {m: s[m] for m in ("out", "kc", "vc", "lens", "status")}


def _token_set(L, keep, g):
    """A random ascending token set of about keep * L tokens and its size, as zipvl_select writes them."""
    n = max(1, int(keep * L))
    idx = torch.full((L,), -1, dtype=torch.int32, device="cuda")
    idx[:n] = torch.sort(torch.randperm(L, generator=g, device="cuda")[:n]).values.to(torch.int32)
    return idx, torch.tensor([n], dtype=torch.int32, device="cuda"), n


def _prepare_quantize(case, g):
    L, H, d, dt = case["L"], case["H"], case["d"], DTYPES[case["dtype"]]
    k, v = _randn((L, H, d), g, dt), _randn((L, H, d), g, dt)
    idx, count, n = _token_set(L, case["keep"], g)
    # room for decoded tokens in the 4-bit block
    cache = z.QuantCache(L, H, d, dt, "cuda", cap_hi=n + 16, cap_lo=L - n + 1)
    return dict(desc=z.layer_desc(k, k), k=k, v=v, idx=idx, count=count, L=L, cache=cache, status=_status())


def _run_quantize(s):
    z.zipvl_quantize_kv(s["desc"], s["k"], s["v"], s["idx"], s["count"], s["L"], s["cache"], status=s["status"])
    out = {m: getattr(s["cache"], m) for m in ("k_hi", "v_hi", "p_hi", "k_lo", "v_lo", "p_lo", "lens")}
    return dict(out, status=s["status"])


def _prepare_decode_quant(case, g):
    n, B, Hkv, d, dt = case["layers"], case["batch"], case["Hkv"], case["d"], DTYPES[case["dtype"]]
    lens = _lens(case)
    s = dict(desc=z.zipvl_decode_desc(B, case["Hq"], Hkv, d, CODES[case["dtype"]], 0.0), max_len=max(lens) + 1, status=_status())
    # the blocks of all layers and requests are slices of one pool, each as large as the largest needs
    sets = [_token_set(L, case["keep"], g) for L in lens]
    hi, lo = max(m for _, _, m in sets) + 16, max(L - m for L, (_, _, m) in zip(lens, sets)) + 1
    shapes = {"k_hi": (hi, Hkv, d // 2), "v_hi": (hi, Hkv, d // 2), "k_lo": (lo, Hkv, d // 4), "v_lo": (lo, Hkv, d // 4)}
    s["pool"] = {m: torch.zeros((n, B) + t, dtype=torch.uint8, device="cuda") for m, t in shapes.items()}
    s["pool"].update({m: torch.zeros((n, B, r, Hkv, 4), dtype=dt, device="cuda") for m, r in (("p_hi", hi), ("p_lo", lo))})
    s["pool"]["lens"] = torch.zeros(n, B, 2, dtype=torch.int32, device="cuda")
    s["tables"] = []
    for i in range(n):
        row = []
        for b, L in enumerate(lens):
            k, v = _randn((L, Hkv, d), g, dt), _randn((L, Hkv, d), g, dt)
            idx, count, _ = sets[b]
            c = z.QuantCache(L, Hkv, d, dt, "cuda", cap_hi=1, cap_lo=1)
            c.cap_hi, c.cap_lo = hi, lo
            for m, t in s["pool"].items():
                setattr(c, m, t[i, b])
            z.zipvl_quantize_kv(z.layer_desc(k, k), k, v, idx, count, L, c, status=s["status"])
            row.append(c)
        s["tables"].append(z.quant_cache_table(row, "cuda"))
    s["lens"] = s["pool"]["lens"]
    s["lens0"] = s["lens"].clone()
    s["q"], s["kn"], s["vn"] = _new_tokens(case, g)
    s["out"] = torch.empty_like(s["q"])
    s["ws"] = _decode_ws(case, s["max_len"])
    s["layers"] = [(s["q"][i], s["kn"][i], s["vn"][i], s["tables"][i], s["out"][i]) for i in range(n)]
    return s


def _run_decode_quant(s):
    s["lens"].copy_(s["lens0"])
    for q, kn, vn, table, out in s["layers"]:
        z.zipvl_decode_quant_batch(s["desc"], q, kn, vn, table, s["max_len"], out=out, ws=s["ws"], status=s["status"])
    return dict(s["pool"], out=s["out"], status=s["status"])


def _prepare_host(case, g):
    q, k, v = (t.cpu().pin_memory() for t in _layer_inputs(case, g))
    dt, d = q.dtype, case["d"]
    s = dict(desc=z.layer_desc(q, k), tau=case["tau"], q=q, k=k, v=v)
    s["probe"] = _probe_positions(case["L"], 64, 64, g).cpu().pin_memory()
    s["qn"], s["kn"], s["vn"] = (_randn((1, h, d), g, dt).cpu().pin_memory() for h in (case["Hq"], case["Hkv"], case["Hkv"]))
    s["out"], s["kc"], s["vc"], s["dec"] = (torch.zeros_like(t).pin_memory() for t in (q, k, v, s["qn"]))
    s["idx"] = torch.zeros(case["L"], dtype=torch.int32).pin_memory()
    return s


def _run_host(s):
    return z.zipvl_layer_step_host(s["desc"], s["q"], s["k"], s["v"], s["probe"], s["tau"], s["qn"], s["kn"], s["vn"],
                                   out=s["out"], k_cache=s["kc"], v_cache=s["vc"], idx=s["idx"], decode_out=s["dec"])


PREPARE = {"prefill": _prepare_prefill, "decode": _prepare_decode, "quantize": _prepare_quantize,
           "decode_quant": _prepare_decode_quant, "host": _prepare_host}
RUN = {"prefill": _run_prefill, "decode": _run_decode, "quantize": _run_quantize,
       "decode_quant": _run_decode_quant, "host": _run_host}


def prepare(case, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return dict(PREPARE[case["kind"]](case, g), run=RUN[case["kind"]])


def run(state):
    return state["run"](state)


# ---- what a pass cannot do without ----------------------------------------------------------------

def _kept(case):
    """Tokens that the selection keeps, about: keys scaled by s carry exp(s^2 / 2) of the score of
    a plain one, as far as a row's few thousand samples reach; the rest of the share comes from plain tokens."""
    if case.get("recipe") == "video":
        return 0.93 * case["L"]
    f, s = case.get("frac", 0.10), case.get("scale", 3.0)
    heavy = f * math.exp(min(s * s / 2, 5.0))
    plain = (1 - f) * math.exp(0.5)
    share = heavy / (heavy + plain)
    tau = case["tau"]
    return case["L"] * (f * tau / share if tau < share else f + (1 - f) * (tau - share) / (1 - share))


def _row(case, H):
    return H * case["d"] * (4 if case["dtype"] == "f32" else 2)


def _prefill_work(case):
    """Scores: one product of the probe rows with all keys.  Attention: the kept tokens' causal half.
    Bytes: q, k, v read once (queries and values of the kept tokens), scores, index, padded output and
    caches written once."""
    L, Hq, Hkv, d, n, P = case["L"], case["Hq"], case["Hkv"], case["d"], case.get("n_seq", 1), case.get("probes", 128)
    k = _kept(case)
    flops = 2.0 * P * L * Hq * d + 4.0 * d * Hq * k * (k + 1) / 2
    bytes_ = (k + P) * _row(case, Hq) + (L + k) * _row(case, Hkv) + L * _row(case, Hq) + 2 * k * _row(case, Hkv) + 12.0 * L
    return {"bytes": n * bytes_, "flops": n * flops}


def work(case):
    kind = case["kind"]
    if kind == "prefill":
        return _prefill_work(case)
    if kind == "decode":
        rows = sum(_lens(case)) + case["batch"]
        per = 2 * rows * _row(case, case["Hkv"]) + case["batch"] * 2 * (_row(case, case["Hq"]) + _row(case, case["Hkv"]))
        return {"bytes": case["layers"] * per, "flops": case["layers"] * 4.0 * rows * case["Hq"] * case["d"]}
    if kind == "quantize":
        n = max(1, int(case["keep"] * case["L"]))
        m = case["L"] - n
        codes = 2 * case["H"] * case["d"] * (n / 2 + m / 4) + 8.0 * case["H"] * case["L"]
        return {"bytes": 2 * case["L"] * _row(case, case["H"]) + codes + 4 * n, "flops": 0}
    if kind == "decode_quant":
        total, rows = 0.0, 0
        for L in _lens(case):
            n = max(1, int(case["keep"] * L)) + 1
            m = L + 1 - n
            total += case["Hkv"] * (2 * case["d"] * (n / 2 + m / 4) + 8.0 * (n + m))
            rows += n + m
        total += case["batch"] * 2 * (_row(case, case["Hq"]) + _row(case, case["Hkv"]))
        return {"bytes": case["layers"] * total, "flops": case["layers"] * 4.0 * rows * case["Hq"] * case["d"]}
    # host: the layer's work, then a decode step on the cache it left; what crosses the bus is counted once
    w = _prefill_work(dict(case, n_seq=1))
    rows = _kept(case) + 1
    return {"bytes": w["bytes"] + 2 * rows * _row(case, case["Hkv"]), "flops": w["flops"] + 4.0 * rows * case["Hq"] * case["d"]}


def tolerance(case):
    """Codes are whole numbers decided by correctly rounded operations.  Elsewhere: probabilities and outputs
    are rounded to the storage type (8 bits of mantissa for bf16, 11 for fp16), sums are in fp32;
    the fp32 path differs by the order of its sums and the last bits of exp2.  The token set and its
    size are whole numbers and come out the same."""
    if case["kind"] == "quantize":
        return "exact"
    return {"bf16": {"rel": 1e-2, "max": 0.1}, "f16": {"rel": 2e-3, "max": 0.02}, "f32": {"rel": 2e-5, "max": 1e-3}}[case["dtype"]]
