"""The calls whose speed counts: what a DSA-style model or serving engine has the indexer do.

A case is one call of a public entry point of paper_2607_24593_b200.binding on synthetic indexer
activations (the generator of paper_2607_24593_b200/inputs.py, drawn on the GPU), 64 heads x 128, with
the budgets of the paper's Implementation paragraph (k = 2048, c = 4096, g = 4) or those of this
repository's small configurations.  Index rows are sets in unspecified order, so `run` ends with the
step that makes them a mask over the keys, as a masked attention takes it: booleans where that is
small, a bit per key packed into 32-bit words otherwise.
"""
import math
import random

import torch

from paper_2607_24593_b200 import binding as pv
from paper_2607_24593_b200 import inputs

H, D = 64, 128
MODES = {"refine": pv.REFINE, "reuse": pv.REUSE}
MASK_MAX = 1 << 30          # rows x keys up to which the mask is of booleans


def _prefill(name, L, dtype, g, c, k, mode, row0=0, W=0):
    return {"name": name, "kind": "prefill", "L": L, "dtype": dtype, "g": g, "c": c, "k": k, "mode": mode,
            "row0": row0, "W": W}


def _decode(name, B, lo, hi, dtype, g, c, k, mode, paged=False, W=0):
    return {"name": name, "kind": "decode", "B": B, "lo": lo, "hi": hi, "dtype": dtype, "g": g, "c": c, "k": k,
            "mode": mode, "paged": paged, "W": W}


def listed():
    return [
        # a short prompt, the repository's smallest configuration: launches and latency count
        _prefill("prefill_2k_bf16", 2048, "bf16", 4, 512, 256, "refine"),
        # a prompt of ordinary length whose size divides nothing, larger groups
        _prefill("prefill_5003_fp8_g8", 5003, "fp8", 8, 2048, 1024, "refine"),
        # a long document in either operand type (the second one ragged)
        _prefill("prefill_32k_bf16", 32768, "bf16", 4, 4096, 2048, "refine"),
        _prefill("prefill_30001_fp8", 30001, "fp8", 4, 4096, 2048, "refine"),
        # the variant without a re-score
        _prefill("prefill_64k_fp8_reuse", 65536, "fp8", 4, 4096, 2048, "reuse"),
        # the headline: one whole 128K request
        _prefill("prefill_128k_fp8", 131072, "fp8", 4, 4096, 2048, "refine"),
        # chunked prefill: a serving engine's 8192-token chunk at the end of a 256K prompt
        _prefill("chunk_8k_of_256k_fp8", 262144, "fp8", 4, 4096, 2048, "refine", row0=253952),
        # continuous batching: a batch of short prompts packed back to back
        {"name": "varlen_12_fp8", "kind": "varlen", "lens": "644,3000,128,1896,5212,412,2364,900,4096,256,1500,2777",
         "dtype": "fp8", "g": 4, "c": 1024, "k": 512, "mode": "refine"},
        # the dense indexer (short prompts and layers that keep it)
        {"name": "dense_16k_fp8", "kind": "dense", "L": 16384, "dtype": "fp8", "k": 2048},
        # decode steps: a few short contexts, a long-context batch, a mixed batch on a paged cache
        _decode("decode_4x3k-9k_bf16", 4, 3000, 9000, "bf16", 2, 2048, 1024, "refine"),
        _decode("decode_32x64k-128k_fp8", 32, 65536, 131072, "fp8", 2, 4096, 2048, "refine"),
        _decode("decode_paged_48x4k-48k_fp8_w4", 48, 4500, 49000, "fp8", 4, 4096, 2048, "refine", paged=True, W=4),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw(rng):
    kind = rng.choice(["prefill", "prefill", "prefill", "varlen", "dense", "decode", "decode", "decode"])
    dtype = rng.choice(["fp8", "fp8", "bf16"])
    mode = rng.choice(["refine", "refine", "reuse"])
    k = rng.choice([256, 512, 1024, 2048, 2048, 2048])
    c = rng.choice([2 * k, 2 * k, 2 * k, 3 * k // 2, 3 * k])
    if kind == "prefill":
        g = rng.choice([2, 4, 4, 4, 8, 16])
        L = _log_int(rng, 1500, 262144 if dtype == "fp8" else 65536)
        row0 = (L * rng.randrange(1, 8) // 8) // g * g if L > 16384 and rng.random() < 0.4 else 0
        return _prefill("", L, dtype, g, c, k, mode, row0, rng.choice([0, 0, 0, 4]))
    if kind == "varlen":
        lens = [_log_int(rng, 100, 16384) // 4 * 4 for _ in range(rng.randrange(2, 17))]
        lens[-1] += rng.randrange(4)
        return {"kind": "varlen", "lens": ",".join(map(str, lens)), "dtype": dtype, "g": rng.choice([2, 4, 4, 8]), "c": c,
                "k": k, "mode": mode}
    if kind == "dense":
        return {"kind": "dense", "L": _log_int(rng, 1000, 49152), "dtype": dtype, "k": k}
    B = _log_int(rng, 1, 96)
    hi = _log_int(rng, 2500, 200000)
    paged = rng.random() < 0.4
    g = rng.choice([1, 2, 2, 4])
    W = 4 if mode == "refine" and rng.random() < 0.25 else 0
    return _decode("", B, max(hi // rng.choice([1, 2, 8]), 1000), hi, dtype, g, c, k, mode, paged, W)


def draw(rng):
    """Sizes over the whole range of the listed cases, odd ones among them, none costlier than the largest."""
    most = work(next(x for x in listed() if x["name"] == "prefill_128k_fp8"))
    while True:
        case = _draw(rng)
        case.pop("name", None)
        w = work(case)
        scale = 2 if case["dtype"] == "bf16" else 1
        longest = max(_lens(case)) if case["kind"] == "varlen" else case.get("L", case.get("lo"))
        if w["flops"] * scale <= most["flops"] and w["bytes"] <= most["bytes"] and _out_rows(case) * case["k"] <= 1 << 28 \
                and longest > case["k"] * 5 // 4:            # (with fewer keys than k there is nothing to select)
            return case


# ---------------------------------------------------------------------------------------- inputs

def _lens(case):
    return [int(v) for v in case["lens"].split(",")]


def _visible(case):
    """Visible prefix lengths of a decode batch: part of the case, not of its inputs."""
    r = random.Random(case["B"] * 1000003 + case["lo"] * 1009 + case["hi"])
    return [r.randint(case["lo"], case["hi"]) for _ in range(case["B"])]


def _keys(n, gen):
    z = torch.randn((n, D), device="cuda", generator=gen) / math.sqrt(D)
    u = torch.randn(D, device="cuda", generator=gen)
    hit = torch.rand(n, device="cuda", generator=gen) < inputs.OUTLIER_P
    return (z + hit[:, None] * (inputs.OUTLIER_GAIN * u / u.norm())).to(torch.bfloat16)


def _queries(n, gen, dtype):
    """AR(1) along the positions, per head and channel, after a run-in; eight heads at a time."""
    codes, scales = [], []
    for _ in range(0, H, 8):
        x = torch.randn((n + 128, 8 * D), device="cuda", generator=gen) / math.sqrt(D)
        step, f = 1, inputs.RHO
        while step < 128:                    # sums of 2, 4, ... 128 terms: rho^128 ~ 1e-6
            x[step:] += f * x[:-step].clone()
            step, f = 2 * step, f * f
        q = x[128:].to(torch.bfloat16).view(n, 8, D)
        if dtype == "fp8":
            q, s = inputs.quantize_e4m3(q)
            scales.append(s)
            q = q.view(torch.uint8)
        codes.append(q)
    q = torch.cat(codes, 1)
    return (q.view(torch.float8_e4m3fn), torch.cat(scales, 1).contiguous()) if dtype == "fp8" else (q, None)


def _stored(keys, dtype):
    return inputs.quantize_e4m3(keys) if dtype == "fp8" else (keys, None)


def _gates(n, gen):
    return torch.randn((n, H), device="cuda", generator=gen).abs() / math.sqrt(H)


def _out_rows(case):
    if case["kind"] == "decode":
        return case["B"] * case["g"]
    if case["kind"] == "varlen":
        return sum(_lens(case))
    return case["L"] - case.get("row0", 0)


def prepare(case, seed):
    gen = torch.Generator("cuda").manual_seed(seed)
    dtype = case["dtype"]
    if case["kind"] != "decode":
        L = sum(_lens(case)) if case["kind"] == "varlen" else case["L"]
        if case["kind"] == "varlen":
            keys = torch.cat([_keys(n, gen) for n in _lens(case)])
        else:
            keys = _keys(L, gen)
        k, ks = _stored(keys, dtype)
        q, qs = _queries(L, gen, dtype)
        # (rows outside a chunk belong to earlier chunks of the request)
        out = torch.full((L, case["k"]), -1, dtype=torch.int32, device="cuda")
        return {"case": case, "q": q, "qs": qs, "w": _gates(L, gen), "k": k, "ks": ks, "out": out}
    B, g, n0 = case["B"], case["g"], _visible(case)
    Lmax = (max(n0) + g + 127) // 128 * 128
    n_pages = B * Lmax // 128
    k = torch.zeros((B, Lmax, D), dtype=torch.uint8 if dtype == "fp8" else torch.bfloat16, device="cuda")
    ks = torch.zeros((B, Lmax), device="cuda") if dtype == "fp8" else None
    for b, n in enumerate(n0):
        kb, sb = _stored(_keys(n + g - 1, gen), dtype)
        k[b, : n + g - 1] = kb.view(torch.uint8) if dtype == "fp8" else kb
        if ks is not None:
            ks[b, : n + g - 1] = sb
    table = None
    if case["paged"]:                        # 128-key pages scattered over a pool
        perm = torch.randperm(n_pages, device="cuda", generator=gen)
        pages = torch.empty((n_pages, 128, D), dtype=k.dtype, device="cuda")
        pages[perm] = k.view(n_pages, 128, D)
        k = pages.view(n_pages * 128, D)
        if ks is not None:
            scales = torch.empty((n_pages, 128), device="cuda")
            scales[perm] = ks.view(n_pages, 128)
            ks = scales.view(-1)
        table = perm.to(torch.int32).view(B, Lmax // 128).contiguous()
    if dtype == "fp8":
        k = k.view(torch.float8_e4m3fn)
    q = torch.empty((B, g, H, D), dtype=torch.uint8 if dtype == "fp8" else torch.bfloat16, device="cuda")
    qs = torch.empty((B, g, H), device="cuda") if dtype == "fp8" else None
    for b in range(B):
        qb, sb = _queries(g, gen, dtype)
        q[b] = qb.view(torch.uint8) if dtype == "fp8" else qb
        if qs is not None:
            qs[b] = sb
    if dtype == "fp8":
        q = q.view(torch.float8_e4m3fn)
    return {"case": case, "q": q, "qs": qs, "w": _gates(B * g, gen).view(B, g, H), "k": k, "ks": ks, "table": table,
            "pos0": torch.tensor([n - 1 for n in n0], dtype=torch.int32, device="cuda"), "Lmax": Lmax,
            "n_pages": n_pages, "out": torch.empty((B, g, case["k"]), dtype=torch.int32, device="cuda")}


# ---------------------------------------------------------------------------------------- the pass

def _selection(out, n_keys):
    rows = out.view(-1, out.shape[-1])
    if rows.shape[0] * n_keys <= MASK_MAX:   # column 0 collects the -1 of rows with fewer than k keys
        mask = torch.zeros((rows.shape[0], n_keys + 1), dtype=torch.bool, device=out.device)
        return mask.scatter_(1, rows.long() + 1, True)
    # word 0 collects the -1; the positions of a row are distinct, so adding their bits sets them
    words = torch.zeros((rows.shape[0], n_keys // 32 + 2), dtype=torch.int32, device=out.device)
    one = torch.ones((), dtype=torch.int32, device=out.device)
    return words.scatter_add_(1, (rows >> 5).long().add_(1), torch.bitwise_left_shift(one, rows & 31))


def run(s):
    c, q, w, k, out, sc = s["case"], s["q"], s["w"], s["k"], s["out"], {"q_scale": s["qs"], "k_scale": s["ks"]}
    if c["kind"] == "prefill":
        L, row0 = c["L"], c["row0"]
        pv.pivot_index_prefill(q, w, k, L, H, D, c["g"], c["c"], c["k"], MODES[c["mode"]], out, W=c["W"],
                               rows=(row0, L) if row0 else None, **sc)
        return _selection(out[row0:], L)
    if c["kind"] == "varlen":
        cu = [0]
        for n in _lens(c):
            cu.append(cu[-1] + n)
        pv.pivot_index_prefill_varlen(q, w, k, cu, H, D, c["g"], c["c"], c["k"], MODES[c["mode"]], out, **sc)
        return _selection(out, max(_lens(c)))
    if c["kind"] == "dense":
        pv.dense_index(q, w, k, c["L"], H, D, c["k"], out, **sc)
        return _selection(out, c["L"])
    if c["paged"]:
        pv.pivot_index_decode_paged(q, w, k, s["table"], s["pos0"], c["B"], s["Lmax"] // 128, s["n_pages"], H, D, c["g"],
                                    c["c"], c["k"], MODES[c["mode"]], out, W=c["W"], **sc)
    else:
        pv.pivot_index_decode(q, w, k, s["pos0"], c["B"], s["Lmax"], H, D, c["g"], c["c"], c["k"], MODES[c["mode"]], out,
                              W=c["W"], **sc)
    return _selection(out, s["Lmax"])


# ---------------------------------------------------------------------------------------- what it takes

def _prefill_scores(L, row0, g, c, k, mode):
    """(query, key) scores of a request's rows row0 .. L - 1: guarded groups densely, one row per proxy
    (Eq. 5) and the re-scored candidates (Eq. 8)."""
    n = 0
    first = min((L + g - 1) // g, (c - 1 + g - 1) // g)      # groups whose prefix is shorter than c
    dense = min(L, first * g)
    if row0 < dense:
        n += (dense * (dense + 1) - row0 * (row0 + 1)) // 2
    lo = max(row0, dense) // g
    groups = (L + g - 1) // g - lo
    if groups > 0:
        n += g * (groups * lo + groups * (groups - 1) // 2) + groups
        if mode == "refine":
            n += (L - lo * g) * c
    return n


def work(case):
    """Every operand of the rows indexed and every key once, the index rows once; 2 H d operations per score."""
    esz, sb = (1, 4) if case["dtype"] == "fp8" else (2, 0)
    rows = _out_rows(case)
    per_row = H * (D * esz + sb + 4) + 4 * case["k"]
    if case["kind"] == "decode":
        n0, g, c = _visible(case), case["g"], case["c"]
        n = sum(n0)
        if case["mode"] == "refine":
            n += sum(g * min(c, m) for m in n0)
        if not case["paged"]:                                # sequences under the guardrail are scored densely
            n += sum((g - 1) * m + g * (g - 1) // 2 - (g * m if case["mode"] == "refine" else 0) for m in n0 if m < c)
        keys = sum(n0) + case["B"] * (g - 1)
    elif case["kind"] == "dense":
        keys = case["L"]
        n = keys * (keys + 1) // 2
    else:
        lens = _lens(case) if case["kind"] == "varlen" else [case["L"]]
        keys = sum(lens)
        n = sum(_prefill_scores(m, case.get("row0", 0), case["g"], case["c"], case["k"], case["mode"]) for m in lens)
    return {"bytes": rows * per_row + keys * (D * esz + sb), "flops": 2 * H * D * n}


def tolerance(case):
    """Share of mask entries (words) of another correct implementation that differ: scores within the
    rounding of the sums around a cut-off trade places.  fp8, this library's default (ReLU values rounded
    to bf16) against its fp32 head sums on the same inputs: a key or two of the k in a third of the rows, at
    most 2.8e-4 of a boolean mask, 0.8e-3 .. 2.2e-3 of the words.  bf16 against the CUDA-core kernels: 0 ..
    6e-8, and 1.7e-6 of the words."""
    n_keys = max(_lens(case)) if case["kind"] == "varlen" else case.get("L", case.get("hi"))
    if case["dtype"] == "bf16":
        return {"differ": 1e-5}
    return {"differ": 1e-3 if _out_rows(case) * n_keys <= MASK_MAX else 0.01}
