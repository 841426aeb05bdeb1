"""The work that a decoding program has this library do, as cases to be timed.

A case is one decode step's evaluation of one layer (of several for
``path = "layers"``), through the functions of ``paper_2602_18750_gb300.hill``:

* ``step``    hill_evict_step: score the whole cache, select the top-k tokens,
              attend over them; with ``accum`` the running importance of the
              sweep workload is updated and ranked;
* ``bkp``     hill_evict_step_bkp: the same with the recent window pinned and
              the hit-rate table updated;
* ``kvh``     hill_evict_step_kvh: every KV head keeps a set of its own;
* ``f8``      hill_quantize_k of the token just appended, then
              hill_evict_step_f8: scoring from the E4M3 key shadow;
* ``shadow``  hill_quantize_k over whole prompts: the encoding of the keys
              that comes before the first f8 step of a sequence;
* ``layers``  the layer-pipelined decode step: hill_evict_step_begin on one
              stream, hill_evict_step_end on a second, the attention
              (hill_gather_sparse_attn) on a third.

Inputs come from the package's own seeded generators (Zipf, planted and
outlier attention skews).  The budget k[b] is the one within a few tokens of
floor(frac * length) with the widest gap between the last kept and the first
dropped token, so that the kept set is decided by the importance and not by
the last bits of a sum: index sets are then compared exactly.
"""
from __future__ import annotations

import math
import random
import zlib

import torch

from paper_2602_18750_gb300 import hill, inputs

D = 128
DTYPES = {"fp16": torch.float16, "bf16": torch.bfloat16}
APPEND = 64   # tokens the cache has room for beyond the longest prompt (decode steps to come)
BASE = dict(path="step", mode="attn", batch=1, heads=32, kv_heads=32, tokens=4096, ragged=False, dtype="fp16",
            skew="zipf", frac=0.2, accum=False, recent=0, layout="head", layers=1)


def _case(name, **over):
    return dict(BASE, name=name, **over)


def listed():
    return [
        # the smallest call: one sequence of 4K tokens of a 32-head model, k = 819 (a single chat turn; launches
        # and latency count)
        _case("step-1x4k-mha", skew="planted"),
        # the paper's own setting: batch 8, 4K tokens, fp16, alpha = 20 % (Sec. 5.2)
        _case("step-8x4k-mha", batch=8),
        # long documents of different lengths, 16K to 32K tokens, alpha = 10 % (the benchmark's default workload)
        _case("step-4x32k-mha-ragged", batch=4, tokens=32768, ragged=True, frac=0.1),
        # one very long context of a grouped-query model in bf16, 2048 tokens kept
        _case("step-1x128k-gqa-bf16", kv_heads=8, tokens=131072, dtype="bf16", skew="outlier", frac=2048 / 131072),
        # the largest: 8 sequences of 64K tokens with the importance accumulated over the steps (the sweep)
        _case("accum-8x64k-mha", batch=8, tokens=65536, accum=True),
        # multi-query attention: 32 query heads share one KV head, odd lengths
        _case("step-4x16k-mqa", batch=4, kv_heads=1, tokens=16001, ragged=True, dtype="bf16", frac=0.1),
        # raw inner products (Sec. 4.4) with a pinned window and the hit table (Sec. 4.2), the cache stored token
        # by token as many serving programs keep it
        _case("bkp-3x12k-gqa-raw", path="bkp", mode="raw", batch=3, kv_heads=8, tokens=12345, ragged=True, recent=128,
              layout="token"),
        # every KV head keeps its own tokens
        _case("kvh-2x16k-gqa-bf16", path="kvh", batch=2, kv_heads=8, tokens=16384, dtype="bf16", frac=0.1),
        # scoring from the 8-bit key shadow (Sec. 4.4), long documents of a 32-head model
        _case("f8-4x32k-mha-ragged", path="f8", batch=4, tokens=32768, ragged=True, frac=0.1),
        # the same on one very long context of a grouped-query model
        _case("f8-1x128k-gqa-bf16", path="f8", kv_heads=8, tokens=131072, dtype="bf16", skew="outlier",
              frac=2048 / 131072),
        # building that shadow for the prompts of a batch
        _case("shadow-4x16k-mha", path="shadow", batch=4, tokens=16384, ragged=True),
        # the layer-pipelined decode step (Sec. 4.3) over four layers
        _case("layers-4x2x16k-mha", path="layers", batch=2, tokens=16384, frac=0.1, layers=4),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """A case of the listed ones' ranges: 1 to 16 sequences of 1K to 128K tokens, every head layout, both
    importance rules, budgets from 2 % to 50 %; at most half the keys of the largest listed case."""
    while True:
        path = rng.choice(["step"] * 4 + ["bkp", "kvh", "f8", "f8", "shadow", "layers"])
        c = dict(BASE, path=path)
        c["heads"], c["kv_heads"] = rng.choice([(32, 32), (32, 32), (32, 8), (32, 8), (64, 8), (28, 4), (40, 40), (32, 1)])
        c["batch"] = _log(rng, 1, 16)
        c["tokens"] = _log(rng, 1000, 131072)
        c["ragged"] = rng.random() < 0.5
        c["dtype"] = rng.choice(["fp16", "bf16"])
        c["skew"] = rng.choice(["zipf", "zipf", "outlier", "normal"])
        c["frac"] = round(math.exp(rng.uniform(math.log(0.02), math.log(0.5))), 4)
        c["mode"] = "raw" if rng.random() < 0.25 else "attn"
        if path in ("step", "bkp", "layers"):
            c["accum"] = rng.random() < 0.3
        if path == "bkp":
            c["recent"] = rng.choice([32, 128, 500])
        if path != "f8" and rng.random() < 0.25:
            c["layout"] = "token"
        if path == "layers":
            c["layers"] = rng.randint(2, 4)
        keys = c["batch"] * c["tokens"] * c["kv_heads"] * c["layers"]
        if keys > 8 * 65536 * 32 // 2:
            continue
        if path == "kvh" and c["kv_heads"] > 8:   # separate sets: grouped and multi-query models
            continue
        if c["tokens"] * c["frac"] < 16:
            continue
        return c


# ---------------------------------------------------------------- inputs
def _lens(case):
    """Cached tokens of every sequence; ragged: the longest, and others between half of it and it."""
    n, B = case["tokens"], case["batch"]
    if not case["ragged"]:
        return [n] * B
    r = random.Random(zlib.crc32(repr(sorted((k, v) for k, v in case.items() if k != "name")).encode()))
    return [n] + [r.randint(max(1, n // 2), n) for _ in range(B - 1)]


def _layer(case, seed, layer):
    """(q, K, V) of one layer, on the GPU."""
    w = inputs.Workload("case", case["layers"], case["batch"], case["heads"], case["kv_heads"], D, tuple(_lens(case)),
                        APPEND, DTYPES[case["dtype"]], case["skew"], None, 1, planted=64, outlier_frac=0.005,
                        seed=int(seed))
    K, V = inputs.layer_cache(w, layer, "cuda")
    if case["layout"] == "token":   # [B][cap][Hkv][d] in memory
        K, V = (x.transpose(1, 2).contiguous().transpose(1, 2) for x in (K, V))
    return inputs.step_query(w, layer, 0, "cuda"), K, V


def _budget_frac(case):
    return [int(math.floor(case["frac"] * n)) for n in _lens(case)]


def _span(case):
    """How far a budget may move from its nominal value."""
    return max(4, min(32, min(_budget_frac(case)) // 8))


def _max_k(case):
    return max(_budget_frac(case)) + _span(case) + case["recent"]


def _previous_importance(case, seed, layer):
    """The running importance of the steps before this one, as the caller holds it."""
    g = torch.Generator(device="cuda").manual_seed(zlib.crc32(repr((int(seed), "accum", layer)).encode()))
    cap = max(_lens(case)) + APPEND - 1
    mean = case["heads"] / max(_lens(case)) if case["mode"] == "attn" else math.sqrt(case["heads"])
    return torch.rand(case["batch"], cap, generator=g, device="cuda") * mean


def _budgets(case, per_layer):
    """k[b]: near floor(frac * len), where the kept and the dropped tokens lie furthest apart in every one of the
    rankings in `per_layer` (lists of [b] -> rows of 64-bit keys)."""
    ks = []
    for b, (n, k0) in enumerate(zip(_lens(case), _budget_frac(case))):
        older, span = n - min(case["recent"], n), _span(case)
        lo, hi = max(1, k0 - span), min(older - 1, k0 + span)
        if hi <= lo:
            ks.append(max(1, min(k0, older)))
            continue
        worst = None
        for keys in per_layer:
            top = torch.topk(keys[b][..., :older].reshape(-1, older), hi + 1, dim=-1).values
            a, c = top[:, lo - 1:hi], top[:, lo:hi + 1]
            gap = ((a - c) / torch.maximum(a.abs(), c.abs()).clamp_min(1e-30)).amin(0)
            worst = gap if worst is None else torch.minimum(worst, gap)
        ks.append(lo + int(worst.argmax()))
    return torch.tensor(ks, dtype=torch.int32, device="cuda")


def prepare(case, seed):
    hill.load()
    mode = hill.HILL_SCORE_RAW if case["mode"] == "raw" else hill.HILL_SCORE_ATTN
    path, B, H, Hkv = case["path"], case["batch"], case["heads"], case["kv_heads"]
    lens = torch.tensor(_lens(case), dtype=torch.int32, device="cuda")
    s = {"case": case, "mode": mode, "lens": lens, "layers": []}
    if path == "shadow":
        q, K, V = _layer(case, seed, 0)
        s["desc"] = hill.make_desc(q, K)
        k8, ks = hill.alloc_shadow(s["desc"])
        s.update(K=K, k8=k8, ks=ks, zero=torch.zeros_like(lens), max_rows=max(_lens(case)))
        return s
    max_k, rankings = _max_k(case), []
    for l in range(case["layers"]):
        q, K, V = _layer(case, seed, l)
        cap = K.shape[2]
        rows = (B, Hkv) if path == "kvh" else (B,)
        y = {"q": q, "K": K, "V": V}
        y["scores"] = torch.zeros(*rows, cap, device="cuda")
        y["idx"] = torch.full((*rows, max_k), -1, dtype=torch.int32, device="cuda")
        y["count"] = torch.zeros(*rows, dtype=torch.int32, device="cuda")
        y["out"] = torch.zeros(B, H, D, device="cuda")
        y["accum"] = _previous_importance(case, seed, l) if case["accum"] else None
        s["desc"] = hill.make_desc(q, K, V)
        y["ws"] = hill.alloc_workspace(s["desc"], mode, max_k)
        keys = K
        if path == "f8":   # the shadow of everything but the token of this step, as the steps before left it
            y["k8"], y["ks"] = hill.alloc_shadow(s["desc"])
            hill.hill_quantize_k(s["desc"], K, torch.zeros_like(lens), lens - 1, cap, y["k8"], y["ks"])
            keys = None
        if path == "bkp":
            y["hits"] = torch.zeros(B, cap, dtype=torch.int16, device="cuda")
        imp = _importance(case, q, K, group=path == "kvh", f8=keys is None)
        if case["accum"]:   # this pass and the one after it rank different sums
            prev = [y["accum"][b, :n].double() for b, n in enumerate(_lens(case))]
            rankings += [[p + i * m for p, i in zip(prev, imp)] for m in (1, 2)]
        else:
            rankings.append(imp)
        s["layers"].append(y)
    s["max_k"] = max_k
    s["k"] = _budgets(case, rankings)
    if path == "f8":
        s["new"] = lens - 1
    if path == "layers":
        s["side"], s["att"] = torch.cuda.Stream(), torch.cuda.Stream()
        s["wsa"] = [hill.alloc_workspace(s["desc"], mode, max_k) for _ in range(2)]
    torch.cuda.synchronize()
    return s


# ---------------------------------------------------------------- one pass
def _outputs(s):
    names = ["scores", "idx", "count", "out"] + [n for n in ("accum", "hits") if s["layers"][0].get(n) is not None]
    return [{n: y[n] for n in names} for y in s["layers"]]


def run(s):
    case, path = s["case"], s["case"]["path"]
    if path == "shadow":
        hill.hill_quantize_k(s["desc"], s["K"], s["zero"], s["lens"], s["max_rows"], s["k8"], s["ks"])
        return {"codes": s["k8"], "scales": s["ks"]}
    desc, mode, lens, k, max_k = s["desc"], s["mode"], s["lens"], s["k"], s["max_k"]
    if path == "layers":
        _pipelined(s)
        return _outputs(s)
    y = s["layers"][0]
    if path == "step":
        hill.hill_evict_step(desc, y["q"], y["K"], y["V"], lens, k, max_k, mode, y["accum"], y["scores"], y["idx"],
                             y["count"], y["out"], y["ws"])
    elif path == "bkp":
        hill.hill_evict_step_bkp(desc, y["q"], y["K"], y["V"], lens, k, case["recent"], max_k, mode, y["accum"],
                                 y["scores"], y["idx"], y["count"], y["hits"], y["out"], y["ws"])
    elif path == "kvh":
        hill.hill_evict_step_kvh(desc, y["q"], y["K"], y["V"], lens, k, max_k, mode, None, y["scores"], y["idx"],
                                 y["count"], y["out"], y["ws"])
    else:
        hill.hill_quantize_k(desc, y["K"], s["new"], lens, 1, y["k8"], y["ks"])
        hill.hill_evict_step_f8(desc, y["q"], y["k8"], y["ks"], y["K"], y["V"], lens, k, max_k, mode, None, y["scores"],
                                y["idx"], y["count"], y["out"], y["ws"])
    return _outputs(s)


def _pipelined(s):
    """The K stream of every layer on the current stream, normalisation and selection on a second, the attention on
    a third; one evaluation workspace per layer, two attention workspaces in turn."""
    st, side, att = torch.cuda.current_stream(), s["side"], s["att"]
    fork = torch.cuda.Event()
    fork.record(st)
    side.wait_event(fork)
    att.wait_event(fork)
    for l, y in enumerate(s["layers"]):
        hill.hill_evict_step_begin(s["desc"], y["q"], y["K"], s["lens"], s["max_k"], s["mode"], y["accum"], y["scores"],
                                   y["ws"], st)
        streamed = torch.cuda.Event()
        streamed.record(st)
        side.wait_event(streamed)
        hill.hill_evict_step_end(s["desc"], s["lens"], s["k"], s["max_k"], s["mode"], y["accum"], y["scores"], y["idx"],
                                 y["count"], y["ws"], stream=side)
        kept = torch.cuda.Event()
        kept.record(side)
        att.wait_event(kept)
        hill.hill_gather_sparse_attn(s["desc"], y["q"], y["K"], y["V"], y["idx"], y["count"], s["max_k"], y["out"],
                                     s["wsa"][l % 2], att)
    for h in (side, att):
        join = torch.cuda.Event()
        join.record(h)
        st.wait_event(join)


# ---------------------------------------------------------------- what a pass cannot do without
def work(case):
    B, H, Hkv, n = case["batch"], case["heads"], case["kv_heads"], sum(_lens(case))
    if case["path"] == "shadow":
        return {"bytes": n * Hkv * (2 * D + D + 4), "flops": 2 * n * Hkv * D}
    kept = sum(min(k + case["recent"], m) for k, m in zip(_budget_frac(case), _lens(case)))
    rows = Hkv if case["path"] == "kvh" else 1
    key = D + 4 if case["path"] == "f8" else 2 * D
    # keys once (from the shadow: and the kept rows of the 16-bit keys), the kept rows of the values, the
    # importance written, the indices written, queries and outputs
    b = n * Hkv * key + kept * Hkv * 2 * D + n * rows * 4 + kept * rows * 4 + B * H * D * 6
    b += kept * Hkv * 2 * D if case["path"] == "f8" else 0
    b += n * 8 if case["accum"] else 0
    b += kept * 4 if case["path"] == "bkp" else 0
    return {"bytes": b * case["layers"], "flops": (2 * n + 4 * kept) * H * D * case["layers"]}


def tolerance(case):
    """Whole values (indices, counts, hits, codes) are the same.  Importance and attention hold 32-bit sums: measured
    2e-7 to 6e-6 from the same in 64 bits, so two of them may lie four times that apart; scales are one rounding."""
    return {"rel": 1e-6} if case["path"] == "shadow" else {"rel": 2e-5}


# ---------------------------------------------------------------- the same in 64 bits
def _e4m3(x):
    """(values, scale) of the E4M3 form of rows x [..., 128]: 32-bit steps, round to nearest even, saturating."""
    x = x.float()
    amax = x.abs().amax(-1, keepdim=True)
    top = torch.full_like(amax, 448.0)   # tensor by tensor: a division by or of a number may become a product
    r = torch.where(amax > 0, top / amax, torch.zeros_like(amax))
    return (x * r).clamp(-448.0, 448.0).to(torch.float8_e4m3fn), amax / top


def _logits(case, q, K, b, f8):
    """[H][n] logits of sequence b in 64 bits."""
    n, G = _lens(case)[b], case["heads"] // case["kv_heads"]
    out = torch.empty(case["heads"], n, dtype=torch.float64, device=q.device)
    qb = q[b]
    if f8:
        c, sc = _e4m3(qb)
        qb = c.double() * sc.double()
    for g in range(case["kv_heads"]):
        kb = K[b, g, :n]
        if f8:
            c, sc = _e4m3(kb)
            kb = c.double() * sc.double()
        out[g * G:(g + 1) * G] = qb[g * G:(g + 1) * G].double() @ kb.double().T
    return out / math.sqrt(D)


def _importance(case, q, K, group=False, f8=False):
    """Per sequence: [n] (or [Hkv][n]) importance in 64 bits."""
    got = []
    for b in range(case["batch"]):
        z = _logits(case, q, K, b, f8)
        if case["mode"] == "attn":
            z = torch.softmax(z, -1)
        got.append(z.reshape(case["kv_heads"], -1, z.shape[-1]).sum(1) if group else z.sum(0))
    return got


def _attend(case, q, K, V, b, kept):
    """[H][d]: attention of sequence b over kept tokens (one set, or one for every KV head)."""
    G, out = case["heads"] // case["kv_heads"], []
    for g in range(case["kv_heads"]):
        t = kept[g] if isinstance(kept, list) else kept
        p = torch.softmax(q[b, g * G:(g + 1) * G].double() @ K[b, g, t].double().T / math.sqrt(D), -1)
        out.append(p @ V[b, g, t].double())
    return torch.cat(out)


def exact(case, seed):
    lens, path = _lens(case), case["path"]
    if path == "shadow":
        _, K, _ = _layer(case, seed, 0)
        B, Hkv, cap, _ = K.shape
        scales = torch.zeros(B, Hkv, (cap + 31) // 32 * 32, dtype=torch.float64, device="cuda")
        for b, n in enumerate(lens):
            scales[b, :, :n] = K[b, :, :n].double().abs().amax(-1) / 448.0
        return {"codes": None, "scales": scales}
    layers = []
    max_k, group = _max_k(case), path == "kvh"
    for l in range(case["layers"]):
        q, K, V = _layer(case, seed, l)
        layers.append((q, K, V, _importance(case, q, K, group, path == "f8"),
                       _previous_importance(case, seed, l).double() if case["accum"] else None))
    rankings = []
    for q, K, V, imp, prev in layers:
        if prev is not None:
            rankings += [[prev[b, :n] + m * imp[b] for b, n in enumerate(lens)] for m in (1, 2)]
        else:
            rankings.append(imp)
    ks = _budgets(case, rankings).tolist()
    got = []
    for q, K, V, imp, prev in layers:
        B, cap = case["batch"], K.shape[2]
        rows = (B, case["kv_heads"]) if group else (B,)
        scores = torch.zeros(*rows, cap, dtype=torch.float64, device="cuda")
        idx = torch.full((*rows, max_k), -1, dtype=torch.int32, device="cuda")
        count = torch.zeros(*rows, dtype=torch.int32, device="cuda")
        out = torch.zeros(B, case["heads"], D, dtype=torch.float64, device="cuda")
        accum = prev.clone() if prev is not None else None
        hits = torch.zeros(B, cap, dtype=torch.int16, device="cuda")
        for b, n in enumerate(lens):
            scores[b, ..., :n] = imp[b]
            key = imp[b]
            if accum is not None:
                accum[b, :n] += imp[b]
                key = accum[b, :n]
            older = n - min(case["recent"], n)
            window = torch.arange(older, n, device="cuda")
            k = min(ks[b], older)
            top = [torch.topk(r[:older], k).indices.sort().values for r in key.reshape(-1, n)]
            kept = [torch.cat([t, window]) for t in top]
            for g, t in enumerate(kept):
                row = (b, g) if group else (b,)
                idx[row][:len(t)] = t.int()
                count[row] = len(t)
            out[b] = _attend(case, q, K, V, b, kept if group else kept[0])
            hits[b, kept[0]] += 1
        one = {"scores": scores, "idx": idx, "count": count, "out": out}
        if accum is not None:
            one["accum"] = accum
        if path == "bkp":
            one["hits"] = hits
        got.append(one)
    return got
