"""Performance cases: the work a user of this library has it do, over the range of sizes it is used at.

A retrieval-augmented generation service goes through four phases, and the cases follow them:

  docs        offline cache construction: the tokens of retrieved-passage documents attend a shared prefix and
              themselves (cf_document_prefill_attn), in one call for several layers or layer by layer
  stack       a query arrives: every layer's query rows attend the cached documents, documents are scored and pruned
              at the scheduled layers, the survivors are re-positioned (Session.run_stack, or Session.init / attend /
              prune from a model that issues one layer at a time), and the final cache is left in place ("keys") or
              packed per request ("cache", Session.assemble)
  reposition  the cached keys of every document moved to the positions an allocation gives them (Session.reposition)
  decode      one generated token: its key and value rows are appended and its query attends the final cache
              (cf_decode_plan, cf_decode_append, cf_decode_attn)

Tensor contents are normal variates drawn on the GPU from the seed; document lengths are uniform in the case's range,
their order differs from seed to seed.
Keys carry a per-document scale that falls in steps at the cuts of the pruning schedule, so that which documents
survive is a property of the inputs and not of rounding.
"""
from __future__ import annotations

import random
from typing import Dict, List, Tuple

import numpy as np
import torch

import paper_2502_11101_b200 as cf
from paper_2502_11101_b200.session import Session

STRATEGIES = {"none": cf.CF_ALLOC_NONE, "align": cf.CF_ALLOC_ALIGN, "sort": cf.CF_ALLOC_SORT}


def _stack(name: str, **kw) -> Dict:
    case = {"name": name, "kind": "stack", "dtype": "bf16", "q_heads": 12, "kv_heads": 2, "head_dim": 128,
            "theta": 1.0e6, "pos_range": 32768, "layers": 28, "docs": 50, "len_lo": 128, "len_hi": 192, "q_len": 48,
            "requests": 1, "schedule": "", "strategy": "align", "mode": "batched", "final": "keys", "prefix": 0,
            "self_block": False, "interleaved": False}
    case.update(kw)
    return case


def listed() -> List[Dict]:
    mha = {"q_heads": 32, "kv_heads": 32, "theta": 1.0e4, "pos_range": 4096}
    gqa7 = {"q_heads": 28, "kv_heads": 4}
    return [
        # the smallest request: a toy model in fp32 (what a correctness check or a CPU-sized experiment runs)
        _stack("stack_tiny_fp32", dtype="f32", q_heads=4, kv_heads=4, head_dim=64, theta=1.0e4, pos_range=256, layers=1,
               docs=8, len_lo=32, len_hi=32, q_len=16, schedule="1:4"),
        # one layer of a multi-head model over twenty passages, the survivors ordered by score
        _stack("stack_one_layer_mha", **mha, layers=1, docs=20, len_lo=120, len_hi=200, q_len=32, schedule="1:10",
               strategy="sort"),
        # scoring pass with stored query states: a small grouped-query model, fifty passages, three pruning layers
        _stack("stack_small_gqa", schedule="4:25,12:12,20:6"),
        # the same request inside a running model: one attention call per layer, pruning in between, packed final cache
        _stack("model_small_gqa", schedule="4:25,12:12,20:6", mode="model", final="cache"),
        # a batch of requests on a larger grouped-query model, layer by layer, with a shared prefix and the query's own block
        _stack("stack_batch_gqa_prefix_self", **gqa7, docs=100, q_len=64, requests=4, schedule="4:50,12:25,20:12",
               mode="layers", final="cache", prefix=64, self_block=True),
        # the largest batch: eight requests of 120 passages on a multi-head model (four layers of its stack resident)
        _stack("stack_batch_mha", **mha, layers=4, docs=120, len_lo=160, len_hi=200, q_len=64, requests=8,
               schedule="1:60,2:30,3:15"),
        # nothing is a round number: ragged passages, odd query and prefix lengths, interleaved slices, gaps left in place
        _stack("stack_ragged_interleaved", q_heads=32, kv_heads=8, layers=10, docs=37, len_lo=33, len_hi=317, q_len=29,
               requests=3, schedule="3:19,7:7", strategy="none", prefix=77, self_block=True, interleaved=True),
        # a generated token for one request, after pruning: a short cache, one call per layer
        {"name": "decode_one_gqa", "kind": "decode", "dtype": "bf16", "q_heads": 12, "kv_heads": 2, "head_dim": 128,
         "layers": 28, "requests": 1, "rows": 1011, "per_call": 1},
        # a generated token for a batch of eight on a multi-head model
        {"name": "decode_batch_mha", "kind": "decode", "dtype": "bf16", "q_heads": 32, "kv_heads": 32, "head_dim": 128,
         "layers": 32, "requests": 8, "rows": 2764, "per_call": 1},
        # cache construction of 400 passages behind a prefix, several layers per call
        {"name": "docs_gqa_prefix", "kind": "docs", "dtype": "bf16", "q_heads": 12, "kv_heads": 2, "head_dim": 128,
         "layers": 4, "docs": 400, "len_lo": 128, "len_hi": 192, "prefix": 64, "per_call": 4},
        # cache construction inside a running multi-head model: ragged passages, odd prefix, one layer per call
        {"name": "docs_mha_ragged", "kind": "docs", "dtype": "bf16", "q_heads": 32, "kv_heads": 32, "head_dim": 128,
         "layers": 4, "docs": 60, "len_lo": 47, "len_hi": 391, "prefix": 41, "per_call": 1},
        # every key of a large store moved to new positions
        {"name": "reposition_store", "kind": "reposition", "dtype": "bf16", "q_heads": 32, "kv_heads": 32,
         "head_dim": 128, "theta": 1.0e4, "pos_range": 4096, "layers": 4, "docs": 120, "len_lo": 160, "len_hi": 200,
         "requests": 8, "q_len": 64, "interleaved": False},
    ]


# ------------------------------------------------------------------------------------------------ drawn cases

def _between(rng: random.Random, lo: int, hi: int) -> int:
    """An integer of [lo, hi], its logarithm uniform."""
    return min(hi, max(lo, int(round(lo * (hi / lo) ** rng.random()))))


def _lengths(rng: random.Random, lo: int, hi: int) -> Tuple[int, int]:
    a, b = sorted((_between(rng, lo, hi), _between(rng, lo, hi)))
    return a, b


_GEOMETRIES = [(12, 2, 1.0e6, 32768), (28, 4, 1.0e6, 32768), (32, 8, 1.0e6, 32768), (32, 32, 1.0e4, 4096)]


def _draw_stack(rng: random.Random) -> Dict:
    case = _stack("")
    del case["name"]
    if rng.random() < 0.2:                                     # experiments in fp32 stay small
        case.update(dtype="f32", theta=1.0e4, pos_range=4096, layers=_between(rng, 1, 4), docs=_between(rng, 4, 24),
                    q_len=_between(rng, 4, 32))
        case["q_heads"], case["kv_heads"], case["head_dim"] = rng.choice([(4, 4, 64), (8, 2, 64), (8, 2, 128)])
        case["len_lo"], case["len_hi"] = _lengths(rng, 16, 200)
        case["mode"] = rng.choice(["batched", "model"])
    else:
        case["q_heads"], case["kv_heads"], case["theta"], case["pos_range"] = rng.choice(_GEOMETRIES)
        case.update(layers=_between(rng, 1, 28), docs=_between(rng, 4, 120), q_len=_between(rng, 7, 80),
                    requests=_between(rng, 1, 8), mode=rng.choice(["batched", "layers", "model"]),
                    final=rng.choice(["keys", "cache"]), interleaved=rng.random() < 0.25)
        case["len_lo"], case["len_hi"] = _lengths(rng, 32, 330)
        if case["mode"] != "model":
            case["self_block"] = rng.random() < 0.4
            case["prefix"] = rng.choice([0, 0, _between(rng, 9, 300)])
    case["strategy"] = rng.choice(["align", "none"] + (["sort"] if case["docs"] <= 20 and case["requests"] <= 2 else []))
    return case


def _draw_decode(rng: random.Random) -> Dict:
    q_heads, kv_heads, _, _ = rng.choice(_GEOMETRIES)
    case = {"kind": "decode", "dtype": "bf16", "q_heads": q_heads, "kv_heads": kv_heads, "head_dim": 128,
            "layers": _between(rng, 1, 32), "requests": _between(rng, 1, 16), "rows": _between(rng, 100, 20000)}
    case["per_call"] = case["layers"] if rng.random() < 0.2 else 1
    return case


def _draw_docs(rng: random.Random) -> Dict:
    q_heads, kv_heads, _, _ = rng.choice(_GEOMETRIES)
    lo, hi = _lengths(rng, 24, 400)
    case = {"kind": "docs", "dtype": "bf16", "q_heads": q_heads, "kv_heads": kv_heads, "head_dim": 128,
            "layers": _between(rng, 1, 28), "docs": _between(rng, 4, 400), "len_lo": lo, "len_hi": hi,
            "prefix": rng.choice([0, 64, _between(rng, 9, 300)])}
    case["per_call"] = rng.choice([1, case["layers"]])
    return case


def _draw_reposition(rng: random.Random) -> Dict:
    q_heads, kv_heads, theta, pos_range = rng.choice(_GEOMETRIES)
    lo, hi = _lengths(rng, 32, 330)
    return {"kind": "reposition", "dtype": rng.choice(["bf16", "bf16", "f32"]), "q_heads": q_heads, "kv_heads": kv_heads,
            "head_dim": 128, "theta": theta, "pos_range": pos_range, "layers": _between(rng, 1, 28),
            "docs": _between(rng, 4, 120), "len_lo": lo, "len_hi": hi, "requests": _between(rng, 1, 8), "q_len": 64,
            "interleaved": rng.random() < 0.25}


def _halving(case: Dict, rng: random.Random) -> str:
    """A pruning schedule like the configurations': half of the documents go at each of up to three layers."""
    layers, keep, cuts = case["layers"], case["docs"], {}
    for at in ([1 / 7, 3 / 7, 5 / 7] if layers >= 3 else [1.0])[:rng.randint(1, 3)]:
        keep = max(2, keep // 2)
        cuts[max(1, int(round(at * layers)))] = keep
    return ",".join("%d:%d" % c for c in sorted(cuts.items()))


def draw(rng: random.Random) -> Dict:
    make = rng.choice([_draw_stack] * 5 + [_draw_decode] * 2 + [_draw_docs] * 2 + [_draw_reposition])
    case = make(rng)
    most = [max(_cost(c) for c in listed()), max(_state_bytes(c) for c in listed())]
    while _cost(case) > most[0] or _state_bytes(case) > most[1]:
        grown = max((k for k in ("layers", "requests", "docs", "rows") if case.get(k, 1) > 1), key=lambda k: case[k] if k != "rows" else case[k] // 100)
        case[grown] = max(1, case[grown] * 2 // 3)
        if case["kind"] in ("decode", "docs") and case["per_call"] > 1:
            case["per_call"] = case["layers"]
    if case["kind"] == "stack":
        case["schedule"] = _halving(case, rng)
    return case


# ------------------------------------------------------------------------------------------------- what a pass needs

def _schedule(case: Dict) -> List[Tuple[int, int]]:
    return [tuple(int(x) for x in part.split(":")) for part in case["schedule"].split(",") if part]


def _kept(case: Dict) -> List[int]:
    """Documents of a request that each layer attends, and those left at the end."""
    cuts, keep, kept = dict(_schedule(case)), case["docs"], []
    for layer in range(1, case["layers"] + 1):
        kept.append(keep)
        keep = min(keep, cuts.get(layer, keep))
    return kept + [keep]


def work(case: Dict) -> Dict[str, float]:
    e = 2 if case["dtype"] == "bf16" else 4
    hq, hkv, d, layers = case["q_heads"], case["kv_heads"], case["head_dim"], case["layers"]
    row = hkv * d * e                                          # one token's keys (or values) of one layer
    if case["kind"] == "stack":
        length, b, lq = (case["len_lo"] + case["len_hi"]) / 2, case["requests"], case["q_len"]
        kept = _kept(case)
        tokens = b * length * sum(kept[:-1])
        nbytes = tokens * 2 * row + layers * b * lq * hq * (2 * d * e + 4) + layers * b * case["docs"] * 4
        flops = 4.0 * d * hq * lq * tokens
        if case["self_block"]:
            nbytes += layers * b * lq * 2 * row
            flops += 4.0 * d * hq * layers * b * lq * (lq + 1) / 2
        if case["prefix"]:
            nbytes += layers * case["prefix"] * 2 * row
            flops += 4.0 * d * hq * layers * b * lq * case["prefix"]
        last = layers * b * length * kept[-1]
        nbytes += 2 * last * row if case["final"] == "keys" else 4 * (last + layers * b * lq) * row
        return {"bytes": nbytes, "flops": flops + 3.0 * last * hkv * d}
    if case["kind"] == "decode":
        rows = layers * case["requests"] * (0.75 * case["rows"] + 1)
        each = layers * case["requests"]
        return {"bytes": rows * 2 * row + each * (hq * d * e * 2 + 4 * row), "flops": 4.0 * d * hq * rows}
    if case["kind"] == "docs":
        lo, hi, n = case["len_lo"], case["len_hi"], case["docs"] * layers
        mean, square = (lo + hi) / 2, (lo * lo + lo * hi + hi * hi) / 3
        nbytes = n * mean * (2 * row + hq * (2 * d * e + 4)) + layers * case["prefix"] * 2 * row
        return {"bytes": nbytes, "flops": 4.0 * d * hq * n * (mean * case["prefix"] + (square + mean) / 2)}
    tokens = layers * case["requests"] * case["docs"] * (case["len_lo"] + case["len_hi"]) / 2
    return {"bytes": 2 * tokens * row, "flops": 3.0 * tokens * hkv * d}


def _cost(case: Dict) -> float:
    w = work(case)
    return w["bytes"] + w["flops"] / 250


def _state_bytes(case: Dict) -> float:
    row = case["kv_heads"] * case["head_dim"] * (2 if case["dtype"] == "bf16" else 4)
    if case["kind"] == "decode":
        return 2.0 * case["layers"] * case["requests"] * case["rows"] * row
    tokens = case["layers"] * case.get("requests", 1) * case["docs"] * (case["len_lo"] + case["len_hi"]) / 2
    if case["kind"] == "docs":
        return tokens * (2 * row + 2 * row * case["q_heads"] / case["kv_heads"])
    return tokens * row * 3


def tolerance(case: Dict):
    if case["kind"] == "reposition":                           # one rounding to the storage type
        return {"rel": 2e-3, "max": 8e-3} if case["dtype"] == "bf16" else {"rel": 1e-6, "max": 1e-5}
    # bf16: keys, probabilities and outputs are rounded to 8 bits of significand; fp32: sums in another order
    return {"rel": 1e-2, "max": 1e-1} if case["dtype"] == "bf16" else {"rel": 1e-5, "max": 1e-3}


# --------------------------------------------------------------------------------------------------- inputs

def _dtype(case: Dict) -> torch.dtype:
    return torch.bfloat16 if case["dtype"] == "bf16" else torch.float32


class _Source:
    """Normal variates on the GPU and integers on the host, both from one seed."""

    def __init__(self, case: Dict, seed: int):
        self.gen = torch.Generator(device="cuda")
        self.gen.manual_seed(seed)
        self.rng = np.random.default_rng(seed)
        self.dtype = _dtype(case)

    def normal(self, *shape: int) -> torch.Tensor:
        return torch.empty(shape, dtype=self.dtype, device="cuda").normal_(generator=self.gen)

    def lengths(self, case: Dict, requests: int) -> np.ndarray:
        """Document lengths: the same ones for every seed (so that buffers have one size), in another order."""
        drawn = np.random.default_rng([case["len_lo"], case["len_hi"], case["docs"]])
        lens = drawn.integers(case["len_lo"], case["len_hi"] + 1, size=(requests, case["docs"]))
        return self.rng.permuted(lens, axis=1).reshape(-1).astype(np.int32)


def _session(case: Dict, lens: np.ndarray) -> Session:
    b = case["requests"]
    return Session(case["q_heads"], case["kv_heads"], case["head_dim"], _dtype(case), case["pos_range"], case["theta"],
                   case["q_len"], lens, np.arange(b + 1, dtype=np.int32) * case["docs"], np.zeros(len(lens), np.int32),
                   tail_reserve=case["q_len"], prefix_len=case.get("prefix", 0),
                   rope_layout=cf.CF_ROPE_INTERLEAVED if case["interleaved"] else cf.CF_ROPE_HALF)


def _key_scales(case: Dict, src: _Source) -> np.ndarray:
    """Per-document key scale, best documents of a request first in a random order of ids: a ladder with a wider
    step wherever the schedule cuts."""
    n = case["docs"]
    keeps = [k for _, k in _schedule(case)]
    ladder = np.array([1.6 - 0.7 * r / max(1, n - 1) - 0.1 * sum(k <= r for k in keeps) for r in range(n)], np.float32)
    scales = np.empty((case["requests"], n), np.float32)
    for b in range(case["requests"]):
        scales[b, src.rng.permutation(n)] = ladder
    return scales.reshape(-1)


def _prepare_stack(case: Dict, src: _Source) -> Dict:
    layers, b, lq = case["layers"], case["requests"], case["q_len"]
    hq, hkv, d = case["q_heads"], case["kv_heads"], case["head_dim"]
    lens = src.lengths(case, b)
    total = int(lens.sum())
    s = {"case": case, "schedule": _schedule(case), "strategy": STRATEGIES[case["strategy"]]}
    s["session"] = _session(case, lens)
    s["q"] = src.normal(layers, b, lq, hq, d)
    s["k"], s["v"] = src.normal(layers, total, hkv, d), src.normal(layers, total, hkv, d)
    scales = torch.from_numpy(np.repeat(_key_scales(case, src), lens)).to("cuda").to(s["k"].dtype)
    s["k"].mul_(scales[None, :, None, None])
    s["out"] = torch.zeros_like(s["q"])
    s["lse"] = torch.zeros((layers, b, hq, lq), device="cuda")
    s["layer_scores"] = torch.zeros((layers, len(lens)), device="cuda")
    s["k_self"] = s["v_self"] = s["k_prefix"] = s["v_prefix"] = s["k_final"] = None
    if case["self_block"] or case["final"] == "cache":
        s["k_self"], s["v_self"] = src.normal(layers, b, lq, hkv, d), src.normal(layers, b, lq, hkv, d)
    if case["prefix"]:
        s["k_prefix"], s["v_prefix"] = (src.normal(layers, case["prefix"], hkv, d) for _ in range(2))
    if case["final"] == "keys":
        s["k_final"] = torch.zeros_like(s["k"])
    else:
        keep = _kept(case)[-1]
        rows = max(int(np.sort(part)[::-1][:keep].sum()) for part in lens.reshape(b, -1)) + lq
        s["k_cache"] = torch.zeros((layers, b, rows, hkv, d), dtype=s["k"].dtype, device="cuda")
        s["v_cache"] = torch.zeros_like(s["k_cache"])
        s["cache_rows"] = torch.zeros(b, dtype=torch.int32, device="cuda")
    # the model's own views of its layers
    s["per_layer"] = [(s["q"][i], s["k"][i], s["v"][i], s["out"][i], s["lse"][i]) for i in range(layers)]
    s["positions"] = s["session"].field("dst_start", len(lens))
    return s


def _prepare_decode(case: Dict, src: _Source) -> Dict:
    layers, b, hq, hkv, d = case["layers"], case["requests"], case["q_heads"], case["kv_heads"], case["head_dim"]
    room = case["rows"] + 64
    s = {"case": case, "room": room, "geom": cf.make_geom(hq, hkv, d, _dtype(case), 1 << 20, 1.0e4)}
    # requests have kept different amounts: from half of the largest cache to all of it
    s["rows"] = torch.from_numpy(src.rng.integers((case["rows"] + 1) // 2, case["rows"] + 1, size=b).astype(np.int32)).to("cuda")
    s["k"], s["v"] = src.normal(layers, b, room, hkv, d), src.normal(layers, b, room, hkv, d)
    s["q"], s["k_new"], s["v_new"] = src.normal(layers, b, hq, d), src.normal(layers, b, hkv, d), src.normal(layers, b, hkv, d)
    s["out"] = torch.zeros_like(s["q"])
    s["lse"] = torch.zeros((layers, b, hq), device="cuda")
    s["plan"] = torch.zeros(cf.cf_decode_plan_bytes(s["geom"], b, room), dtype=torch.uint8, device="cuda")
    s["workspace"] = torch.empty(cf.cf_decode_workspace_bytes(s["geom"], b, room, case["per_call"]), dtype=torch.uint8, device="cuda")
    s["calls"] = [tuple(s[n][i:i + case["per_call"]] for n in ("k", "v", "k_new", "v_new", "q", "out", "lse"))
                  for i in range(0, layers, case["per_call"])]
    return s


def _prepare_docs(case: Dict, src: _Source) -> Dict:
    layers, hq, hkv, d = case["layers"], case["q_heads"], case["kv_heads"], case["head_dim"]
    lens = src.lengths(case, 1)
    total = int(lens.sum())
    s = {"case": case, "longest": int(lens.max()), "geom": cf.make_geom(hq, hkv, d, _dtype(case), 32768, 1.0e6)}
    s["offsets"] = torch.from_numpy(np.concatenate([[0], np.cumsum(lens)]).astype(np.int32)).to("cuda")
    s["q"], s["k"], s["v"] = src.normal(layers, total, hq, d), src.normal(layers, total, hkv, d), src.normal(layers, total, hkv, d)
    s["out"] = torch.zeros_like(s["q"])
    s["lse"] = torch.zeros((layers, hq, total), device="cuda")
    prefix = [src.normal(layers, case["prefix"], hkv, d) if case["prefix"] else None for _ in range(2)]
    s["calls"] = []
    for i in range(0, layers, case["per_call"]):
        j = i + case["per_call"]
        s["calls"].append(tuple(s[n][i:j] for n in ("q", "k", "v", "out")) + tuple(None if p is None else p[i:j] for p in prefix) + (s["lse"][i:j],))
    return s


def _prepare_reposition(case: Dict, src: _Source) -> Dict:
    lens = src.lengths(case, case["requests"])
    s = {"case": case, "session": _session(case, lens)}
    s["k"] = src.normal(case["layers"], int(lens.sum()), case["kv_heads"], case["head_dim"])
    s["k_out"] = torch.zeros_like(s["k"])
    s["session"].init()                                        # where the documents go is known before the keys are moved
    return s


_PREPARE = {"stack": _prepare_stack, "decode": _prepare_decode, "docs": _prepare_docs, "reposition": _prepare_reposition}


def prepare(case: Dict, seed: int) -> Dict:
    return _PREPARE[case["kind"]](case, _Source(case, seed))


# --------------------------------------------------------------------------------------------------- a pass

def _run_stack(s: Dict) -> Dict:
    case, sess = s["case"], s["session"]
    if case["mode"] == "model":
        cuts = dict(s["schedule"])
        sess.set_live_docs(case["docs"])
        sess.init()
        for layer, (q, k, v, out, lse) in enumerate(s["per_layer"], 1):
            sess.attend(q, k, v, out, lse)
            if layer in cuts:
                sess.prune(cuts[layer], s["strategy"])
        if case["final"] == "keys":
            sess.reposition(s["k"], s["k_final"], case["layers"], s["k"].stride(0))
    else:
        own = case["self_block"]
        sess.run_stack(s["q"], s["k"], s["v"], s["schedule"], s["strategy"], s["out"], s["lse"], s["k_final"],
                       s["layer_scores"], batch_layers=case["mode"] == "batched", k_self=s["k_self"] if own else None,
                       v_self=s["v_self"] if own else None, k_prefix=s["k_prefix"], v_prefix=s["v_prefix"])
    result = {"out": s["out"], "lse": s["lse"], "scores": sess.score_accum, "positions": s["positions"]}
    if case["mode"] != "model":
        result["layer_scores"] = s["layer_scores"]
    if case["final"] == "keys":
        result["k_final"] = s["k_final"]
    else:
        sess.assemble(s["k"], s["v"], s["k_self"], s["v_self"], s["k_cache"], s["v_cache"], s["cache_rows"])
        result.update(k_cache=s["k_cache"], v_cache=s["v_cache"], cache_rows=s["cache_rows"])
    return result


def _run_decode(s: Dict) -> Dict:
    geom, b, room, rows, plan = s["geom"], s["case"]["requests"], s["room"], s["rows"], s["plan"]
    cf.cf_decode_plan(geom, b, room, rows, 1, plan)
    for k, v, k_new, v_new, q, out, lse in s["calls"]:
        cf.cf_decode_append(geom, b, room, k, v, rows, 0, k_new, v_new)
        cf.cf_decode_attn(geom, b, room, plan, q, k, v, out, s["workspace"], lse)
    return {"out": s["out"], "lse": s["lse"], "k": s["k"], "v": s["v"]}


def _run_docs(s: Dict) -> Dict:
    for q, k, v, out, k_prefix, v_prefix, lse in s["calls"]:
        cf.cf_document_prefill_attn(s["geom"], s["offsets"], s["longest"], q, k, v, out, k_prefix, v_prefix, lse)
    return {"out": s["out"], "lse": s["lse"]}


def _run_reposition(s: Dict) -> Dict:
    s["session"].reposition(s["k"], s["k_out"], s["case"]["layers"], s["k"].stride(0))
    return {"k_out": s["k_out"]}


_RUN = {"stack": _run_stack, "decode": _run_decode, "docs": _run_docs, "reposition": _run_reposition}


def run(state: Dict) -> Dict:
    return _RUN[state["case"]["kind"]](state)
