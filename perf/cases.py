"""Cases of the framework's work, one pass of which is timed: building an index, searching it, scoring against it, turning
codes back into vectors, storing codes, and attention over a compressed KV cache.

A case is a dict of plain values; "op" says which of the paths below it takes:
  index        tq_quantize_prod / tq_quantize_mse of n vectors
  search       tq_topk of nq queries over n codes
  score        tq_score: the dense nq x n estimates
  reconstruct  tq_dequantize of n codes
  store        tq_entropy_pack and tq_entropy_unpack of n index rows
  prefill      the keys and values of a prompt into a compressed KV cache (one call per channel group and side)
  decode       one decoding step of one layer: tq_kv_append of the new token, tq_attend_decode over the whole context
"""
import math

import torch

import paper_2504_19874_b200 as tq

GROUP, HEAD_DIM = 64, 128           # a head's channels: two groups of 64 (outlier channels and the rest)
PLAN_SEED = 82


def listed():
    return [
        # One decoding step of a chat that has just begun: the smallest calls, launches and host work count.
        {"name": "decode_1k", "op": "decode", "heads": 8, "q_per_kv": 4, "tokens": 1000, "high_bits": 3, "low_bits": 2},
        # The same layer (64 channels at 3 bits, 64 at 2) over a long context.
        {"name": "decode_32k", "op": "decode", "heads": 8, "q_per_kv": 4, "tokens": 32768, "high_bits": 3, "low_bits": 2},
        # A context at the end of what the model takes, in the 3.5-bit split.
        {"name": "decode_104k", "op": "decode", "heads": 8, "q_per_kv": 4, "tokens": 106496, "high_bits": 4, "low_bits": 3},
        # A prompt of 4,096 tokens written to the cache.
        {"name": "prefill_4k", "op": "prefill", "heads": 8, "tokens": 4096, "high_bits": 3, "low_bits": 2},
        # A million embeddings indexed: the benchmark's workload and the largest quantisation.
        {"name": "index_1m", "op": "index", "d": 1536, "bits": 4, "mode": "prod", "nibble": True, "n": 1_000_000, "dtype": "f32"},
        # A batch of new documents added to an index of long embeddings, in the type that the network gives them in.
        {"name": "index_batch", "op": "index", "d": 3072, "bits": 2, "mode": "prod", "nibble": False, "n": 1001, "dtype": "bf16"},
        # One user's query against a million documents.
        {"name": "search_one", "op": "search", "d": 1536, "bits": 4, "mode": "prod", "nibble": True, "n": 1_000_000, "nq": 1, "k": 10, "dtype": "f32"},
        # A server's batch of queries against the cheapest index (two bits, no residual).
        {"name": "search_batch", "op": "search", "d": 1536, "bits": 2, "mode": "mse", "nibble": False, "n": 1_000_000, "nq": 8, "k": 100, "dtype": "f32"},
        # Ten thousand queries of a short, odd dimension: a whole evaluation set, or a k-nearest-neighbour graph.
        {"name": "search_many", "op": "search", "d": 200, "bits": 3, "mode": "prod", "nibble": False, "n": 1_000_000, "nq": 10_000, "k": 100, "dtype": "f32"},
        # A few thousand candidates scored for a batch of queries (re-ranking, a small collection).
        {"name": "score_small", "op": "score", "d": 128, "bits": 2, "mode": "mse", "nibble": False, "n": 4096, "nq": 64, "dtype": "f32"},
        # Vectors read back from an index, for export or exact re-ranking.
        {"name": "reconstruct", "op": "reconstruct", "d": 1536, "bits": 4, "mode": "prod", "nibble": True, "n": 50_000},
        # A segment of an index entropy-coded for storage and read back.
        {"name": "store", "op": "store", "d": 1536, "bits": 4, "mode": "mse", "n": 100_000},
    ]


def _size(rng, low, high):
    """A whole number from low to high, spread over its logarithm."""
    return max(low, min(high, int(round(math.exp(rng.uniform(math.log(low), math.log(high)))))))


def draw(rng):
    op = rng.choice(["decode", "prefill", "index", "search", "score", "reconstruct", "store"])
    if op in ("decode", "prefill"):
        case = {"op": op, "heads": rng.randint(1, 8), "tokens": _size(rng, 16, 106496 if op == "decode" else 16384)}
        case["high_bits"], case["low_bits"] = rng.choice([(3, 2), (4, 3), (4, 2), (3, 3)])
        if op == "decode":
            case["q_per_kv"] = rng.randint(1, 4)
        return case
    d = rng.choice([128, 200, 384, 768, 1024, 1536, 3072]) if rng.random() < 0.6 else _size(rng, 128, 3072)
    mode = "mse" if op == "store" else rng.choice(["mse", "prod"])
    bits = rng.randint(2, 4)
    case = {"op": op, "d": d, "bits": bits, "mode": mode}
    if op == "store":
        return dict(case, n=_size(rng, 100, min(200_000, 200_000 * 1536 // d)))
    terms = 2 if mode == "prod" else 1
    case["nibble"] = mode == "prod" and bits == 4 and rng.random() < 0.5
    if op == "reconstruct":
        return dict(case, n=_size(rng, 1, min(200_000, 100_000 * 1536 ** 2 // (terms * d * d))))
    case["dtype"] = rng.choice(["f32", "bf16"])
    if op == "index":
        return dict(case, n=_size(rng, 1, min(1_000_000, 2_000_000 * 1536 ** 2 // (terms * d * d))))
    case["n"] = _size(rng, 1000, min(1_000_000, 1_000_000 * 1536 // d))
    if op == "score":
        return dict(case, nq=_size(rng, 1, min(256, 64_000_000 // case["n"])))
    case["nq"] = _size(rng, 1, min(10_000, int(4e12 / (case["n"] * d * terms))))
    return dict(case, k=rng.choice([1, 10, 100]))


# ------------------------------------------------------------------------------------------ what a program has in hand

_plans = {}


def _plan(d, bits, mode, nibble=False, seed=PLAN_SEED):
    """The index's global parameters (rotation, projection, codebook), made once per program as they are once per index."""
    key = (d, bits, mode, nibble, seed)
    if key not in _plans:
        prod = mode == "prod"
        cent, _ = tq.tq_codebook(d, bits - 1 if prod else bits)
        plan = tq.Plan(d, bits, tq.TQ_PROD if prod else tq.TQ_MSE, tq.tq_rotation(d, seed),
                       tq.tq_rotation(d, seed + 1, tq.TQ_GAUSSIAN) if prod else None, cent)
        if nibble:
            plan.set_layout(tq.TQ_LAYOUT_NIBBLE)
        _plans[key] = plan
    return _plans[key]


def _bytes(count):
    return torch.empty(max(int(count), 256), dtype=torch.uint8, device="cuda")


def _embeddings(n, d, seed):
    """Unit vectors of decaying spectrum around a shared mean: the law of the repository's embedding workloads."""
    g = torch.Generator(device="cuda").manual_seed(int(seed))
    lam = torch.arange(1, d + 1, dtype=torch.float32, device="cuda").pow(-0.4)
    mean = torch.randn(d, device="cuda", generator=torch.Generator(device="cuda").manual_seed(17))
    mean *= 0.3 / mean.norm()
    x = torch.empty((n, d), dtype=torch.float32, device="cuda")
    for r in range(0, n, 131072):
        w = torch.randn((min(131072, n - r), d), generator=g, dtype=torch.float32, device="cuda")
        w *= lam
        w /= w.norm(dim=1, keepdim=True)
        w += mean
        w /= w.norm(dim=1, keepdim=True)
        x[r:r + w.shape[0]] = w
    return x


def _cast(x, dtype):
    return x.to(torch.bfloat16) if dtype == "bf16" else x


def _code_arrays(plan, n):
    prod = plan.mode == tq.TQ_PROD
    return {"idx": torch.zeros((n, plan.idx_row_bytes), dtype=torch.uint8, device="cuda"),
            "qjl": torch.zeros((n, plan.qjl_row_bytes), dtype=torch.uint8, device="cuda") if prod else None,
            "gamma": torch.zeros(n, device="cuda") if prod else None,
            "norms": torch.zeros(n, device="cuda")}


def _quantize(plan, x, codes, scratch):
    if plan.mode == tq.TQ_PROD:
        tq.tq_quantize_prod(plan, x, codes["idx"], codes["qjl"], codes["gamma"], codes["norms"], scratch)
    else:
        tq.tq_quantize_mse(plan, x, codes["idx"], codes["norms"], scratch)


def _indexed(plan, n, seed):
    """Codes of n vectors, quantised a block at a time (the vectors themselves are not kept)."""
    codes = _code_arrays(plan, n)
    block = min(n, 131072)
    scratch = _bytes(tq.tq_workspace_bytes(plan, tq.TQ_OP_QUANTIZE, block))
    for k, r in enumerate(range(0, n, block)):
        part = {name: v[r:r + block] if v is not None else None for name, v in codes.items()}
        _quantize(plan, _embeddings(min(block, n - r), plan.d, seed * 1009 + k), part, scratch)
    return codes


def _cache_plans(case):
    """(key plan, value plan) of the two channel groups: keys keep inner products (prod), values reconstruct (mse)."""
    return [(_plan(GROUP, b, "prod", seed=72 + 4 * g), _plan(GROUP, b, "mse", seed=74 + 4 * g))
            for g, b in enumerate((case["high_bits"], case["low_bits"]))]


def _keys_or_values(heads, tokens, g, outlier):
    """[heads, tokens, 128] of N(0, 1), eight channels of a head ten times as large."""
    x = torch.randn((heads, tokens, HEAD_DIM), generator=g, device="cuda")
    scale = torch.ones((heads, 1, HEAD_DIM), device="cuda")
    scale.scatter_(2, outlier[:, None, :8], 10.0)
    return (x * scale).to(torch.bfloat16)


def _cache(case, seed, tokens):
    """A compressed cache of `tokens` tokens, the groups as tq_attend_decode takes them, and what was written to it."""
    heads = case["heads"]
    g = torch.Generator(device="cuda").manual_seed(int(seed))
    # channels of a head in an order of its own: the first 64 are the group with more bits, the outliers among them
    order = torch.stack([torch.randperm(HEAD_DIM, generator=g, device="cuda") for _ in range(heads)])
    K, V = _keys_or_values(heads, tokens, g, order), _keys_or_values(heads, tokens, g, order)
    groups, parts = [], []
    for k, (pk, pv) in enumerate(_cache_plans(case)):
        channels = order[:, GROUP * k:GROUP * (k + 1)].sort(dim=1).values
        at = channels[:, None, :].expand(heads, tokens, GROUP)
        kc, vc = _code_arrays(pk, heads * tokens), _code_arrays(pv, heads * tokens)
        need = max(tq.tq_workspace_bytes(p, tq.TQ_OP_QUANTIZE, heads * tokens) for p in (pk, pv))
        parts.append({"pk": pk, "pv": pv, "xk": K.gather(2, at).reshape(-1, GROUP), "xv": V.gather(2, at).reshape(-1, GROUP),
                      "kc": kc, "vc": vc, "scratch": _bytes(need)})
        groups.append({"plan_k": pk, "plan_v": pv, "k_idx": kc["idx"], "k_qjl": kc["qjl"], "k_gamma": kc["gamma"],
                       "k_norms": kc["norms"], "v_idx": vc["idx"], "v_norms": vc["norms"],
                       "k_channels": channels.to(torch.int32).contiguous(), "v_channels": channels.to(torch.int32).contiguous()})
    return groups, parts, g


def prepare(case, seed):
    op = case["op"]
    if op == "prefill":
        _, parts, _ = _cache(case, seed, case["tokens"])
        return {"op": op, "parts": parts}
    if op == "decode":
        heads, tokens = case["heads"], case["tokens"]
        groups, parts, g = _cache(case, seed, tokens)
        for p in parts:
            _quantize(p["pk"], p["xk"], p["kc"], p["scratch"])
            _quantize(p["pv"], p["xv"], p["vc"], p["scratch"])
        codes = ("k_idx", "k_qjl", "k_gamma", "k_norms", "v_idx", "v_norms")
        written = [gr[name].view(heads, tokens, -1)[:, tokens - 1] for gr in groups for name in codes]
        new = lambda rows: torch.randn((rows, HEAD_DIM), generator=g, device="cuda").to(torch.bfloat16)  # noqa: E731
        return {"op": op, "groups": groups, "heads": heads, "tokens": tokens, "q_per_kv": case["q_per_kv"], "K": new(heads), "V": new(heads),
                "Q": new(heads * case["q_per_kv"]), "out": torch.zeros((heads * case["q_per_kv"], HEAD_DIM), device="cuda"),
                "workspace": _bytes(tq.tq_attend_decode_workspace_bytes(len(groups), heads, tokens, GROUP)), "written": written}
    d, n = case["d"], case["n"]
    plan = _plan(d, case["bits"], case["mode"], case.get("nibble", False))
    state = {"op": op, "plan": plan, "n": n}
    if op == "index":
        return dict(state, x=_cast(_embeddings(n, d, seed), case["dtype"]), codes=_code_arrays(plan, n),
                    scratch=_bytes(tq.tq_workspace_bytes(plan, tq.TQ_OP_QUANTIZE, n)))
    state["codes"] = _indexed(plan, n, seed)
    if op == "store":
        return dict(state, lengths=tq.tq_entropy_lengths(d, case["bits"], tq.tq_codebook(d, case["bits"])[0]),
                    segment=torch.zeros(n * (plan.idx_row_bytes + d // 32 + 8), dtype=torch.uint8, device="cuda"),
                    back=torch.zeros_like(state["codes"]["idx"]))
    if op == "reconstruct":
        return dict(state, x=torch.zeros((n, d), device="cuda"))
    nq = case["nq"]
    state["q"] = _cast(_embeddings(nq, d, seed + 500_009), case["dtype"])
    if op == "score":
        return dict(state, scores=torch.zeros((nq, n), device="cuda"), workspace=_bytes(tq.tq_workspace_bytes(plan, tq.TQ_OP_SCORE, n, nq)))
    k = case["k"]
    return dict(state, k=k, scores=torch.zeros((nq, k), device="cuda"), ids=torch.zeros((nq, k), dtype=torch.int32, device="cuda"),
                workspace=_bytes(tq.tq_workspace_bytes(plan, tq.TQ_OP_TOPK, n, nq, k)))


# ------------------------------------------------------------------------------------------ one pass

def run(s):
    op = s["op"]
    if op == "decode":
        tq.tq_kv_append(s["groups"], s["heads"], s["tokens"], s["tokens"] - 1, s["K"], s["V"])
        tq.tq_attend_decode(s["groups"], s["heads"], s["tokens"], s["q_per_kv"], s["Q"], 1.0 / math.sqrt(HEAD_DIM), s["out"], s["workspace"])
        return [s["out"]] + s["written"]
    if op == "prefill":
        for p in s["parts"]:
            _quantize(p["pk"], p["xk"], p["kc"], p["scratch"])
            _quantize(p["pv"], p["xv"], p["vc"], p["scratch"])
        return [[p["kc"], p["vc"]] for p in s["parts"]]
    c = s["codes"]
    if op == "index":
        _quantize(s["plan"], s["x"], c, s["scratch"])
        return c
    if op == "search":
        tq.tq_topk(s["plan"], s["q"], s["n"], c["idx"], c["qjl"], c["gamma"], c["norms"], s["k"], s["scores"], s["ids"], s["workspace"])
        return [s["scores"], s["ids"]]
    if op == "score":
        tq.tq_score(s["plan"], s["q"], s["n"], c["idx"], c["qjl"], c["gamma"], c["norms"], s["scores"], s["workspace"])
        return s["scores"]
    if op == "reconstruct":
        tq.tq_dequantize(s["plan"], s["n"], c["idx"], c["qjl"], c["gamma"], c["norms"], s["x"])
        return s["x"]
    packed, offsets = tq.tq_entropy_pack(s["plan"], s["lengths"], s["n"], c["idx"])
    s["segment"][:packed.numel()] = packed             # its place in the segment that is written out
    tq.tq_entropy_unpack(s["plan"], s["lengths"], s["n"], packed, offsets, s["back"])
    return [s["segment"], offsets, s["back"]]


# ------------------------------------------------------------------------------------------ what a pass cannot do without

def _row_bytes(d, bits, mode):
    """Bytes of one vector's codes and scalars."""
    if mode == "prod":
        return tq.tq_idx_row_bytes(d, bits - 1) + tq.tq_qjl_row_bytes(d) + 8
    return tq.tq_idx_row_bytes(d, bits) + 4


def work(case):
    op = case["op"]
    if op in ("decode", "prefill"):
        heads, tokens = case["heads"], case["tokens"]
        bits = (case["high_bits"], case["low_bits"])
        cache = heads * tokens * sum(_row_bytes(GROUP, b, "prod") + _row_bytes(GROUP, b, "mse") for b in bits)
        matrices = len(bits) * 3 * GROUP * GROUP * 4                       # rotations of both sides, projection of the keys
        if op == "prefill":   # rotation of keys and values, projection of the keys' residuals
            return {"bytes": 2 * 2 * heads * tokens * HEAD_DIM + cache + matrices, "flops": 2 * 3 * len(bits) * heads * tokens * GROUP * GROUP}
        q = heads * case["q_per_kv"]
        # per token and query: the centroid sum and the sign sum of the key, the sum over the values
        flops = 2 * q * tokens * HEAD_DIM * 3 + 2 * 3 * len(bits) * (q + heads) * GROUP * GROUP
        return {"bytes": cache + matrices + q * HEAD_DIM * (2 + 4) + 2 * heads * HEAD_DIM * 2, "flops": flops}
    d, n, terms = case["d"], case["n"], 2 if case["mode"] == "prod" else 1
    codes, matrices = n * _row_bytes(d, case["bits"], case["mode"]), terms * d * d * 4
    if op == "store":   # index rows read, coded (about 0.97 of their bits) into the segment, read again and written back; the offsets too
        rows = n * tq.tq_idx_row_bytes(d, case["bits"])
        return {"bytes": rows * (1 + 3 * 0.97 + 1) + 2 * 8 * n, "flops": 0}
    wide = 2 if case.get("dtype") == "bf16" else 4
    if op == "index":
        return {"bytes": n * d * wide + codes + matrices, "flops": 2 * terms * n * d * d}
    if op == "reconstruct":
        return {"bytes": codes + n * d * 4 + matrices, "flops": 2 * terms * n * d * d}
    nq = case["nq"]
    out = nq * n * 4 if op == "score" else nq * case["k"] * 8
    return {"bytes": codes + matrices + nq * d * wide + out, "flops": 2 * terms * nq * d * (n + d)}


def tolerance(case):
    op = case["op"]
    if op == "store":
        return "exact"
    if op in ("index", "prefill"):
        # a rotated coordinate within rounding (1e-7) of a decision boundary, or a projected one of zero, may go either
        # way; with it go that row's later signs: at most one byte in a thousand
        return {"rel": 1e-5, "max": 4e-4, "differ": 1e-3}
    if op == "search":
        return {"rel": 1e-5, "differ": 1e-3}          # neighbours whose scores agree in the last bits may change places
    return {"rel": 1e-5}
