"""The work that a user of this library has it do, as measurable cases.

Five operations, each through the public binding (``paper_2506_11498_b200.lrsa``):
  train    one post-training step of an attention layer: score/select, forward, backward
  prefill  score/select and forward of a whole prompt (inference, or evaluation of a sequence)
  score    score/select alone (the selection made ahead of the attention, on its own stream)
  append   a prompt enters the condensed KV cache, in one call or in pieces (chunked prefill)
  step     one generated token: its key and value enter the cache, its query attends over it

``listed`` holds a fixed set of them; ``draw`` gives more of the same ranges.
"""
import math

import torch

from paper_2506_11498_b200 import lrsa


def _case(name, op, heads, d, N, L, K, S, B=1, values="normal", **kw):
    Hq, Hkv = heads
    case = {"name": name, "op": op, "B": B, "Hq": Hq, "Hkv": Hkv, "d": d, "N": N, "L": L, "K": K, "S": S,
            "values": values, "ndp": 1, "ddof": 1, "residual": False, "seqs": "", "piece": 0}
    case.update(kw)
    return case


def listed():
    return [
        # One token generated with a short context on a small multi-head layer: the smallest call there is.
        _case("step_4k_mha_d64", "step", (8, 8), 64, 3583, 512, 128, 16),
        # One token generated at 32K on the 7B-shaped GQA layer, batch 1 (interactive use).
        _case("step_32k_gqa7", "step", (28, 4), 128, 31743, 1024, 256, 4, values="channel_offset"),
        # The same layer serving sixteen sequences at once (throughput-oriented generation).
        _case("step_32k_gqa7_b16", "step", (28, 4), 128, 31743, 1024, 256, 4, B=16, values="channel_offset"),
        # A 32K prompt enters the cache in one call.
        _case("append_32k_gqa7", "append", (28, 4), 128, 32768, 1024, 256, 4, values="channel_offset"),
        # A short prompt of odd length: the attention work is small, launches count.
        _case("prefill_1777_gqa7", "prefill", (28, 4), 128, 1777, 512, 128, 4, values="channel_offset"),
        # Evaluation of a 64K sequence.
        _case("prefill_64k_gqa7", "prefill", (28, 4), 128, 65536, 2048, 512, 4, values="channel_offset"),
        # The selection alone at the 32K post-training shape.
        _case("score_32k_gqa7", "score", (28, 4), 128, 32768, 1024, 256, 4, values="channel_offset"),
        # The smallest training configuration: 4K tokens, multi-head, head_dim 64.
        _case("train_4k_mha_d64", "train", (8, 8), 64, 4096, 512, 128, 16),
        # The 32K post-training step (one layer of a 7B-shaped GQA model).
        _case("train_32k_gqa7", "train", (28, 4), 128, 32768, 1024, 256, 4, values="channel_offset"),
        # The same 32K row packed with eight ragged sequences, as a data loader packs post-training data.
        _case("train_32k_packed8", "train", (28, 4), 128, 32768, 1024, 256, 4, values="channel_offset",
              seqs="9001,1337,7777,402,5003,3130,4099,2019"),
        # A ragged length with short windows, half of the tokens kept, the previous window compressed too, and the
        # more accurate dK (the rounding remainder of O handed from forward to backward).
        _case("train_20k_l256_r2_residual", "train", (32, 8), 128, 19777, 256, 128, 4, ndp=0, ddof=0, residual=True),
        # The largest configuration: two sequences of 128K tokens with salient keys.
        _case("train_128k_b2_gqa4", "train", (32, 8), 128, 131072, 4096, 1024, 4, B=2, values="salient"),
    ]


def draw(rng):
    op = rng.choice(("train", "train", "train", "prefill", "prefill", "score", "append", "append", "step", "step", "step"))
    heads, d = rng.choice((((8, 8), 64), ((16, 2), 64), ((28, 4), 128), ((28, 4), 128), ((32, 8), 128)))
    lo, hi = {"train": (900, 65536), "prefill": (300, 131072), "score": (4096, 131072), "append": (1500, 65536),
              "step": (1000, 131072)}[op]
    N = int(math.exp(rng.uniform(math.log(lo), math.log(hi))))
    lags = [L for L in (256, 333, 512, 1000, 1024, 2048, 4096) if L <= max(256, N // 3)]
    L = rng.choice(lags)
    K = max(1, L // rng.choice((2, 4, 8, 16)))
    S = rng.choice((0, 4, 16))
    case = _case("", op, heads, d, N, L, K, S, values=rng.choice(("normal", "channel_offset")))
    del case["name"]
    if op == "step":
        room = max(1, (2 << 20) // N)   # cached tokens of a batch: at most 2 M
        case["B"] = min(room, rng.choice((1, 1, 2, 4, 8, 16, 32)))
        if N > S and (N - 1 - S) % L == 0:
            case["N"] = N + 1           # the token that closes a window is one in L steps: not this one
    elif op == "append":
        case["piece"] = rng.choice((0, 0, 512, 2048))
        case["B"] = rng.choice((1, 1, 2, 4)) if N < 32768 else 1
    else:
        case["B"] = rng.choice((1, 1, 2)) if N < 32768 else 1
        case["ndp"] = rng.choice((1, 1, 1, 0))
        if op == "train":
            case["residual"] = rng.random() < 0.25
        if op != "score" and rng.random() < 0.3:
            cuts = sorted({0, N} | {rng.randrange(1, N) for _ in range(rng.randint(1, 7))})
            case["seqs"] = ",".join(str(b - a) for a, b in zip(cuts[:-1], cuts[1:]))
    return case


def _params(case, capacity=0):
    cu = [0]
    for n in case["seqs"].split(",") if case["seqs"] else ():
        cu.append(cu[-1] + int(n))
    return lrsa.Params(case["B"], case["Hq"], case["Hkv"], capacity or case["N"], case["d"], case["L"], case["K"], case["S"],
                       n_dense_prev=case["ndp"], std_ddof=case["ddof"], cu_seqlens=tuple(cu) if len(cu) > 1 else ())


def _normal(g, *shape):
    return torch.randn(shape, generator=g, device="cuda", dtype=torch.float32)


def _inputs(case, seed, names):
    """bf16 tensors [B, heads, N, d] with the value structure of the repository's workloads: unit normals; keys
    with per-channel offsets of standard deviation 2 (outlier channels), or one key in a hundred eight times as
    large (salient tokens)."""
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    out = {}
    for name in names:
        H = case["Hq"] if name in ("Q", "dO") else case["Hkv"]
        t = torch.empty((case["B"], H, case["N"], case["d"]), dtype=torch.bfloat16, device="cuda")
        offset = 2.0 * _normal(g, H, 1, case["d"])
        for b in range(case["B"]):
            x = _normal(g, H, case["N"], case["d"])
            if name == "K" and case["values"] == "channel_offset":
                x += offset
            if name == "K" and case["values"] == "salient":
                x = torch.where(torch.rand((H, case["N"], 1), generator=g, device="cuda") < 0.01, x * 8.0, x)
            t[b].copy_(x)
        out[name] = t
    return out


def prepare(case, seed):
    op = case["op"]
    if op in ("train", "prefill", "score"):
        p = _params(case)
        state = _inputs(case, seed, {"train": "Q K V dO", "prefill": "Q K V", "score": "K V"}[op].split())
        state.update(op=op, p=p, ws=[lrsa.new_workspace(n) for n in lrsa.lrsa_workspace_bytes(p)], residual=case["residual"])
        return state
    # a cache with room for the tokens to come, as a server allocates it
    p = _params(case, capacity=case["N"] + case["L"])
    cache = lrsa.KVCache(p)
    x = _inputs(case, seed, ("K", "V"))
    if op == "append":
        step = case["piece"] or case["N"]
        pieces = [(x["K"][:, :, i:i + step].contiguous(), x["V"][:, :, i:i + step].contiguous()) for i in range(0, case["N"], step)]
        return {"op": op, "cache": cache, "pieces": pieces}
    n = case["N"] - 1
    cache.append(x["K"][:, :, :n].contiguous(), x["V"][:, :, :n].contiguous())
    g = torch.Generator(device="cuda")
    g.manual_seed(seed + 1)
    q = _normal(g, case["B"], case["Hq"], case["d"]).bfloat16()
    return {"op": op, "cache": cache, "n": n, "k": x["K"][:, :, n:].contiguous(), "v": x["V"][:, :, n:].contiguous(), "q": q}


def run(state):
    op = state["op"]
    if op == "step":
        cache = state["cache"]
        cache.n_tokens = state["n"]          # the pass can be repeated: the token takes the same place again
        cache.append(state["k"], state["v"])
        o, lse = cache.decode(state["q"])
        return {"o": o, "lse": lse, "cache": cache.buf}
    if op == "append":
        cache = state["cache"]
        cache.n_tokens = 0
        for k, v in state["pieces"]:
            cache.append(k, v)
        return {"cache": cache.buf}
    p, ws, K, V = state["p"], state["ws"], state["K"], state["V"]
    idx, _ = lrsa.lrsa_score_select(p, K, V, workspace=ws[0])
    if op == "score":
        return {"idx": idx}
    Q = state["Q"]
    rest = torch.empty_like(Q) if state["residual"] else None
    O, LSE = lrsa.lrsa_attn_fwd(p, Q, K, V, idx, workspace=ws[1], o_residual=rest)
    if op == "prefill":
        return {"idx": idx, "O": O, "LSE": LSE}
    dQ, dK, dV = lrsa.lrsa_attn_bwd(p, Q, K, V, O, state["dO"], LSE, idx, workspace=ws[2], o_residual=rest)
    return {"idx": idx, "O": O, "LSE": LSE, "dQ": dQ, "dK": dK, "dV": dV}


def _pairs(n, L, K, S, ndp):
    """Visible (query, key) pairs of one head of a sequence of n tokens, and its scored windows."""
    S = min(S, n)
    W = (n - S) // L
    sel = max(W - 1, 0)
    pairs = S * (S + 1) // 2
    for c in range(W + (1 if n > S + W * L else 0)):
        rows = min(L, n - S - c * L)
        hist = min(max(c - ndp, 0), sel)
        pairs += rows * (S + hist * K + (c - hist) * L) + rows * (rows + 1) // 2
    return pairs, sel


def work(case):
    B, Hq, Hkv, N, d, L, K, S = (case[k] for k in ("B", "Hq", "Hkv", "N", "d", "L", "K", "S"))
    q, kv = B * Hq * N * d * 2, B * Hkv * N * d * 2      # bytes of a tensor shaped like Q, like K
    if case["op"] in ("step", "append"):
        chunk = (N - 1 - S) // L if N > S else 0
        kept = max(chunk - 1, 0)
        keys = S + kept * K + (N - S - kept * L) if N > S else N
        if case["op"] == "step":
            return {"bytes": 2 * B * Hkv * keys * d * 2 + 2 * B * Hq * d * 2 + 4 * B * Hq, "flops": 4 * d * B * Hq * keys}
        # every new row is read once; the kept rows, the rows of the ring and the positions are written
        return {"bytes": 2 * kv + 2 * B * Hkv * keys * d * 2 + 4 * B * Hkv * kept * K, "flops": 0}
    pairs = sel = 0
    for n in [int(s) for s in case["seqs"].split(",")] if case["seqs"] else [N]:
        a, b = _pairs(n, L, K, S, case["ndp"])
        pairs, sel = pairs + a, sel + b
    idx, lse = 4 * B * Hkv * sel * K, 4 * B * Hq * N
    if case["op"] == "score":
        return {"bytes": 2 * kv + idx, "flops": 0}
    flops = 4 * d * pairs * Hq * B
    nbytes = 2 * q + 2 * kv + idx + lse                   # Q, K, V in; O, LSE, idx out
    if case["residual"]:
        nbytes += q
    if case["op"] == "train":
        flops += 10 * d * pairs * Hq * B
        nbytes += 2 * q + 2 * kv                          # dO in; dQ, dK, dV out
    return {"bytes": nbytes, "flops": flops}


def tolerance(case):
    # Positions and cached rows are whole values and bytes: a score that ties with the K-th one in fp32 may fall on
    # either side when sums are taken in another order, which moves the rest of that window's list.
    if case["op"] in ("score", "append"):
        return {"rel": 0.0, "differ": 0.005}
    # Measured on the path: decode against fp64 differs by 0.0020 (2-norm) and 0.0066 (largest); forward and
    # gradients against the library's fp32 CUDA-core implementation by up to 0.0025 and 0.08 (O), 0.0053 and 0.32
    # (gradients; 0.8 in dQ where the fp32 implementation's D = rowsum(dO O) is the less accurate side).  The bf16
    # rounding of P and dS in sums that cancel sets these figures.
    if case["op"] == "step":
        return {"rel": 0.008, "max": 0.027, "differ": 0.0}
    if case["op"] == "prefill":
        return {"rel": 0.01, "max": 0.32, "differ": 0.005}
    return {"rel": 0.012, "max": 0.9, "differ": 0.005}
