"""The workloads that the attention library's speed is judged by, over the ranges in which it is used.

A case is one call, or one forward and backward pair, through the package's public entry points:

    train    forward + backward of a training step, one key/value head per query head or grouped heads
    infer    the forward alone (small-batch inference without a cache)
    prefill  a chunk of new tokens against a cache that ends with them (grouped heads)
    decode   one or a few new tokens per sequence against a cache
    ragged   training step on documents packed without padding
    padded   training step on a padded batch with one learnable bias per (sample, head)

listed() names twelve of them, from the smallest call to the longest sequence; draw() gives others
of the same ranges.
"""
import math
import random

import torch

import paper_2409_04431_b200 as sa

BF16_CODE, FP32_CODE = 0, 1


def listed():
    return [
        # the float32 path at the size its users run it: a check of one head, forward and backward
        {"name": "fp32_check", "kind": "train", "dtype": "fp32", "B": 1, "H": 1, "H_kv": 1, "N": 128, "D": 64,
         "causal": False, "alibi": False, "qk_norm": False, "std": 1.0},
        # one 224-pixel image through a ViT-B/16 layer: 197 tokens, the smallest bf16 call
        {"name": "vit_infer_b1", "kind": "infer", "dtype": "bf16", "B": 1, "H": 12, "N": 197, "D": 64},
        # the same layer in training, 32 images
        {"name": "vit_train", "kind": "train", "dtype": "bf16", "B": 32, "H": 12, "H_kv": 12, "N": 197, "D": 64,
         "causal": False, "alibi": False, "qk_norm": False, "std": 1.0},
        # high-resolution images (64 x 64 patches): long sequences without a mask, heads of 64
        {"name": "vit_highres_train", "kind": "train", "dtype": "bf16", "B": 8, "H": 12, "H_kv": 12, "N": 4096, "D": 64,
         "causal": False, "alibi": False, "qk_norm": False, "std": 1.0},
        # 1B language model, context 2048, ALiBi, heads of 64
        {"name": "lm_alibi_train", "kind": "train", "dtype": "bf16", "B": 8, "H": 16, "H_kv": 16, "N": 2048, "D": 64,
         "causal": True, "alibi": True, "qk_norm": False, "std": 1.0},
        # language model, context 4096, normalised q and k, heads of 128
        {"name": "lm_qknorm_train", "kind": "train", "dtype": "bf16", "B": 2, "H": 16, "H_kv": 16, "N": 4096, "D": 128,
         "causal": True, "alibi": False, "qk_norm": True, "std": 1.0},
        # long context, one sequence: the largest case
        {"name": "long_context_train", "kind": "train", "dtype": "bf16", "B": 1, "H": 32, "H_kv": 32, "N": 16384,
         "D": 128, "causal": True, "alibi": False, "qk_norm": False, "std": 0.5},
        # a chunk of a prompt read into the cache, four query heads per key/value head
        {"name": "gqa_prefill", "kind": "prefill", "dtype": "bf16", "B": 1, "H": 32, "H_kv": 8, "N_q": 1024, "N_k": 8192,
         "D": 128, "alibi": False},
        # generation, one sequence with a short cache: latency
        {"name": "decode_b1", "kind": "decode", "dtype": "bf16", "B": 1, "H": 32, "H_kv": 8, "N_q": 1, "N_k": 2000,
         "D": 128, "alibi": False},
        # generation, eight sequences with long caches: bandwidth
        {"name": "decode_b8_long", "kind": "decode", "dtype": "bf16", "B": 8, "H": 32, "H_kv": 8, "N_q": 1,
         "N_k": 16384, "D": 128, "alibi": False},
        # documents of different lengths packed into one row of tokens
        {"name": "ragged_train", "kind": "ragged", "dtype": "bf16", "H": 16, "H_kv": 4, "T": 16384, "docs": 16,
         "cut": 1, "D": 128, "causal": True},
        # utterances of different lengths in a padded batch, bias -log(length) learnt per sample and head
        {"name": "speech_padded_train", "kind": "padded", "dtype": "bf16", "B": 16, "H": 8, "N": 1500, "cut": 2, "D": 64},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _most_batches(most_pairs, H, N, cap):
    """Batch entries that keep B H N^2 below `most_pairs`, between 1 and `cap`."""
    return max(1, min(cap, int(most_pairs / (H * float(N) * N))))


def draw(rng):
    kind = rng.choice(["fp32", "vit_infer", "vit", "vit_highres", "lm64", "lm128", "long", "prefill", "decode", "decode",
                       "ragged", "padded"])
    if kind == "fp32":
        H = rng.randint(1, 4)
        return {"kind": "train", "dtype": "fp32", "B": rng.randint(1, 2), "H": H, "H_kv": H,
                "N": _log_int(rng, 16, 512), "D": rng.choice([64, 128]), "causal": rng.random() < 0.5, "alibi": False,
                "qk_norm": False, "std": 1.0}
    if kind == "vit_infer":
        return {"kind": "infer", "dtype": "bf16", "B": _log_int(rng, 1, 16), "H": rng.choice([6, 12, 16]),
                "N": _log_int(rng, 50, 1100), "D": 64}
    if kind in ("vit", "vit_highres"):
        H = rng.choice([6, 12, 16])
        N = _log_int(rng, 50, 1100) if kind == "vit" else _log_int(rng, 1100, 8100)
        B = min(_log_int(rng, 4, 64), _most_batches(2.0e9, H, N, 64))
        return {"kind": "train", "dtype": "bf16", "B": B, "H": H, "H_kv": H, "N": N, "D": 64, "causal": False,
                "alibi": False, "qk_norm": False, "std": 1.0}
    if kind in ("lm64", "lm128", "long"):
        H = rng.choice([8, 16, 32])
        N = _log_int(rng, 4096, 16384) if kind == "long" else _log_int(rng, 512, 4096)
        B = min(_log_int(rng, 1, 16), _most_batches(2.0e9, H, N, 16))
        H_kv = H // rng.choice([1, 1, 4])
        return {"kind": "train", "dtype": "bf16", "B": B, "H": H, "H_kv": H_kv, "N": N, "D": 64 if kind == "lm64" else 128,
                "causal": True, "alibi": rng.random() < 0.5, "qk_norm": rng.random() < 0.5, "std": 1.0}
    if kind == "prefill":
        N_q = _log_int(rng, 200, 2048)
        return {"kind": "prefill", "dtype": "bf16", "B": rng.choice([1, 2, 4]), "H": 32, "H_kv": rng.choice([4, 8, 32]),
                "N_q": N_q, "N_k": N_q + _log_int(rng, 128, 12000), "D": rng.choice([64, 128]), "alibi": rng.random() < 0.3}
    if kind == "decode":
        B, H_kv, N_k = _log_int(rng, 1, 32), rng.choice([4, 8, 32]), _log_int(rng, 200, 65536)
        B = max(1, min(B, int(2.0e6 / (H_kv * N_k))))
        return {"kind": "decode", "dtype": "bf16", "B": B, "H": 32, "H_kv": H_kv, "N_q": rng.choice([1, 1, 1, 4]),
                "N_k": N_k, "D": rng.choice([64, 128, 128]), "alibi": rng.random() < 0.3}
    if kind == "ragged":
        H = rng.choice([8, 16])
        return {"kind": "ragged", "dtype": "bf16", "H": H, "H_kv": H // rng.choice([1, 4]), "T": _log_int(rng, 4096, 32768),
                "docs": _log_int(rng, 4, 64), "cut": rng.randint(3, 10 ** 6), "D": rng.choice([64, 128]), "causal": True}
    H = rng.choice([4, 8, 16])
    return {"kind": "padded", "dtype": "bf16", "B": _log_int(rng, 4, 32), "H": H, "N": _log_int(rng, 200, 2500),
            "cut": rng.randint(3, 10 ** 6), "D": 64}


# ----------------------------------------------------------------------------- sizes


def _doc_lengths(case):
    """Lengths of the packed documents: a spread of about a factor of ten, every one at least one row."""
    r = random.Random(case["cut"])
    w = [math.exp(r.gauss(0.0, 0.8)) for _ in range(case["docs"])]
    left = case["T"] - case["docs"]
    lens = [1 + int(left * x / sum(w)) for x in w]
    lens[-1] += case["T"] - sum(lens)
    return lens


def _padded_lengths(case):
    """Valid rows of each batch entry, between a quarter of the padded length and all of it (one is full)."""
    r = random.Random(case["cut"])
    N = case["N"]
    return [N] + [r.randint(max(1, N // 4), N) for _ in range(case["B"] - 1)]


def _pairs(case):
    """(query, key) pairs that carry weight, over all query heads."""
    kind = case["kind"]
    if kind == "ragged":
        return case["H"] * sum(n * (n + 1) / 2 for n in _doc_lengths(case))
    if kind == "padded":
        return case["H"] * sum(float(n) * n for n in _padded_lengths(case))
    if kind in ("prefill", "decode"):
        n_q, n_k = case["N_q"], case["N_k"]
        return case["B"] * case["H"] * (n_q * float(n_k) - n_q * (n_q - 1) / 2)
    N = float(case["N"])
    return case["B"] * case["H"] * (N * (N + 1) / 2 if case.get("causal") else N * N)


def work(case):
    """Every input read once, every output written once; 4 D FLOP per weighted pair forward, 10 D backward."""
    kind, D = case["kind"], case["D"]
    e = 4 if case["dtype"] == "fp32" else 2
    if kind == "ragged":
        rows_q, rows_kv = case["H"] * case["T"], case["H_kv"] * case["T"]
    elif kind == "padded":
        rows_q = rows_kv = case["H"] * case["B"] * case["N"]
    elif kind in ("prefill", "decode"):
        rows_q, rows_kv = case["B"] * case["H"] * case["N_q"], case["B"] * case["H_kv"] * case["N_k"]
    else:
        rows_q = case["B"] * case["H"] * case["N"]
        rows_kv = case["B"] * case.get("H_kv", case["H"]) * case["N"]
    forward = (2 * rows_q + 2 * rows_kv) * D * e
    if kind in ("infer", "prefill", "decode"):
        return {"bytes": forward, "flops": 4.0 * D * _pairs(case)}
    # a training step reads q, k, v and dO and writes O, dQ, dK, dV
    return {"bytes": (4 * rows_q + 4 * rows_kv) * D * e, "flops": 14.0 * D * _pairs(case)}


# ----------------------------------------------------------------------------- one pass


def prepare(case, seed):
    kind, D = case["kind"], case["D"]
    dev = torch.device("cuda")
    dtype = torch.float32 if case["dtype"] == "fp32" else torch.bfloat16
    code = FP32_CODE if case["dtype"] == "fp32" else BF16_CODE
    g = torch.Generator(device=dev)
    g.manual_seed(int(seed))
    std = case.get("std", 1.0)

    def normal(b, h, n, unit_rows=False):
        x = torch.randn((b, h, n, D), generator=g, device=dev, dtype=torch.float32)
        if unit_rows:   # q, k normalisation: every row of length sqrt(D)
            x *= math.sqrt(D) / torch.linalg.vector_norm(x, dim=-1, keepdim=True)
        return x.mul_(std).to(dtype)

    def slopes(h):
        if not case.get("alibi"):
            return None
        return torch.exp2(-8.0 * torch.arange(1, h + 1, device=dev, dtype=torch.float32) / h)

    s = {"kind": kind, "scale": 1.0 / math.sqrt(D), "causal": bool(case.get("causal", kind in ("prefill", "decode")))}
    H = case["H"]
    H_kv = case.get("H_kv", H)
    s["grouped"] = H_kv != H
    s["slopes"] = slopes(H)
    if kind == "ragged":
        B, n_q, n_k = 1, case["T"], case["T"]
    elif kind in ("prefill", "decode"):
        B, n_q, n_k = case["B"], case["N_q"], case["N_k"]
    else:
        B, n_q, n_k = case["B"], case["N"], case["N"]
    s["q"] = normal(B, H, n_q, case.get("qk_norm", False))
    s["k"] = normal(B, H_kv, n_k, case.get("qk_norm", False))
    s["v"] = normal(B, H_kv, n_k)
    s["bias"] = -math.log(n_k)
    if kind in ("train", "ragged", "padded"):
        s["d_o"] = normal(B, H, n_q)
        need = sa.sigattn_bwd_workspace_bytes(B, H, n_q, D, code)
        s["workspace"] = torch.empty(need, dtype=torch.uint8, device=dev) if need else None
    if kind == "ragged":
        lens = torch.tensor(_doc_lengths(case), dtype=torch.int64)
        s["cu_seqlens"] = torch.cat([torch.zeros(1, dtype=torch.int64), lens.cumsum(0)]).to(torch.int32).to(dev)
        s["bias"] = (-lens.to(torch.float32).log())[:, None].repeat(1, H).contiguous().to(dev)
    if kind == "padded":
        lens = torch.tensor(_padded_lengths(case), dtype=torch.int32)
        s["seqlens"] = lens.to(dev)
        s["bias"] = (-lens.to(torch.float32).log())[:, None].repeat(1, H).contiguous().to(dev)
    if kind == "decode":
        need = sa.sigattn_fwd_decode_workspace_bytes(B, H, n_q, D, code)
        s["workspace"] = torch.empty(need, dtype=torch.uint8, device=dev)
        s["out"] = torch.empty_like(s["q"])
    return s


def run(s):
    kind = s["kind"]
    q, k, v, scale, bias, causal, slopes = s["q"], s["k"], s["v"], s["scale"], s["bias"], s["causal"], s["slopes"]
    if kind == "infer":
        return sa.sigattn_fwd(q, k, v, scale, bias, causal, slopes)
    if kind == "prefill":
        return sa.sigattn_fwd_nk(q, k, v, scale, bias, causal, slopes)
    if kind == "decode":
        return sa.sigattn_fwd_decode(q, k, v, scale, bias, causal, slopes, workspace=s["workspace"], out=s["out"])
    if kind == "ragged":
        o = sa.sigattn_fwd_ragged(q, k, v, s["cu_seqlens"], scale, bias, causal, slopes)
        dq, dk, dv, db = sa.sigattn_bwd_ragged(q, k, v, s["d_o"], s["cu_seqlens"], scale, bias, causal, slopes,
                                               workspace=s["workspace"])
        return {"o": o, "dq": dq, "dk": dk, "dv": dv}
    if kind == "padded":
        o = sa.sigattn_fwd_varlen(q, k, v, scale, bias, s["seqlens"], causal, slopes)
        dq, dk, dv, db = sa.sigattn_bwd_varlen(q, k, v, s["d_o"], scale, bias, s["seqlens"], causal, slopes,
                                               want_dbias=True, workspace=s["workspace"])
        return {"o": o, "dq": dq, "dk": dk, "dv": dv, "db": db}
    if s["grouped"]:
        o = sa.sigattn_fwd_gqa(q, k, v, scale, bias, causal, slopes)
        dq, dk, dv, db = sa.sigattn_bwd_gqa(q, k, v, s["d_o"], scale, bias, causal, slopes, workspace=s["workspace"])
        return {"o": o, "dq": dq, "dk": dk, "dv": dv}
    o = sa.sigattn_fwd(q, k, v, scale, bias, causal, slopes)
    dq, dk, dv = sa.sigattn_bwd(q, k, v, s["d_o"], scale, bias, causal, slopes, workspace=s["workspace"])
    return {"o": o, "dq": dq, "dk": dk, "dv": dv}


def tolerance(case):
    """About four times what the path differs from the same formula evaluated in float64: with bf16 tensors 2.4e-3
    (3.0e-3 where a result is the sum of rounded parts) in the norm and up to 5e-2 in the largest difference over the
    root mean square (weights, dS and results are rounded to bf16); with float32 ones 4.6e-7 and 3e-6."""
    if case["dtype"] == "fp32":
        return {"rel": 2e-6, "max": 1.5e-5}
    return {"rel": 1e-2, "max": 2e-1}
