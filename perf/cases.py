"""The calls that a program built on this library makes, at the sizes it makes them.

A case is a dict of plain values; `kind` says which entry points one pass goes through:

  decompress   ecco_decompress_batch over one or several tensors (compressed blocks -> fp16)
  gemv         products of compressed weight matrices with 1..8 rows of activations: one ecco_gemv per single
               matrix, one ecco_gemv_batch per group of matrices that do not depend on each other
  attn         decode attention over compressed K and V caches: ecco_attn_scores, then ecco_attn_values
  kv_compress  ecco_kv_compress of new K rows and new V rows (fp16 -> blocks)
  act          2x activation format, ecco_act_compress and ecco_act_decompress
  var          ecco_var_decompress of the variable-length container

Weights are Student-t(5) values with a lognormal scale per row, encoded by the host encoder with the least-squares pattern
choice; caches are N(0,1) with four channels of each head ten times as large, encoded by the online compressor.  A weight
tensor is filled with groups drawn at random from a pool that was encoded for it, so that large tensors are quick to make;
caches are encoded group by group.  Patterns and codebooks are calibrated once per kind of tensor, as a user does.
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

from paper_2505_06901_b200 import binding as B
from paper_2505_06901_b200 import synth
from paper_2505_06901_b200 import workloads as W

POOL_ROWS, POOL_COLS = 1024, 1024          # 8192 distinct groups per weight matrix

# A decoder layer of the 7B shape as its data dependencies let it be issued: q+k+v | o | gate+up | down.
LAYER_7B = "4096x4096+4096x4096+4096x4096|4096x4096|11008x4096+11008x4096|4096x11008"


def listed():
    return [
        # All weights of one decoder layer to fp16 in one call: what precedes library GEMMs in prefill.
        {"name": "decompress_layer", "kind": "decompress", "source": "weights",
         "tensors": "131072+131072+131072+131072+352256+352256+352256"},
        # A long-context K cache [16][8][32768][128] back to fp16 (hand-over to an attention kernel that wants fp16).
        {"name": "decompress_kv_long", "kind": "decompress", "source": "kv", "tensors": "4194304"},
        # One projection at batch 1: the smallest product of a decode step, a call of its own.
        {"name": "gemv_proj_b1", "kind": "gemv", "groups": "4096x4096", "batch": 1},
        # The seven products of a layer in a decode step, one sequence.
        {"name": "gemv_layer_b1", "kind": "gemv", "groups": LAYER_7B, "batch": 1},
        # The same for eight sequences decoded together.
        {"name": "gemv_layer_b8", "kind": "gemv", "groups": LAYER_7B, "batch": 8},
        # Decode attention, one query head per KV head, eight sequences of 4096 tokens.
        {"name": "attn_mha_4k", "kind": "attn", "batch": 8, "kv_heads": 32, "seq": 4096, "q_per_kv": 1},
        # Decode attention with grouped queries over sixteen long contexts: the largest call.
        {"name": "attn_gqa_32k", "kind": "attn", "batch": 16, "kv_heads": 8, "seq": 32768, "q_per_kv": 8},
        # Decode attention early in a conversation: few tokens, a length that divides by nothing.
        {"name": "attn_short_ragged", "kind": "attn", "batch": 2, "kv_heads": 8, "seq": 777, "q_per_kv": 4},
        # K and V rows of one new token for 32 sequences with eight KV heads: once per layer and decode step.
        {"name": "kv_append_step", "kind": "kv_compress", "groups": 256},
        # K and V rows of a prompt: eight sequences of 512 tokens, 32 heads.
        {"name": "kv_prefill", "kind": "kv_compress", "groups": 131072},
        # Activations of 4096 tokens put away and fetched again in the 2x format.
        {"name": "act_roundtrip", "kind": "act", "groups": 4096 * 64},
        # A projection kept in the variable-length container (no clipping), back to fp16.
        {"name": "var_proj", "kind": "var", "groups": 131072},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["decompress", "decompress", "gemv", "gemv", "gemv", "attn", "attn", "attn", "kv_compress", "act", "var"])
    if kind == "decompress":
        n = rng.randint(1, 4)
        total = _log_int(rng, 2000, 4_000_000)
        return {"kind": kind, "source": rng.choice(["weights", "kv"]), "tensors": "+".join(str(max(1, int(total * rng.uniform(0.3, 1.0) / n))) for _ in range(n))}
    if kind == "gemv":
        group = []
        for _ in range(rng.randint(1, 3)):
            k = 128 * _log_int(rng, 4, 224)
            n_out = min(_log_int(rng, 96, 28672), 800_000 * 128 // k)
            group.append("%dx%d" % (n_out, k))
        return {"kind": kind, "groups": "+".join(group), "batch": rng.choice([1, 1, 2, 3, 4, 5, 6, 7, 8, 8])}
    if kind == "attn":
        heads = rng.choice([1, 2, 4, 8, 8, 16, 32])
        seq = _log_int(rng, 20, 32768)
        batch = max(1, min(_log_int(rng, 1, 32), 4_000_000 // (heads * seq)))
        return {"kind": kind, "batch": batch, "kv_heads": heads, "seq": seq, "q_per_kv": rng.choice([1, 1, 2, 3, 4, 5, 6, 7, 8, 8])}
    if kind == "kv_compress":
        return {"kind": kind, "groups": _log_int(rng, 8, 400_000)}
    if kind == "act":
        return {"kind": kind, "groups": _log_int(rng, 64, 4_000_000)}
    return {"kind": kind, "groups": _log_int(rng, 1000, 131072)}


# ------------------------------------------------------------------ what a program has in hand
@functools.lru_cache(maxsize=None)
def _weight_calibration():
    return W.calibrate_weights(2, 0.02, True)


@functools.lru_cache(maxsize=None)
def _kv_calibration(heads):
    return W.calibrate_kv(3, heads)


def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _own_meta(base):
    """A tensor's own metadata (its exponent is fitted to it) with the tables of the calibration."""
    S, e, pat, cb, kp = base.tables()
    return B.ecco_meta_create(S, e, pat, cb, kp)


def _weights(n_groups, seed, i, gen):
    """(metadata image, blocks) of a weight tensor of n_groups groups on the device."""
    meta = _own_meta(_weight_calibration())
    pool, _ = B.ecco_encode_host(meta, synth.weight_matrix(POOL_ROWS, POOL_COLS, 64 * seed + i), B.SELECT_MSE, want_stats=False)
    pool = torch.from_numpy(pool).cuda().view(torch.int32)
    pick = torch.randint(0, pool.shape[0], (n_groups,), device="cuda", generator=gen)
    return B.meta_to_device(meta), pool[pick].view(torch.uint8)


def _kv_rows(rows, heads, gen):
    """N(0,1) rows [..., head, token, 128] flattened to [rows][128], four channels of each head ten times as large."""
    scale = torch.ones(heads, 128, device="cuda")
    scale.scatter_(1, torch.rand(heads, 128, device="cuda", generator=gen).argsort(1)[:, :4], 10.0)
    x = torch.empty(rows, 128, dtype=torch.float16, device="cuda")
    per_head = -(-rows // heads)
    for h in range(heads):
        part = x[h * per_head: (h + 1) * per_head]
        if len(part):
            part.copy_(torch.randn(part.shape, device="cuda", generator=gen) * scale[h])
    return x


def _kv_cache(n_groups, heads, gen):
    """(metadata image, blocks) of a cache of n_groups tokens' head vectors."""
    d_meta = B.meta_to_device(_kv_calibration(32))
    x = _kv_rows(n_groups, heads, gen)
    blocks = torch.empty(n_groups, 64, dtype=torch.uint8, device="cuda")
    B.ecco_kv_compress(d_meta, x, n_groups, blocks)
    return d_meta, blocks


def _matrices(case):
    return [[tuple(int(v) for v in m.split("x")) for m in g.split("+")] for g in case["groups"].split("|")]


def prepare(case, seed):
    gen = _generator(seed)
    kind = case["kind"]
    st = {"case": case}
    if kind == "decompress":
        items = []
        for i, n in enumerate(int(t) for t in case["tensors"].split("+")):
            d_meta, blocks = _weights(n, seed, i, gen) if case["source"] == "weights" else _kv_cache(n, 8, gen)
            items.append((d_meta, blocks, n, torch.empty(n, 128, dtype=torch.float16, device="cuda")))
        st["keep"] = items
        st["items"] = B.decompress_items(items)
        st["out"] = [it[3] for it in items]
    elif kind == "gemv":
        batch, i = case["batch"], 0
        st["calls"], st["out"], st["keep"] = [], [], []
        for group in _matrices(case):
            xs, items = {}, []
            for n_out, k in group:
                if k not in xs:
                    xs[k] = torch.randn(batch, k, device="cuda", generator=gen).half()
                d_meta, blocks = _weights(n_out * (k // 128), seed, i, gen)
                items.append((d_meta, blocks, n_out, k, xs[k], torch.empty(batch, n_out, device="cuda")))
                i += 1
            if len(items) == 1:
                size = B.ecco_gemv_workspace_bytes(items[0][2], items[0][3], batch)
                call = items[0]
            else:
                size = B.ecco_gemv_batch_workspace_bytes(items, batch)
                call = B.gemv_items(items)
            st["calls"].append((call, torch.empty(size, dtype=torch.uint8, device="cuda"), size))
            st["keep"].append(items)
            st["out"] += [it[5] for it in items]
    elif kind == "attn":
        b, h, s, q = case["batch"], case["kv_heads"], case["seq"], case["q_per_kv"]
        st["k_meta"], st["k"] = _kv_cache(b * h * s, h, gen)
        st["v_meta"], st["v"] = _kv_cache(b * h * s, h, gen)
        st["q"] = torch.randn(b, h * q, 128, device="cuda", generator=gen).half()
        st["scores"] = torch.empty(b, h * q, s, device="cuda")
        st["out"] = torch.empty(b, h * q, 128, device="cuda")
        st["ws_bytes"] = B.ecco_attn_values_workspace_bytes(b, h, s, q)
        st["ws"] = torch.empty(st["ws_bytes"], dtype=torch.uint8, device="cuda")
    elif kind == "kv_compress":
        n = case["groups"]
        st["meta"] = [B.meta_to_device(_kv_calibration(32)) for _ in range(2)]
        st["x"] = [_kv_rows(n, 8, gen) for _ in range(2)]
        st["blocks"] = [torch.empty(n, 64, dtype=torch.uint8, device="cuda") for _ in range(2)]
    elif kind == "act":
        n = case["groups"]
        st["x"] = (torch.randn(n, 64, device="cuda", generator=gen) * torch.exp(0.5 * torch.randn(n, 1, device="cuda", generator=gen))).half()
        st["blocks"] = torch.empty(n, 64, dtype=torch.uint8, device="cuda")
        st["out"] = torch.empty(n, 64, dtype=torch.float16, device="cuda")
    else:
        n = case["groups"]
        meta = _own_meta(_weight_calibration())
        rows = -(-n // 32)
        w = synth.weight_matrix(rows, 4096, seed).reshape(-1, 128)[:n]
        stream, index, _ = B.ecco_var_encode_host(meta, w, B.SELECT_MSE)
        st["meta"] = B.meta_to_device(meta)
        st["stream"] = torch.from_numpy(stream).cuda()
        st["index"] = torch.from_numpy(np.ascontiguousarray(index)).cuda()
        st["out"] = torch.empty(n, 128, dtype=torch.float16, device="cuda")
    return st


# ------------------------------------------------------------------ one pass
def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind == "decompress":
        B.ecco_decompress_batch(st["items"])
        return st["out"]
    if kind == "gemv":
        batch = case["batch"]
        for call, ws, size in st["calls"]:
            if isinstance(call, tuple):
                d_meta, blocks, n_out, k, x, y = call
                B.ecco_gemv(d_meta, blocks, n_out, k, x, batch, y, ws, size)
            else:
                B.ecco_gemv_batch(call, batch, ws, size)
        return st["out"]
    if kind == "attn":
        b, h, s, q = case["batch"], case["kv_heads"], case["seq"], case["q_per_kv"]
        B.ecco_attn_scores(st["k_meta"], st["k"], b, h, s, q, st["q"], 128 ** -0.5, st["scores"])
        B.ecco_attn_values(st["v_meta"], st["v"], b, h, s, q, st["scores"], st["out"], st["ws"], st["ws_bytes"])
        return [st["scores"], st["out"]]
    if kind == "kv_compress":
        for meta, x, blocks in zip(st["meta"], st["x"], st["blocks"]):
            B.ecco_kv_compress(meta, x, case["groups"], blocks)
        return st["blocks"]
    if kind == "act":
        B.ecco_act_compress(st["x"], case["groups"], st["blocks"])
        B.ecco_act_decompress(st["blocks"], case["groups"], st["out"])
        return [st["blocks"], st["out"]]
    B.ecco_var_decompress(st["meta"], st["stream"], st["index"], case["groups"], st["out"])
    return st["out"]


# ------------------------------------------------------------------ what a pass cannot do without
def work(case):
    kind = case["kind"]
    if kind == "decompress":                               # 64 B in, 256 B out, one product per value
        n = sum(int(t) for t in case["tensors"].split("+"))
        return {"bytes": 320 * n, "flops": 128 * n}
    if kind == "gemv":
        size = flops = 0
        for group in _matrices(case):
            size += sum(2 * case["batch"] * k for k in {k for _, k in group})
            for n_out, k in group:
                size += n_out * (k // 128) * 64 + 4 * case["batch"] * n_out
                flops += 2 * case["batch"] * n_out * k
        return {"bytes": size, "flops": flops}
    if kind == "attn":                                     # K and V blocks; scores written, then read; q and out
        rows = case["batch"] * case["kv_heads"]
        tokens, q = rows * case["seq"], case["q_per_kv"]
        return {"bytes": 128 * tokens + 8 * q * tokens + rows * q * 128 * 6, "flops": 4 * 128 * q * tokens}
    if kind == "kv_compress":
        return {"bytes": 2 * 320 * case["groups"], "flops": 2 * 128 * case["groups"]}
    if kind == "act":                                      # 128 B -> 64 B -> 128 B
        return {"bytes": (192 + 192) * case["groups"], "flops": 4 * 64 * case["groups"]}
    return {"bytes": (63 + 4 + 256) * case["groups"], "flops": 128 * case["groups"]}


def tolerance(case):
    """Decoded values and encoded blocks are defined bit by bit.  Products are fp32 sums of exact fp16 products (and, for
    the attention output, of probabilities held to 22 bits): four times the largest difference seen between this path and
    64-bit sums over the decoded values, 1.7e-6 and 5e-6 for products, 2.5e-6 and 3.5e-5 for attention."""
    if case["kind"] == "gemv":
        return {"rel": 7e-6, "max": 2e-5}
    if case["kind"] == "attn":
        return {"rel": 1e-5, "max": 1.4e-4}
    return "exact"
