"""The work that users of the codec have it do, as cases that can be timed and compared.

Every case goes through the public entry points of ``paper_2508_19263_b200.binding``: histogram, codebook, compress
and decompress of single tensors and of whole sets of tensors, random access to chunks, delta checkpoints, K/V pages
coded with a static dictionary, block-scale bytes.  Inputs are made on the GPU by ``workloads`` (Gaussian weights and
K/V caches in the formats the codec takes); containers and tensors are bytes, so results are compared exactly.

A case has a kind and a pass:

  kind    tensor    one weight matrix, the per-tensor calls
          weights   all tensors of a decoder stack (projections, feed-forward, norms), the batched calls
          delta     the same for two consecutive BF16 checkpoints, coded as their XOR
          pages     K and V pages of a serving step, one dictionary per layer and kind
          scales    the E8M0 block scales of a stack's MXFP4 form
          read      a range of chunks out of one K/V tensor's container
  pass    encode (histogram, codebooks, compress), decode (decompress), both
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2508_19263_b200 import binding as zc
from paper_2508_19263_b200 import workloads as wl

DEVICE = "cuda:0"
FORMATS = {"bf16": zc.FMT_BF16, "fp8": zc.FMT_FP8_E4M3, "fp4": zc.FMT_FP4_E2M1, "e5m2": zc.FMT_FP8_E5M2, "scale": zc.FMT_SCALE_U8}
POLICIES = {"auto": zc.POLICY_AUTO, "all": zc.POLICY_HUFF_ALL, "static": zc.POLICY_STATIC}
BYTES_PER_ELEM = {"bf16": 2.0, "fp8": 1.0, "fp4": 0.5, "e5m2": 1.0, "scale": 1.0}
# container bytes per input byte, about: what the formats come to on these inputs
RATIO = {"bf16": 0.68, "fp8": 0.84, "fp4": 1.0, "e5m2": 0.73, "scale": 0.19}
KV_RATIO = {"bf16": 0.72, "fp8": 0.91}
KV_HEADS, HEAD_DIM = 8, 128


def listed():
    return [
        # Random access while serving: one sequence's 64 KiB of a stored K cache tensor is read back.  Pure latency.
        dict(name="read_kv_bf16", kind="read", fmt="bf16", chunk_kib=4, tokens=4096, first=777, count=16),
        # One small FP8 matrix on its own in the largest chunks, both streams coded: a plugin that compresses
        # tensors as they come, a few per step.  Latency of the calls and of the longest serial unit.
        dict(name="encode_tensor_fp8_64k", kind="tensor", fmt="fp8", chunk_kib=64, rows=1024, cols=1024, policy="all", **{"pass": "encode"}),
        dict(name="decode_tensor_fp8_64k", kind="tensor", fmt="fp8", chunk_kib=64, rows=1024, cols=1024, policy="all", **{"pass": "decode"}),
        # A serving step that evicts K/V pages and fetches as many back: 32 layers' K and V of 257 tokens (ragged
        # against every chunk size), coded with dictionaries made ahead of time, no histogram in the step.
        dict(name="pages_kv_bf16", kind="pages", fmt="bf16", chunk_kib=4, layers=32, tokens=257, policy="static", **{"pass": "both"}),
        # A model or checkpoint in BF16 at the default chunk size: four 8B-shaped decoder layers, norms included.
        dict(name="encode_weights_bf16", kind="weights", fmt="bf16", chunk_kib=4, layers=4, hidden=4096, ffn=14336, policy="auto", **{"pass": "encode"}),
        dict(name="decode_weights_bf16", kind="weights", fmt="bf16", chunk_kib=4, layers=4, hidden=4096, ffn=14336, policy="auto", **{"pass": "decode"}),
        # The same in FP8 E4M3 with per-row scales: half the bytes, as many symbols per byte, longer codes.
        dict(name="encode_weights_fp8", kind="weights", fmt="fp8", chunk_kib=4, layers=4, hidden=4096, ffn=14336, policy="auto", **{"pass": "encode"}),
        dict(name="decode_weights_fp8", kind="weights", fmt="fp8", chunk_kib=4, layers=4, hidden=4096, ffn=14336, policy="auto", **{"pass": "decode"}),
        # Consecutive checkpoints of a fine-tuning run, half of every tensor's rows untouched: XOR form, both streams
        # coded, constant chunks among them.
        dict(name="encode_delta_bf16", kind="delta", fmt="bf16", chunk_kib=4, layers=2, hidden=4096, ffn=14336, frozen=0.5, policy="auto", **{"pass": "encode"}),
        dict(name="decode_delta_bf16", kind="delta", fmt="bf16", chunk_kib=4, layers=2, hidden=4096, ffn=14336, frozen=0.5, policy="auto", **{"pass": "decode"}),
        # Models kept for distribution, where ratio matters more: larger chunks, written once and read back.
        dict(name="archive_fp8_16k", kind="weights", fmt="fp8", chunk_kib=16, layers=2, hidden=4096, ffn=11008, policy="auto", **{"pass": "both"}),
        # The part of an FP4 model that compresses: many tensors of about a megabyte of block scales.
        dict(name="scales_fp4", kind="scales", fmt="scale", chunk_kib=4, layers=4, hidden=4096, ffn=14336, policy="auto", **{"pass": "both"}),
    ]


def _log_int(rng, lo, hi):
    """An integer spread evenly over the logarithm of its range, odd values among them."""
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    """One more case of the same ranges."""
    kind = rng.choice(["read", "tensor", "tensor", "pages", "weights", "weights", "delta", "scales"])
    case = dict(kind=kind, chunk_kib=rng.choice([1, 2, 3, 4, 4, 4, 6, 8, 12, 16, 24, 32, 64]))
    if kind == "read":
        tokens = _log_int(rng, 64, 16384)
        case.update(fmt=rng.choice(["bf16", "fp8"]), tokens=tokens)
        total = -(-int(tokens * KV_HEADS * HEAD_DIM * BYTES_PER_ELEM[case["fmt"]]) // (1024 * case["chunk_kib"]))
        case["count"] = _log_int(rng, 1, min(total, 512))
        case["first"] = rng.randrange(total - case["count"] + 1)
        return case
    case["pass"] = rng.choice(["encode", "decode", "both"])
    case["policy"] = rng.choice(["auto", "auto", "auto", "all"])
    if kind == "tensor":
        fmt = rng.choice(["bf16", "fp8", "fp4", "e5m2", "scale"])
        cols = _log_int(rng, 64, 8192)
        if fmt in ("fp4", "scale"):
            cols = 32 * -(-cols // 32)                          # MX blocks of 32 along the row
        case.update(fmt=fmt, rows=_log_int(rng, 1, 4096), cols=cols)
    elif kind == "pages":
        case.update(fmt=rng.choice(["bf16", "fp8"]), layers=rng.randint(1, 32), tokens=_log_int(rng, 16, 1024), policy="static")
    else:
        fmt = {"weights": rng.choice(["bf16", "fp8", "fp4", "e5m2"]), "delta": "bf16", "scales": "scale"}[kind]
        top = 4096 if 4 <= case["chunk_kib"] <= 8 else 2048
        hidden = 32 * _log_int(rng, 8, top // 32)
        case.update(fmt=fmt, layers=rng.randint(1, 4 if kind == "scales" else 2), hidden=hidden,
                    ffn=32 * int(hidden * rng.uniform(2.5, 3.5) / 32))
        if kind == "delta":
            case["frozen"] = rng.choice([0.0, 0.25, 0.5, 0.75])
    return case


# ---- inputs -------------------------------------------------------------------------------------

def _specs(case, seed):
    """The tensors of a decoder stack: projections with a quarter of the heads for K and V, feed-forward, two norms."""
    h, f, out = case["hidden"], case["ffn"], []
    kv = max(32, h // 4)
    for layer in range(case["layers"]):
        std = 0.02 / math.sqrt(layer + 1)
        for shape in ((h, h), (kv, h), (kv, h), (h, h), (f, h), (f, h), (h, f), (1, h), (1, h)):
            out.append(wl.TensorSpec(f"layers.{layer}.{len(out)}", shape, std, 1000 * seed + len(out)))
    return out


def _arena(sizes):
    """One zeroed buffer and a view per size, each on a 256-byte boundary: how a program keeps a set of tensors."""
    starts, at = [], 0
    for n in sizes:
        starts.append(at)
        at += -(-max(n, 1) // 256) * 256
    buf = torch.zeros(at, dtype=torch.uint8, device=DEVICE)
    return buf, [buf[s: s + n] for s, n in zip(starts, sizes)]


def _inputs(case, seed):
    """Element bytes, element counts and (delta) base tensors."""
    fmt, kind = FORMATS[case["fmt"]], case["kind"]
    if kind == "tensor":
        spec = wl.TensorSpec("tensor", (case["rows"], case["cols"]), 0.02, 1000 * seed)
        data, n, _ = wl.make_weight(spec, fmt, DEVICE)
        return [data], [n], None
    if kind in ("pages", "read"):
        layers = case["layers"] if kind == "pages" else 1
        made = [wl.kv_cache_tensor(fmt, 1000 * seed + layer, which, DEVICE, batch=1, kv_heads=KV_HEADS, seq=case["tokens"], head_dim=HEAD_DIM)
                for layer in range(layers) for which in (0, 1)[: 2 if kind == "pages" else 1]]
        return [d for d, _ in made], [n for _, n in made], None
    if kind == "delta":
        made = [wl.checkpoint_pair(s, DEVICE, frozen_rows=case["frozen"]) for s in _specs(case, seed)]
        return [later for later, _, _ in made], [n for _, _, n in made], [base for _, base, _ in made]
    made = [wl.make_weight(s, fmt, DEVICE) for s in _specs(case, seed)]
    return [d for d, _, _ in made], [n for _, n, _ in made], None


def prepare(case, seed):
    fmt, chunk = FORMATS[case["fmt"]], 1024 * case["chunk_kib"]
    policy = POLICIES[case.get("policy", "auto")]
    ins, counts, bases = _inputs(case, seed)
    plans = [zc.plan(fmt, n, chunk) for n in counts]
    out_arena, outs = _arena([p.max_compressed_bytes for p in plans])
    s = dict(case=case, policy=policy, plans=plans, ins=ins, bases=bases, out_arena=out_arena, outs=outs)
    s["hists"] = torch.zeros((len(plans), 2, 256), dtype=torch.int64, device=DEVICE)
    s["hist_batch"] = zc.HistogramBatch(plans, ins, bases)
    s["enc"] = zc.CompressBatch(plans, ins, outs, bases)
    s["ws"] = torch.zeros(max(s["enc"].workspace_bytes, max(p.workspace_bytes for p in plans)), dtype=torch.uint8, device=DEVICE)
    if case["kind"] == "pages":
        # a dictionary per layer and kind, from an earlier page of the same cache
        earlier, n_earlier, _ = _inputs(dict(case, tokens=64), seed)
        s["dicts"] = [zc.Dictionary(p, zc.histogram(zc.plan(fmt, n, chunk), t).cpu().numpy(), 0.05)
                      for p, t, n in zip(plans, earlier, n_earlier)]
        s["books"] = [d.codebook for d in s["dicts"]]
    if case["kind"] == "read":
        nbytes = _encode(s)["sizes"]
        p = plans[0]
        s["comp_bytes"] = int(nbytes[0])
        s["back"] = torch.zeros(min(case["count"] * chunk, p.input_bytes - case["first"] * chunk), dtype=torch.uint8, device=DEVICE)
        return s
    if case["pass"] != "encode":
        s["back_arena"], s["backs"] = _arena([p.input_bytes for p in plans])
        s["sizes"] = _encode(s)["sizes"]
        s["dec"] = zc.DecompressBatch(plans, outs, s["sizes"], s["backs"], bases)
    return s


# ---- one pass ------------------------------------------------------------------------------------

def _encode(s):
    kind, plans = s["case"]["kind"], s["plans"]
    if kind == "tensor":
        hist = zc.histogram(plans[0], s["ins"][0], s["hists"][0])
        book = zc.build_codebook(plans[0], hist.cpu().numpy(), s["policy"])
        sizes = [zc.compress(plans[0], book, s["ins"][0], s["outs"][0], s["ws"])]
    elif kind == "pages":
        s["enc"].set_codebooks(s["books"])
        sizes = zc.compress_batch(s["enc"], s["ws"])
        for d, p, n in zip(s["dicts"], plans, sizes):
            d.observe(p.input_bytes, n)
        return dict(containers=s["out_arena"], sizes=np.array(sizes, dtype=np.int64))
    else:
        zc.histogram_batch(s["hist_batch"], s["hists"])
        s["enc"].set_codebooks(zc.build_codebooks(plans, s["hists"].cpu().numpy(), s["policy"]))
        sizes = zc.compress_batch(s["enc"], s["ws"])
    return dict(containers=s["out_arena"], hists=s["hists"], sizes=np.array(sizes, dtype=np.int64))


def _decode(s):
    if s["case"]["kind"] == "tensor":
        zc.decompress(s["plans"][0], s["outs"][0], int(s["sizes"][0]), s["backs"][0], s["ws"])
    else:
        zc.decompress_batch(s["dec"], s["ws"])
    return dict(tensors=s["back_arena"])


def run(state):
    case = state["case"]
    if case["kind"] == "read":
        zc.decompress_chunks(state["plans"][0], state["outs"][0], state["comp_bytes"], case["first"], case["count"], state["back"], state["ws"])
        return state["back"]
    out = {}
    if case["pass"] != "decode":
        out.update(_encode(state))
    if case["pass"] != "encode":
        out.update(_decode(state))
    return out


# ---- what a pass cannot do without -----------------------------------------------------------------

def work(case):
    fmt, kind = case["fmt"], case["kind"]
    if kind == "read":
        u = 1024 * case["chunk_kib"] * case["count"]
        return dict(bytes=u * (1 + KV_RATIO[fmt]), flops=0)
    if kind == "tensor":
        elems = case["rows"] * case["cols"] / (32 if fmt == "scale" else 1)
        ratio = RATIO[fmt]
    elif kind == "pages":
        elems, ratio = 2 * case["layers"] * case["tokens"] * KV_HEADS * HEAD_DIM, KV_RATIO[fmt]
    else:
        elems = sum(s.n_elems for s in _specs(case, 0)) / (32 if fmt == "scale" else 1)
        ratio = RATIO[fmt]
    if kind == "delta":
        ratio = 0.06 * case["frozen"] + 0.43 * (1 - case["frozen"])
    u = elems * BYTES_PER_ELEM[fmt]
    one_way = u * (1 + ratio) + (u if kind == "delta" else 0)
    return dict(bytes=one_way * (2 if case["pass"] == "both" else 1), flops=0)


def tolerance(case):
    # Counts, containers and decoded elements are whole numbers and bytes: every correct implementation gives the same.
    return "exact"
