"""Workloads that a program using this library gives it, each through the public entry points: the
preallocated call sequences of ``pipeline`` and the C-ABI binding.

``listed()`` names the representative ones, ``draw(rng)`` gives another of the same ranges,
``prepare``/``run`` set one up and make one pass of it.  The shapes are those of ``inputs.WORKLOADS``
(7B-, 8B- and 26B-class grouped-query decoders and a small one, all with 128 channels a head).

Four kinds of call read scores or ranks to decide WHICH rows move, so that two equally accurate
programs could move different rows where two scores nearly tie.  The inputs keep such decisions away
from ties (the kept tokens' keys stand clear of the rest, a dropped token resembles one kept token) or
hand the deciding numbers in as exact inputs.
"""
from __future__ import annotations

import math
import statistics

import torch

from paper_2509_00419_b200 import binding as L
from paper_2509_00419_b200 import pipeline as P

D = 128
SPREAD = 3.0                # accumulated scores are log-normal: 4 % of the entries hold 90 % of the mass
# (hidden channels, query heads, KV heads): the small shape, the 7B, 8B and 26B classes
SHAPES = {"small": (1024, 8, 8), "7b": (3584, 28, 4), "8b": (4096, 32, 8), "26b": (6144, 48, 8)}
MODES = {"linear": L.W_LINEAR_RANK, "geometric": L.W_GEOMETRIC, "uniform": L.W_UNIFORM}


def _reduce(name, shape, B, n, T, ratio, stages, i0=0, mode="linear"):
    return dict(name=name, kind="reduce", shape=shape, B=B, i0=i0, n=n, T=T, ratio=ratio, stages=stages, mode=mode)


def listed():
    return [
        # Pyramid token merging while a prompt is encoded: score, select, merge and compact at every stage.
        # One image of 576 tokens on the small shape, one stage to half: nothing but latency.
        _reduce("reduce_image", "small", 1, 576, 64, 0.5, 1),
        # The 7B-class pyramid: one high-resolution prompt, three stages down to 3 %.
        _reduce("reduce_pyramid", "7b", 1, 2880, 128, 0.03, 3),
        # Sixteen requests encoded together on the 8B class, two stages to 35 %.
        _reduce("reduce_batch", "8b", 16, 1792, 96, 0.35, 2),
        # A video: one long sequence with a system prompt ahead of it, odd lengths, three stages to 15 %.
        _reduce("reduce_video", "7b", 1, 32767, 131, 0.15, 3, i0=35),
        # The attention of one prefill layer that hands over the token scores: the 7B-class prompt,
        # scored by the rows of the instruction text.
        dict(name="prefill_prompt", kind="prefill", shape="7b", B=1, i0=0, n=2880, T=128, window="text"),
        # The same for a 26B-class prompt of 16640 tokens, scored by all rows (the column sums of the whole
        # attention matrix): the largest call.
        dict(name="prefill_long", kind="prefill", shape="26b", B=1, i0=0, n=16384, T=256, window="all"),
        # One generated token on the 7B class after reduction and cache compression: 28 layers of short,
        # ragged caches, replayed from a CUDA graph as a serving loop does.
        dict(name="decode_token", kind="decode", shape="7b", layers=28, B=1, len=215, ragged=True, acc=False),
        # Eight sequences on the 8B class near the cache budget, probabilities accumulated for the next eviction.
        dict(name="decode_batch", kind="decode", shape="8b", layers=32, B=8, len=1100, ragged=False, acc=True),
        # The first layers of a video prompt, whose caches are not compressed: one sequence, four heads, 32898 rows.
        dict(name="decode_video", kind="decode", shape="7b", layers=6, B=1, len=32898, ragged=False, acc=False),
        # Cache compression once after prefill: cumulative threshold over the image span, 22 layers of one prompt.
        dict(name="compress_beta", kind="compress", shape="7b", layers=22, B=1, len=3008, T=128, beta=0.995, budget=0),
        # Eviction to a budget every 128 generated tokens: 32 layers of eight sequences.
        dict(name="compress_budget", kind="compress", shape="8b", layers=32, B=8, len=1152, T=128, beta=1.0, budget=1024),
        # Merging every dropped token into its most similar kept token: a 26B-class prompt, a quarter kept.
        dict(name="nearest_long", kind="nearest", shape="26b", B=1, n=16384, T=256, keep=4096),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["reduce", "reduce", "prefill", "decode", "decode", "compress", "nearest"])
    shape = rng.choice(["small", "7b", "8b", "26b"])
    C, H, Hkv = SHAPES[shape]
    T = _log_int(rng, 17, 256)
    if kind == "reduce":
        B = _log_int(rng, 1, 16)
        n = _log_int(rng, 150, 32767 // B)
        stages = rng.randint(1, 3)
        return dict(kind=kind, shape=shape, B=B, i0=rng.choice([0, 0, rng.randint(1, 64)]), n=n, T=T,
                    ratio=round(rng.uniform(0.03, 0.6), 3), stages=stages,
                    mode=rng.choice(["linear", "linear", "geometric", "uniform"]))
    if kind == "prefill":
        B = _log_int(rng, 1, 8)
        n = _log_int(rng, 150, int(16000 / math.sqrt(B)))
        return dict(kind=kind, shape=shape, B=B, i0=rng.choice([0, 0, rng.randint(1, 64)]), n=n, T=T,
                    window=rng.choice(["text", "text", "all", "none"]))
    if kind == "decode":
        layers, B = rng.randint(1, 32), _log_int(rng, 1, 16)
        # the caches of all layers together stay below the 1.2 GB of the 8B class at its budget
        most = max(80, min(32898, int(1.2e9 / (layers * B * Hkv * 2 * D * 2))))
        return dict(kind=kind, shape=shape, layers=layers, B=B, len=_log_int(rng, 65, most),
                    ragged=rng.random() < 0.5, acc=rng.random() < 0.5)
    if kind == "compress":
        layers, B = rng.randint(1, 32), _log_int(rng, 1, 8)
        most = max(400, min(16000, int(1.2e9 / (layers * B * Hkv * 2 * D * 2))))
        length = _log_int(rng, 300, most)
        by_budget = rng.random() < 0.5
        return dict(kind=kind, shape=shape, layers=layers, B=B, len=length, T=rng.randint(16, 128),
                    beta=1.0 if by_budget else rng.choice([0.9, 0.98, 0.99, 0.995, 0.999]),
                    budget=int(length * rng.uniform(0.5, 0.92)) if by_budget else 0)
    B = _log_int(rng, 1, 16)
    n = _log_int(rng, 300, 16384 // B)
    return dict(kind="nearest", shape=shape, B=B, n=n, T=T, keep=max(8, int(n * rng.uniform(0.2, 0.7))))


# --------------------------------------------------------------------------------------------------
def _schedule(case):
    """(image tokens before, image tokens after) of every stage."""
    out, n = [], case["n"]
    for M in P.pyramid_schedule(case["n"], case["ratio"], case["stages"]):
        out.append((n, max(2, M)))
        n = max(2, M)
    return out


class _Draws:
    """Seeded tensors on the GPU."""

    def __init__(self, seed):
        self.g = torch.Generator(device="cuda").manual_seed(seed)

    def normal(self, *shape):
        return torch.randn(*shape, generator=self.g, device="cuda", dtype=torch.bfloat16)

    def normal32(self, *shape):
        return torch.randn(*shape, generator=self.g, device="cuda")

    def order(self, B, n):
        """A random permutation of 0..n-1 for every sequence."""
        return torch.argsort(torch.rand(B, n, generator=self.g, device="cuda"), dim=1).to(torch.int32)


def _attention_inputs(d, B, rows, N, H, Hkv, i0, important):
    """Queries and keys in which the image tokens marked by ``important`` [B, n] hold most of the attention
    mass: their keys are pushed along a direction of their KV head that every query carries."""
    u = torch.nn.functional.normalize(d.normal32(B, Hkv, D), dim=-1)
    q = d.normal(B, rows, H, D) + (4.0 * u).repeat_interleave(H // Hkv, dim=1)[:, None].to(torch.bfloat16)
    k = d.normal(B, Hkv, N, D)
    n = important.shape[1]
    k[:, :, i0:i0 + n] += (16.0 * important[:, None, :, None] * u[:, :, None]).to(torch.bfloat16)
    return q, k


def _prepare_reduce(case, d):
    C, H, Hkv = SHAPES[case["shape"]]
    B, i0, T, dev = case["B"], case["i0"], case["T"], torch.device("cuda")
    stages = []
    for n, M in _schedule(case):
        N = i0 + n + T
        st = P.ReduceStage(B, N, C, H, Hkv, N, i0, n, M, dev, mode=MODES[case["mode"]])
        q, k = _attention_inputs(d, B, T, N, H, Hkv, i0, d.order(B, n) < st.k)
        # the keys that the layer projected are scored; the cache, which holds a copy, is compacted in place
        stages.append({"stage": st, "q": q, "k": k, "kc": k.clone(), "vc": d.normal(B, Hkv, N, D),
                       "pos": torch.arange(N, dtype=torch.int32, device=dev).repeat(B, 1)})
    return {"hidden": d.normal(B, i0 + case["n"] + T, C), "stages": stages}


def _prepare_prefill(case, d):
    _, H, Hkv = SHAPES[case["shape"]]
    B, i0, n = case["B"], case["i0"], case["n"]
    N = i0 + n + case["T"]
    q, k = _attention_inputs(d, B, N, N, H, Hkv, i0, d.order(B, n) < max(1, n // 50))
    dims = L.Dims(B=B, H=H, Hkv=Hkv, D=D, N=N, cap=N, i0=i0, n=n, causal=1, q_hi=N,
                  q_lo=0 if case["window"] == "all" else i0 + n)
    return {"q": q, "k": k, "v": d.normal(B, Hkv, N, D), "N": N, "i0": i0, "n": n,
            "window": None if case["window"] == "none" else (dims.q_lo, N),
            "out": torch.empty_like(q), "lse": torch.empty(B, H, N, device="cuda"),
            "score": torch.empty(B, n, device="cuda"), "head": torch.empty(B, Hkv, n, device="cuda"),
            "ws": L.alloc_workspace(L.OP_PREFILL_ATTN, dims, q.device)}


def _lengths(case, d, shape):
    if not case["ragged"]:
        return torch.full(shape, case["len"], dtype=torch.int32, device="cuda")
    u = torch.rand(*shape, generator=d.g, device="cuda")
    return (case["len"] * (0.5 + 0.5 * u)).to(torch.int32).clamp_(min=1)


def _prepare_decode(case, d):
    _, H, Hkv = SHAPES[case["shape"]]
    nl, B = case["layers"], case["B"]
    cap = (case["len"] + 64) // 64 * 64                    # room for the appended row
    dec = P.DecodeLayers(nl, B, H, Hkv, cap, torch.device("cuda"), with_acc=case["acc"])
    dec.K.normal_(generator=d.g)
    dec.V.normal_(generator=d.g)
    length = _lengths(case, d, dec.len.shape)
    q, k_new, v_new = d.normal(nl, B, H, D) * 2, d.normal(nl, B, Hkv, D), d.normal(nl, B, Hkv, D)
    dec.len.copy_(length)
    graph = P.capture(lambda: dec.decode_step(q, k_new, v_new))
    if case["acc"]:
        dec.acc.zero_()
    return {"dec": dec, "length": length, "graph": graph, "inputs": (q, k_new, v_new)}


def _prepare_compress(case, d):
    _, H, Hkv = SHAPES[case["shape"]]
    nl, B, n = case["layers"], case["B"], case["len"]
    dec = P.DecodeLayers(nl, B, H, Hkv, (n + 63) // 64 * 64, torch.device("cuda"))
    dec.K.normal_(generator=d.g)
    dec.V.normal_(generator=d.g)
    # accumulated probabilities: T rows of every query head of the group
    acc = torch.exp(SPREAD * d.normal32(nl, B, Hkv, dec.cap))
    acc[..., n:] = 0
    acc *= case["T"] * (H // Hkv) / acc.sum(dim=-1, keepdim=True)
    span = None
    if not case["budget"]:
        span = [torch.full((nl * B,), v, dtype=torch.int32, device="cuda") for v in (0, n - case["T"])]
    return {"dec": dec, "acc": acc, "length": torch.full_like(dec.len, n), "span": span,
            "beta": case["beta"], "budget": case["budget"], "recent": case["T"] if case["budget"] else 0}


def _prepare_nearest(case, d):
    C, H, Hkv = SHAPES[case["shape"]]
    B, n, k = case["B"], case["n"], case["keep"]
    N = n + case["T"]
    st = P.ReduceStage(B, N, C, H, Hkv, N, 0, n, k, torch.device("cuda"), mode=L.W_NEAREST_KEPT)
    st.rank.copy_(d.order(B, n))
    hidden = d.normal(B, N, C)
    # a dropped token looks like one of the kept ones
    by_rank = torch.argsort(st.rank, dim=1)
    like = torch.randint(0, k, (B, n - k), generator=d.g, device="cuda")
    for b in range(B):
        dropped, target = by_rank[b, k:], by_rank[b, :k][like[b]]
        hidden[b, dropped] = hidden[b, target] + 0.3 * hidden[b, dropped]
    return {"stage": st, "hidden": hidden, "kc": d.normal(B, Hkv, N, D), "vc": d.normal(B, Hkv, N, D),
            "pos": torch.arange(N, dtype=torch.int32, device="cuda").repeat(B, 1)}


_PREPARE = {"reduce": _prepare_reduce, "prefill": _prepare_prefill, "decode": _prepare_decode,
            "compress": _prepare_compress, "nearest": _prepare_nearest}


def prepare(case, seed):
    state = _PREPARE[case["kind"]](case, _Draws(seed))
    state["kind"] = case["kind"]
    return state


# --------------------------------------------------------------------------------------------------
def _run_reduce(s):
    hidden, out = s["hidden"], []
    for t in s["stages"]:
        st = t["stage"]
        st.run_score(t["q"], t["k"])
        st.run_select()
        st.run_merge(hidden, t["kc"], t["vc"], t["pos"])
        hidden = st.hidden_out
        out.append((st.score, hidden, t["kc"], t["vc"], t["pos"], st.new_len))
    return out


def _run_prefill(s):
    if s["window"] is None:
        return L.prefill_attn(s["q"], s["k"], s["v"], N=s["N"], out=s["out"], lse=s["lse"])[:2]
    return L.prefill_attn(s["q"], s["k"], s["v"], N=s["N"], window=s["window"], i0=s["i0"], n=s["n"], out=s["out"],
                          lse=s["lse"], score_out=s["score"], head_out=s["head"], ws=s["ws"])


def _run_decode(s):
    dec = s["dec"]
    dec.len.copy_(s["length"])                             # every pass generates the same token again
    s["graph"].replay()
    return dec.out, dec.len, dec.K, dec.V, dec.acc


def _run_compress(s):
    dec = s["dec"]
    # the caches have been filled again since the last compression
    dec.acc.copy_(s["acc"])
    dec.len.copy_(s["length"])
    e_lo, e_hi = s["span"] or (None, None)
    dec.compress(beta=s["beta"], budget=s["budget"], recent=s["recent"], e_lo=e_lo, e_hi=e_hi)
    return dec.K, dec.V, dec.acc, dec.len


def _run_nearest(s):
    st = s["stage"]
    st.run_merge(s["hidden"], s["kc"], s["vc"], s["pos"])
    return st.hidden_out, s["kc"], s["vc"], s["pos"], st.new_len


_RUN = {"reduce": _run_reduce, "prefill": _run_prefill, "decode": _run_decode, "compress": _run_compress,
        "nearest": _run_nearest}


def run(state):
    return _RUN[state["kind"]](state)


# --------------------------------------------------------------------------------------------------
def work(case):
    C, H, Hkv = SHAPES[case["shape"]]
    B, kind = case["B"], case["kind"]
    bytes_, flops = 0.0, 0.0
    if kind == "reduce":
        for n, M in _schedule(case):
            N, Nout = case["i0"] + n + case["T"], case["i0"] + M + case["T"]
            bytes_ += B * (case["T"] * H * D * 2 + N * Hkv * D * 2 + n * 4)     # queries, scored keys, scores
            bytes_ += B * (N + Nout) * (C * 2 + Hkv * D * 2 * 2 + 4)            # hidden, K and V, position ids
            flops += B * 2.0 * case["T"] * N * D * H                            # Q K^T once
    elif kind == "prefill":
        N = case["i0"] + case["n"] + case["T"]
        bytes_ = B * (N * H * D * 2 * 2 + N * Hkv * D * 2 * 2 + H * N * 4 + case["n"] * 4 * (1 + Hkv))
        flops = B * 4.0 * H * D * (N * (N + 1) / 2)
        if case["window"] != "none":                       # the column sums need the finished normalisers
            rows = N * (N + 1) / 2 if case["window"] == "all" else case["T"] * N
            flops += B * 2.0 * H * D * rows
    elif kind == "decode":
        mean = case["len"] * (0.75 if case["ragged"] else 1.0) + 1
        heads = case["layers"] * B * Hkv
        bytes_ = heads * mean * (2 * D * 2 + (8 if case["acc"] else 0)) + case["layers"] * B * (2 * H + 2 * Hkv) * D * 2
        flops = 4.0 * heads * mean * D * (H // Hkv)
    elif kind == "compress":
        heads, n = case["layers"] * B * Hkv, case["len"]
        kept = case["budget"]
        if not kept:                                       # the share of log-normal scores that carries beta of their sum
            normal = statistics.NormalDist()
            kept = case["T"] + (n - case["T"]) * normal.cdf(normal.inv_cdf(case["beta"]) - SPREAD)
        bytes_ = heads * ((n + kept) * (2 * D * 2) + (2 * n + n + kept) * 4)
    else:
        n, k, N = case["n"], case["keep"], case["n"] + case["T"]
        bytes_ = B * ((N + N - n + k) * (C * 2 + Hkv * D * 2 * 2 + 4) + n * 4)
        flops = B * 2.0 * (n - k) * k * C
    return {"bytes": bytes_, "flops": flops}


def tolerance(case):
    """Four times what the path differs by from itself in 64 bits."""
    kind = case["kind"]
    if kind == "compress":
        return "exact"                                     # rows are moved, nothing is computed
    if kind == "reduce":
        # scores 1.5e-7; kept rows are copies, the one merged row may round to the neighbouring bf16 value; the
        # merged token's position id is that of its heaviest contributor, where two may tie
        return {"rel": 3e-5, "max": 1e-2, "differ": 2e-3}
    return {"rel": 6e-3, "max": 2e-2}                      # bf16 rows: 1.7e-3, largest 3.9e-3
