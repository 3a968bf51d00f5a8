"""The work that users of this package have it do, as measurable cases.

Every case runs one pass of the L2A conditional attention layer through the public entry points of
``paper_2603_17484_b200.l2a`` on synthetic bf16 tensors (i.i.d. N(0, 1), the distribution of ``synth``), with the head
counts, head sizes, window and routing of ``synth.CONFIGS`` and of the tests.  Kinds of pass:

  forward  routing + compaction + forward: prefill of a model whose router decisions are known
  train    the same with the tensors saved for it, then the backward: one layer of a training step
  packed   a training step on documents of mixed length laid end to end on one token axis
  layer    the layer as the paper trains it, under activation checkpointing: Local Attention, router on its output,
           Global Attention on projections of its own, and the backward of all three in the order the chain rule gives;
           the routing decisions are those stored in the first forward, so that recomputing cannot flip a near tie
  chunk    prefill of the next chunk of a prompt against the keys cached so far (Lk > Lq)
  decode   one new token per sequence against the key/value cache
"""
from __future__ import annotations

import math
import random

import torch

from paper_2603_17484_b200 import l2a, synth

KINDS = ("forward", "train", "packed", "layer", "chunk", "decode")


def _case(name, kind, B, Lq, Lk, Hq, Hkv, D, W, routing, density, n_seq=0, shared=False):
    c = {"kind": kind, "B": B, "Lq": Lq, "Lk": Lk, "Hq": Hq, "Hkv": Hkv, "D": D, "W": W, "routing": routing,
         "density": density, "n_seq": n_seq, "shared": shared}
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # smallest call: one head over a thousand tokens; what counts is launches and latency
        _case("forward_1k_one_head", "forward", 1, 1024, 1024, 1, 1, 64, 128, "bernoulli", 0.2),
        # a short prompt of ragged length, where the passes around the attention kernels are a large share
        _case("forward_4k", "forward", 1, 4001, 4001, 28, 4, 128, 4096, "bernoulli", 0.2),
        # ordinary long-context prefill
        _case("forward_32k", "forward", 1, 32768, 32768, 28, 4, 128, 4096, "bernoulli", 0.2),
        # the longest prefill, a tenth of the tokens routed
        _case("forward_128k", "forward", 1, 131072, 131072, 32, 8, 128, 4096, "bernoulli", 0.1),
        # prefill in chunks: 2000 new tokens against a cache of 32K, with the shared-window option a model with one
        # set of projections uses
        _case("chunk_2k_of_34k", "chunk", 1, 2000, 34768, 32, 8, 128, 4096, "bernoulli", 0.2, shared=True),
        # training on short sequences, a small batch
        _case("train_4k", "train", 2, 4096, 4096, 28, 4, 128, 4096, "bernoulli", 0.2),
        # the training configuration: decisions from router logits
        _case("train_64k", "train", 1, 65536, 65536, 28, 4, 128, 4096, "logits", 0.0808),
        # the headline: a 128K training step with clustered routing
        _case("train_128k_clustered", "train", 1, 131072, 131072, 32, 8, 128, 4096, "clustered", 0.2),
        # training on documents of mixed length, packed
        _case("packed_64k_24_documents", "packed", 1, 65536, 65536, 32, 8, 128, 4096, "clustered", 0.2, n_seq=24),
        # the paper's layer, router and both modules trained, ragged length
        _case("layer_8k", "layer", 1, 8155, 8155, 28, 4, 128, 4096, "bernoulli", 0.2),
        # decode of a large batch over full caches, a quarter of the tokens routed
        _case("decode_16_of_128k", "decode", 16, 1, 131072, 32, 8, 128, 4096, "bernoulli", 0.25),
        # decode for a single user
        _case("decode_1_of_9k", "decode", 1, 1, 9001, 28, 4, 128, 4096, "all", 1.0),
    ]


def draw(rng):
    """One more case of the same ranges.  The largest drawn cases stay below the 128K training step."""
    def size(lo, hi):
        n = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
        return n if rng.random() < 0.6 else max(lo, n // 128 * 128)

    kind = rng.choice(KINDS)
    Hq, Hkv, D = rng.choice([(28, 4, 128), (32, 8, 128), (28, 4, 128), (32, 8, 128), (4, 4, 64), (12, 2, 64), (8, 1, 128)])
    W = rng.choice([128, 1000, 4096, 4096])
    routing = rng.choice(["bernoulli", "clustered", "logits"])
    density = rng.choice([0.05, 0.1, 0.2, 0.2, 0.3, 0.5])
    shared = rng.random() < 0.2
    if kind == "forward":
        n = size(256, 131072)
        return _case(None, kind, 1 if n > 16384 else rng.choice([1, 1, 2, 3]), n, n, Hq, Hkv, D, W, routing, density,
                     shared=shared)
    if kind == "train":
        n = size(256, 65536)
        return _case(None, kind, 1 if n > 8192 else rng.choice([1, 1, 2, 3]), n, n, Hq, Hkv, D, W, routing, density,
                     shared=shared)
    if kind == "packed":
        n = size(2048, 131072)
        return _case(None, kind, 1, n, n, Hq, Hkv, D, W, routing, density, n_seq=rng.randint(2, 2 + n // 1024))
    if kind == "layer":
        n = size(512, 32768)
        return _case(None, kind, 1 if n > 8192 else rng.choice([1, 2]), n, n, Hq, Hkv, D, W,
                     rng.choice(["bernoulli", "clustered"]), density)
    if kind == "chunk":
        n = size(64, 8192)
        return _case(None, kind, 1, n, n + size(2048, 122880), Hq, Hkv, D, W, routing, density, shared=shared)
    n = size(512, 131072)
    B = rng.randint(1, min(32, (1 << 21) // n))
    return _case(None, kind, B, 1, n, Hq, Hkv, D, W, rng.choice(["bernoulli", "all", "none"]), density)


# ----------------------------------------------------------------------------------------------------------------------
def _documents(case):
    """Lengths of the packed documents (a function of the case alone): log-normal, at least 16 tokens, summing to Lq."""
    r = random.Random(case["n_seq"] * 1000003 + case["Lq"])
    w = [math.exp(r.gauss(0.0, 0.8)) for _ in range(case["n_seq"])]
    spare = case["Lq"] - 16 * case["n_seq"]
    n = [16 + int(spare * x / sum(w)) for x in w]
    n[-1] += case["Lq"] - sum(n)
    return n


def _flags(case):
    f = l2a.FLAG_SHARED_WINDOW if case["shared"] else 0
    return f | (l2a.FLAG_SAVE_FOR_BWD if case["kind"] in ("train", "packed", "layer") else 0)


def _threshold_mean(density):
    """Mean of N(mean, 1) logits whose share above zero is `density`."""
    lo, hi = -8.0, 8.0
    for _ in range(60):
        mid = 0.5 * (lo + hi)
        lo, hi = (mid, hi) if 0.5 * math.erfc(-mid / math.sqrt(2.0)) < density else (lo, mid)
    return 0.5 * (lo + hi)


def prepare(case, seed):
    kind, B, Lq, Lk, Hq, Hkv, D = (case[k] for k in ("kind", "B", "Lq", "Lk", "Hq", "Hkv", "D"))
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))

    def normal(*shape, dtype=torch.bfloat16):
        return torch.randn(shape, generator=g, device="cuda", dtype=dtype)

    def mask(n_rows, n):
        if case["routing"] == "clustered":
            return torch.from_numpy(synth.mask_clustered(n_rows, n, case["density"], int(seed))).cuda()
        rho = {"all": 1.0, "none": 0.0}.get(case["routing"], case["density"])
        return (torch.rand((n_rows, n), generator=g, device="cuda") < rho).to(torch.uint8)

    s = {"kind": kind}
    if kind == "decode":
        p = l2a.params(B, 1, Lk, Hq, Hkv, D, case["W"])
        d = mask(B, 1)[:, 0].contiguous()
        if case["routing"] == "bernoulli":       # a batch of this kind has routed tokens in the stated share
            d.zero_()
            d[torch.randperm(B, generator=g, device="cuda")[:max(1, round(B * case["density"]))]] = 1
        s.update(p=p, q=normal(B, 1, Hq, D), K=normal(B, Lk, Hkv, D), V=normal(B, Lk, Hkv, D), d=d,
                 O=torch.empty((B, 1, Hq, D), dtype=torch.bfloat16, device="cuda"),
                 ws=torch.empty(l2a.l2a_decode_workspace_bytes(p), dtype=torch.uint8, device="cuda"))
        return s

    train = kind in ("train", "packed", "layer")
    logits = case["routing"] == "logits"
    bounds = None
    if kind == "packed":
        n = torch.tensor([0] + _documents(case), dtype=torch.int64)
        s["cu_seqlens"] = torch.cumsum(n, 0).to(torch.int32).cuda()
        bounds = s["seq_bounds"] = torch.empty((Lq, 2), dtype=torch.int32, device="cuda")
    p = l2a.params(B, Lq, Lk, Hq, Hkv, D, case["W"], flags=_flags(case), seq_bounds=bounds)
    b = l2a.Buffers.allocate(p, backward=train, router_dtype=torch.float32 if logits else torch.uint8)
    if case["shared"] and not train:             # the forward reads it back
        b.lse_loc = torch.empty((B, Hq, Lq), dtype=torch.float32, device="cuda")
    for name in ("Q", "K", "V") + (("dO",) if train else ()):
        getattr(b, name).normal_(generator=g)
    mean = _threshold_mean(case["density"])
    b.router.copy_(normal(B, Lq, dtype=torch.float32) + mean if logits else mask(B, Lq))
    s.update(p=p, b=b, router_kind=l2a.ROUTER_LOGITS_F32 if logits else l2a.ROUTER_MASK_U8)
    if kind == "layer":
        # Global Attention's own projections, the router's parameters, and the gradients of both.  The local output of
        # N(0, 1) values averages a window of them, so weights of this size give logits of about unit variance.
        keys = 0.5 * (min(case["W"], Lq) + 1)
        w = normal(Hq * D, dtype=torch.float32) * math.sqrt(keys / (2.7 * Hq * D))
        own = {n: torch.empty_like(getattr(b, n[0])).normal_(generator=g) for n in ("Qg", "Kg", "Vg")}
        grad = {n: torch.empty_like(getattr(b, n[1])) for n in ("dQg", "dKg", "dVg")}
        s.update(own, **grad)
        s.update(p_local=l2a.params(B, Lq, Lk, Hq, Hkv, D, case["W"], flags=l2a.FLAG_SAVE_FOR_BWD | l2a.FLAG_SKIP_GLOBAL),
                 p_global=l2a.params(B, Lq, Lk, Hq, Hkv, D, case["W"], flags=l2a.FLAG_SAVE_FOR_BWD | l2a.FLAG_GLOBAL_PHASE),
                 p_bwd_global=l2a.params(B, Lq, Lk, Hq, Hkv, D, case["W"], flags=l2a.FLAG_SAVE_FOR_BWD | l2a.FLAG_SKIP_LOCAL),
                 w=w, bias=mean, reg=1e-3, z=torch.empty((B, Lq), dtype=torch.float32, device="cuda"),
                 sum_sq=torch.empty(B, dtype=torch.float32, device="cuda"),
                 dz=torch.empty((B, Lq), dtype=torch.float32, device="cuda"), dw=torch.empty_like(w),
                 dbias=torch.empty(1, dtype=torch.float32, device="cuda"), dS=torch.empty_like(b.dO))
    return s


def run(s):
    kind = s["kind"]
    if kind == "decode":
        l2a.l2a_decode(s["p"], s["q"], s["K"], s["V"], s["d"], s["O"], s["ws"])
        return s["O"]
    b = s["b"]
    if kind == "layer":
        return _run_layer(s, b)
    if kind == "packed":
        l2a.l2a_pack_sequences(s["cu_seqlens"], b.p.Lq, s["seq_bounds"])
    b.route(s["router_kind"])
    b.forward()
    if kind in ("forward", "chunk"):
        return {"O": b.O, "q_idx": b.q_idx, "n_routed": b.n_routed}
    b.backward()
    return {"O": b.O, "dQ": b.dQ, "dK": b.dK, "dV": b.dV, "q_idx": b.q_idx, "n_routed": b.n_routed}


def _run_layer(s, b):
    pl, pg = s["p_local"], s["p_global"]
    l2a.l2a_forward(pl, b.Q, b.K, b.V, None, None, None, None, b.O, b.S_save, b.A_c, b.lse_loc, b.lse_glb, b.fwd_ws)
    l2a.l2a_router_logits(pl, b.S_save, s["w"], s["bias"], s["z"], s["sum_sq"])
    b.route(s["router_kind"])
    l2a.l2a_forward(pg, s["Qg"], s["Kg"], s["Vg"], b.d_mask, b.q_idx, b.n_routed, b.prefix, b.O, b.S_save, b.A_c, b.lse_loc,
                    b.lse_glb, b.fwd_ws)
    l2a.l2a_backward(s["p_bwd_global"], s["Qg"], s["Kg"], s["Vg"], b.d_mask, b.q_idx, b.n_routed, b.prefix, b.dO, None,
                     b.A_c, None, b.lse_glb, s["dQg"], s["dKg"], s["dVg"], b.dgate, b.bwd_ws)
    l2a.l2a_router_backward(pl, b.S_save, s["w"], s["z"], b.dgate, s["reg"], b.dO, s["dz"], s["dw"], s["dbias"], s["dS"])
    l2a.l2a_backward(pl, b.Q, b.K, b.V, None, None, None, None, s["dS"], b.S_save, None, b.lse_loc, None, b.dQ, b.dK, b.dV,
                     None, b.bwd_ws)
    return {"O": b.O, "dQ": b.dQ, "dK": b.dK, "dV": b.dV, "dQg": s["dQg"], "dKg": s["dKg"], "dVg": s["dVg"],
            "dz": s["dz"], "dw": s["dw"], "sum_sq": s["sum_sq"]}     # dbias is the sum of dz, which mostly cancels


# ----------------------------------------------------------------------------------------------------------------------
def _density(case):
    return {"all": 1.0, "none": 0.0}.get(case["routing"], case["density"])


def _pairs(case):
    """(query, key) pairs per query head of one batch entry: in the window, and causal ones of the routed share."""
    off = case["Lk"] - case["Lq"]
    docs = _documents(case) if case["kind"] == "packed" else [case["Lq"]]

    def upto(n, w):          # sum over positions t < n of min(t, w) + 1
        return n * (n + 1) / 2 if n <= w else w * (w + 1) / 2 + (w + 1) * (n - w)

    loc = sum(upto(off + n, case["W"]) - upto(off, case["W"]) for n in docs)
    glb = sum((off + n) * (off + n + 1) / 2 - off * (off + 1) / 2 for n in docs) * _density(case)
    if case["shared"]:       # a routed row's pairs inside its window are the local ones
        glb -= loc * _density(case)
    return loc, glb


def work(case):
    kind, B, Lq, Lk, Hq, Hkv, D, W = (case[k] for k in ("kind", "B", "Lq", "Lk", "Hq", "Hkv", "D", "W"))
    rho = _density(case)
    if kind == "decode":
        n_routed = B if rho == 1.0 else 0 if rho == 0.0 else max(1, round(B * rho))
        # a routed token reads the whole cache, its window with it; the others their window
        keys = n_routed * Lk + (B - n_routed) * min(W + 1, Lk)
        pairs = n_routed * Lk + B * min(W + 1, Lk)
        return {"bytes": 4.0 * D * Hkv * keys + 4.0 * B * Hq * D, "flops": 4.0 * D * Hq * pairs}
    loc, glb = _pairs(case)
    q, kv = 2.0 * B * Lq * Hq * D, 2.0 * B * Lk * Hkv * D
    fwd = 4.0 * D * Hq * B * (loc + glb)
    if kind in ("forward", "chunk"):
        return {"bytes": 2 * q + 2 * kv + B * Lq, "flops": fwd}
    if kind == "layer":      # two sets of Q, K, V and their gradients, dO in, O out
        return {"bytes": 6 * q + 8 * kv, "flops": 3.5 * fwd}
    return {"bytes": 4 * q + 4 * kv + B * Lq, "flops": 3.5 * fwd}


def tolerance(case):
    """Four times the distance from the layer evaluated in 64 bits (1024 to 2048 tokens, head size 64 and 128):

        forward outputs           2.1e-3 in the 2-norm, 0.03 at most relative to the larger of value and mean square root
        gradients of Q, K, V      3.0e-3 (3.4e-3 behind the router), 0.08 (the first rows, which see a handful of keys)
        router weight gradient    3.4e-3 to 9.4e-3 (a sum over tokens of products of bf16 results that mostly cancel)

    The probabilities, dS and all results are bf16, sums are fp32.  Indices and counts are exact."""
    if case["kind"] == "layer":
        return {"rel": 0.03, "max": 0.35}
    if case["kind"] in ("train", "packed"):
        return {"rel": 1.2e-2, "max": 0.33}
    return {"rel": 8.5e-3, "max": 0.12}
