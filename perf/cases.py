"""The work that users of the router give it, as cases that can be timed and compared.

A case is a dict of plain values.  ``op`` says which public entry points it goes through:

  route   ``binding.route``: one router call of a serving or inference program (ids, gates, expert counts).
  train   the router's part of a training forward step: ``binding.route`` with the log-sum-exp, then
          ``more_route_psum`` for the load-balancing statistic.
  full    ``more_route_full``: the fused standard (full-rank) router.
  merge   ``more_merge_shards``: the step after the all-gather of an expert-sharded router.

Sizes are those of the library's own configurations (``inputs.CONFIGS``), its tests and its benchmark, or lie between
them.  T is any number of tokens; h, r and M are multiples of 8 (hidden sizes, ranks and expert counts in use are).
"""
import math

import torch

from paper_2609_36301_b200 import binding as mr

# Ranges that the cases stand for.
T_MAX, H_MIN, H_MAX, M_MIN, M_MAX, K_MAX = 65536, 128, 4096, 256, 131072, 16
RANKS = (8, 16, 24, 32, 40, 48, 56, 64)
X_MAX = 65536 * 2048            # largest T * h
LOGITS_MAX = 32768 * 65536      # largest T * M at r <= 32; half of that for larger ranks, a quarter for a training step
FULL_MAX = 16384 * 2048 * 16384  # largest T * h * M of the standard router


def _route(name, T, h, r, M, k, gate, mixture=False):
    return dict(name=name, op="route", T=T, h=h, r=r, M=M, k=k, gate=gate, mixture=mixture)


def listed():
    return [
        # decode, one sequence: a single token against all experts, latency is everything
        _route("decode_1", 1, 2048, 64, 16384, 8, 0),
        # decode, a batch of 64 sequences on the widest router
        _route("decode_64_wide", 64, 4096, 64, 131072, 16, 0),
        # a tiny layer (unit tests, toy models): launch and host cost
        _route("tiny", 256, 128, 8, 256, 2, 0),
        # chunked prefill with nothing round about it: odd token count, hidden size and experts off the tile sizes
        _route("ragged", 3001, 1000, 24, 5000, 6, 1),
        # prefill of a small model, full-softmax gates
        _route("prefill_small", 16384, 512, 16, 4096, 8, 1),
        # prefill with few experts: close to bound by reading X
        _route("prefill_few_experts", 32768, 512, 32, 1024, 8, 0),
        # prefill with very many experts: bound by the sweep over the experts
        _route("prefill_many_experts", 32768, 512, 32, 65536, 8, 0),
        # prefill of a mid-sized model, tokens that cluster (skewed expert load); the benchmark's workload
        _route("prefill_mid", 65536, 2048, 64, 16384, 8, 0, mixture=True),
        # prefill of a large fine-grained model: 131072 experts, full-softmax gates over all of them
        _route("prefill_large", 8192, 4096, 64, 131072, 16, 1),
        # training forward of a 12-layer model's router: route with log-sum-exp, then the column sums for the loss
        dict(name="train_step", op="train", T=65536, h=512, r=64, M=8192, k=4, gate=0, mixture=False),
        # the standard router that the low-rank one replaces, for models that still have it in some layers
        dict(name="standard_router", op="full", T=16384, h=2048, M=16384, k=8, gate=0, mixture=False),
        # eight expert shards' reports merged into the global top-k
        dict(name="merge_8_shards", op="merge", S=8, T=8192, M=131072, k=16, gate=1),
    ]


def _log_int(rng, lo, hi, step=1):
    """An integer spread over the logarithm of [lo, hi], a multiple of ``step``."""
    v = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    return max(lo, min(hi, int(round(v / step)) * step))


def draw(rng):
    op = rng.choices(("route", "train", "full", "merge"), (14, 2, 2, 2))[0]
    M = _log_int(rng, M_MIN, M_MAX, 8)
    k = _log_int(rng, 1, K_MAX)
    gate = rng.randrange(2)
    if op == "merge":
        return dict(op=op, S=rng.choice((2, 4, 8)), T=_log_int(rng, 1, 16384), M=M // 64 * 64, k=k, gate=gate)
    h = _log_int(rng, H_MIN, H_MAX, 8)
    r = rng.choice(RANKS)
    logits_max = LOGITS_MAX // (4 if op == "train" else 1 if r <= 32 else 2)
    T = _log_int(rng, 1, min(T_MAX, X_MAX // h, logits_max // M))
    mixture = rng.random() < 0.25
    if op == "full":
        return dict(op=op, T=max(1, min(T, FULL_MAX // (h * M))), h=h, M=M, k=k, gate=gate, mixture=mixture)
    return dict(op=op, T=T, h=h, r=r, M=M, k=k, gate=gate, mixture=mixture)


def _tokens(c, gen):
    """Token activations: unit Gaussian, or a 64-component mixture whose tokens share favourite experts."""
    x = torch.randn((c["T"], c["h"]), generator=gen, device="cuda", dtype=torch.bfloat16)
    if c["mixture"]:
        means = torch.randn((64, c["h"]), generator=gen, device="cuda", dtype=torch.bfloat16)
        comp = torch.randint(0, 64, (c["T"],), generator=gen, device="cuda")
        x.mul_(0.5).add_(means[comp])
    return x


def prepare(case, seed):
    c = dict(case)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed))

    def randn(shape, sd, dtype=torch.bfloat16):
        return (torch.randn(shape, generator=gen, device="cuda", dtype=torch.float32) * sd).to(dtype)

    if c["op"] == "merge":
        # what the shards report: k local ids per token, distinct, with their logits in descending order, and the
        # log-sum-exp over the shard's experts
        S, T, k, per = c["S"], c["T"], c["k"], c["M"] // c["S"]
        first = torch.randint(0, per, (S, T, 1), generator=gen, device="cuda")
        step = torch.randint(1, max(2, per // k), (S, T, 1), generator=gen, device="cuda")
        c["idx"] = ((first + step * torch.arange(k, device="cuda")) % per).to(torch.int32)
        c["val"] = (randn((S, T, k), 0.25, torch.float32) + 3.0).sort(dim=-1, descending=True).values.contiguous()
        c["lse"] = randn((S, T), 0.1, torch.float32) + (math.log(per) + 0.5)
        c["base"] = [s * per for s in range(S)]
        return c
    c["X"] = _tokens(c, gen)
    # weights that keep the logits of a unit-variance token at unit variance
    if c["op"] == "full":
        c["W"] = randn((c["h"], c["M"]), c["h"] ** -0.5)
    else:
        c["R1"] = randn((c["h"], c["r"]), c["h"] ** -0.5)
        c["R2"] = randn((c["r"], c["M"]), c["r"] ** -0.5)
    return c


def run(s):
    k, gate = s["k"], s["gate"]
    if s["op"] == "route":
        res = mr.route(s["X"], s["R1"], s["R2"], k, gate)
        return dict(idx=res.idx, gate=res.gate, counts=res.counts)
    if s["op"] == "train":
        res = mr.route(s["X"], s["R1"], s["R2"], k, gate, want_lse=True)
        psum = torch.empty((s["M"],), dtype=torch.float32, device="cuda")
        mr.more_route_psum(s["X"], s["R1"], s["R2"], res.lse, psum)
        return dict(idx=res.idx, gate=res.gate, counts=res.counts, lse=res.lse, psum=psum)
    idx = torch.empty((s["T"], k), dtype=torch.int32, device="cuda")
    out_gate = torch.empty((s["T"], k), dtype=torch.float32, device="cuda")
    counts = torch.empty((s["M"],), dtype=torch.int32, device="cuda")
    if s["op"] == "full":
        mr.more_route_full(s["X"], s["W"], k, gate, idx, out_gate, counts)
        return dict(idx=idx, gate=out_gate, counts=counts)
    lse = torch.empty((s["T"],), dtype=torch.float32, device="cuda")
    mr.more_merge_shards(s["idx"], s["val"], s["lse"], s["base"], s["M"], gate, idx, out_gate, counts, None, lse)
    return dict(idx=idx, gate=out_gate, counts=counts, lse=lse)


def work(case):
    T, M, k = case["T"], case["M"], case["k"]
    out = 8 * T * k + 4 * M
    if case["op"] == "merge":
        return dict(bytes=case["S"] * T * (8 * k + 4) + out + 4 * T, flops=0)
    h = case["h"]
    if case["op"] == "full":
        return dict(bytes=2 * T * h + 2 * h * M + out, flops=2 * T * h * M)
    r = case["r"]
    inputs = 2 * T * h + 2 * h * r + 2 * r * M
    flops = 2 * T * (h * r + r * M)
    if case["op"] == "train":
        # the column sums need every token's log-sum-exp, so the logits are produced twice
        return dict(bytes=2 * inputs + out + 8 * T + 4 * M, flops=2 * flops)
    return dict(bytes=inputs + out, flops=flops)


def tolerance(case):
    if case["op"] == "merge":
        # ids and logits are compared as they are, only the exponentials of the gates round
        return dict(rel=1e-5, max=1e-4, differ=0.0)
    # Logits agree to about 1e-5 (fp32 sums of bf16 products; the low-rank router carries z to 16 mantissa bits), gates
    # and log-sum-exp inherit that.  Ids at neighbouring places may swap, and the k-th id be another one, where two
    # logits are closer than that; each such token moves two of the M counts.
    return dict(rel=5e-5, max=1e-3, differ=0.01)
