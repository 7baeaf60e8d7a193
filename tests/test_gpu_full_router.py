"""The fused standard (full-rank) router on the GPU, ``more_route_full``, against the oracle.

The oracle has no separate standard router: with ``R1 = I_h`` (exact in bf16) its low-rank route IS the standard router
``softmax(TopK(X W))`` (the identity pin of the CPU tests), so the GPU result is checked against
``oracle.route(X, I, W)`` with the same acceptance rule as the low-rank path."""
import numpy as np
import pytest

from paper_2609_36301_b200 import binding as mr
from paper_2609_36301_b200 import inputs

from helpers import check_counts, check_rows, to_device

pytestmark = pytest.mark.gpu


def _run(case, msplit=0, gate_mode=None):
    import torch
    gm = case.gate_mode if gate_mode is None else gate_mode
    X, _, W = to_device(case)
    T, M, k = case.T, case.M, case.k
    idx = torch.full((T, k), -3, dtype=torch.int32, device="cuda")
    gate = torch.full((T, k), -1.0, dtype=torch.float32, device="cuda")
    counts = torch.full((M,), 77, dtype=torch.int32, device="cuda")
    topval = torch.empty((T, k), dtype=torch.float32, device="cuda")
    lse = torch.empty((T,), dtype=torch.float32, device="cuda")
    mr.more_route_full(X, W, k, gm, idx, gate, counts, topval, lse, msplit)
    torch.cuda.synchronize()
    assert mr.more_route_status() == 0
    stats = check_rows(case, None, idx.cpu().numpy(), gate.cpu().numpy(), topval.cpu().numpy(), lse.cpu().numpy(),
                       gate_mode=gm)
    check_counts(idx.cpu().numpy(), counts.cpu().numpy(), M, stats["ref"].counts, bool(stats["differs_mask"].any()))
    return stats


@pytest.mark.parametrize("gate_mode", [0, 1])
@pytest.mark.parametrize("T,h,M,k", [
    (256, 128, 256, 2),        # one CTA, one full 256-expert step, two k-tiles
    (300, 136, 200, 4),        # ragged everywhere: h not a multiple of 64, M not of 64, T not of 32
    (1000, 512, 1024, 8),      # several CTAs, eight k-tiles through three stages
    (2500, 64, 4096, 8),       # one k-tile per step
    (129, 256, 72, 16),        # list capacity 16, a token group with one live row
    (64, 384, 64, 32),         # list capacity 32, a single step
    (600, 192, 1000, 8),       # four 256-expert steps, the last one ragged (232 experts)
    (260, 128, 520, 4),        # three steps, eight live columns in the last; a second token group with four rows
])
def test_full_router_matches_oracle(T, h, M, k, gate_mode):
    case = inputs.full_rank_case(T, h, M, k, gate_mode, seed=5)
    stats = _run(case)
    assert stats["topval_err"] < 5e-5


@pytest.mark.parametrize("msplit", [2, 3, 7])
def test_full_router_with_expert_split(msplit):
    case = inputs.full_rank_case(700, 256, 2048, 8, 1, seed=9)
    _run(case, msplit=msplit)


@pytest.mark.parametrize("gate_mode", [0, 1])
@pytest.mark.parametrize("T,h,M,k", [
    (1, 72, 37896, 1),            # one token, CTAs of one or two tiles of 256 experts, the last of eight experts
    (1, 72, 37640, 1),            # 148 CTAs of one tile, the last of eight experts
    (1, 512, 40000, 32),          # the longest lists
    (10, 1448, 5000, 3),          # 20 CTAs
    (130, 64, 9000, 17),          # two runs of 128 tokens in one block
    (300, 136, 20008, 16),        # two blocks, ragged
    (600, 64, 520, 8),            # two or three tiles: the fewest lists
])
def test_full_router_with_few_tokens(T, h, M, k, gate_mode):
    """Many CTAs per token block, whose lists the finishing kernels join."""
    _run(inputs.full_rank_case(T, h, M, k, gate_mode, seed=T + M))


@pytest.mark.parametrize("gate_mode", [0, 1])
@pytest.mark.parametrize("T,M,k", [
    (40, 37640, 32),              # 148 CTAs of one tile: more equals than the finishing kernel holds
    (300, 20008, 16),
    (600, 1032, 8),               # a warp per token
])
def test_full_router_with_extreme_logits_and_an_expert_split(T, M, k, gate_mode):
    """Tokens with equal logits, with infinite ones (every second expert), and of NaN: the first two are sorted as any others,
    and none of them changes the other tokens."""
    import torch
    gen = torch.Generator(device="cuda").manual_seed(T + M + k)
    X = torch.randn((T, 72), generator=gen, device="cuda").to(torch.bfloat16)
    W = (torch.randn((72, M), generator=gen, device="cuda") / 8).to(torch.bfloat16)
    W[0, ::2], W[0, 1::2] = 4, 1
    zero, half, nan = (torch.arange(i, T, 17, device="cuda") for i in (3, 4, 5))
    X[zero], X[half], X[nan] = 0, 0, 0

    def run():
        idx = torch.full((T, k), -3, dtype=torch.int32, device="cuda")
        gate, topval, lse = (torch.empty(s, device="cuda") for s in ((T, k), (T, k), (T,)))
        counts = torch.full((M,), 77, dtype=torch.int32, device="cuda")
        mr.more_route_full(X, W, k, gate_mode, idx, gate, counts, topval, lse)
        torch.cuda.synchronize()
        assert mr.more_route_status() == 0 and mr.debug_scratch_guard() == 1
        valid = idx[(idx >= 0) & (idx < M)]
        assert torch.equal(torch.bincount(valid.long(), minlength=M).int(), counts)
        return idx, gate, topval

    clean = run()
    first = torch.arange(k, device="cuda", dtype=torch.int32)
    assert bool((clean[0][zero] == first).all()) and bool((clean[0][nan] == first).all())
    X[half, 0], X[nan, 1] = 2e38, float("nan")
    idx, gate, topval = run()
    assert bool((idx[zero] == first).all()) and bool((idx[half] == 2 * first).all()) and bool(torch.isinf(topval[half]).all())
    others = torch.ones(T, dtype=torch.bool, device="cuda")
    others[half], others[nan] = False, False
    for a, b in zip(clean, (idx, gate, topval)):
        assert torch.equal(a[others], b[others])


@pytest.mark.parametrize("values", ["plain", "equal", "infinite", "gave up"])
@pytest.mark.parametrize("T,k,parts", [
    (3, 16, 100),             # more than 64 lists: a CTA of 512 threads per token
    (2, 32, 256),             # the most and the longest lists
    (200, 8, 16),             # 512 threads
    (600, 8, 20),             # 128 threads
    (700, 16, 8),             # a warp per token, up to 512 entries in registers
    (900, 8, 8),              # ... up to 256
    (300, 3, 4),              # a warp per token, the short code
])
def test_joining_lists(T, k, parts, values):
    """The split router's second half alone.  Lists of 0 to k entries, some tokens without any; logits that are all equal or
    infinite; and parts whose CTA gave up waiting, which must count as empty whatever the scratch held before."""
    import torch
    rng = np.random.default_rng(T + k)
    M = 3 * parts * k
    val = -np.sort(-rng.standard_normal((T, parts, k)).astype(np.float32), axis=-1)
    if values == "equal":
        val[:] = 1.5
    if values == "infinite":
        val = -np.sort(-np.where(rng.random(val.shape) < 0.3, np.float32(np.inf), val), axis=-1)
    length = rng.integers(0, k + 1, (T, parts))
    length[1::50] = 0                                                        # tokens without a candidate
    val[np.arange(k) >= length[..., None]] = -np.inf
    ids = np.argsort(rng.random((T, M)), axis=-1)[:, :parts * k].reshape(T, parts, k).astype(np.int32)
    mz = np.stack([rng.standard_normal((T, parts)) + 3, rng.random((T, parts)) + 1], axis=-1).astype(np.float32)
    swept = np.ones((T, parts), dtype=np.uint8)
    if values == "gave up":
        swept = (rng.random((T, parts)) < 0.6).astype(np.uint8)
        swept[0], swept[-1, 0] = 0, 1

    there = (swept != 0)[..., None] & (val > -np.inf)
    v = np.where(there, val, -np.inf).reshape(T, -1)
    i = np.where(there, ids, 2**31 - 1).reshape(T, -1)
    order = np.lexsort((i, -v), axis=-1)[:, :k]
    want_val, want_idx = np.take_along_axis(v, order, -1), np.take_along_axis(i, order, -1)
    some = swept.any(axis=1)
    m = np.where(swept != 0, mz[..., 0].astype(np.float64), -np.inf)
    top = np.where(some, m.max(axis=1), 0.0)
    with np.errstate(divide="ignore"):
        want_lse = (top + np.log2((mz[..., 1] * np.exp2(m - top[:, None])).sum(axis=1))) * np.log(2.0)

    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    lists = dev(val), dev(ids), dev(mz), dev(swept)
    for gate_mode in (0, 1):
        idx = torch.full((T, k), -3, dtype=torch.int32, device="cuda")
        gate, topval = torch.empty((T, k), device="cuda"), torch.empty((T, k), device="cuda")
        lse, counts = torch.empty((T,), device="cuda"), torch.full((M,), 77, dtype=torch.int32, device="cuda")
        mr.debug_join_lists(*lists, M, gate_mode, idx, gate, counts, topval, lse)
        torch.cuda.synchronize()
        assert mr.debug_scratch_guard() == 1
        assert np.array_equal(idx.cpu().numpy(), want_idx) and np.array_equal(topval.cpu().numpy(), want_val)
        assert np.array_equal(counts.cpu().numpy(), np.bincount(want_idx[want_idx < M], minlength=M))
        # a few hundred fp32 additions and exponentials good to 2^-22
        np.testing.assert_allclose(lse.cpu().numpy()[some], want_lse[some], atol=2e-5)
        sure = np.isfinite(want_val).all(axis=1)
        e = np.exp(want_val[sure].astype(np.float64) - (want_lse[sure, None] if gate_mode else want_val[sure, :1]))
        want_gate = e if gate_mode else e / e.sum(-1, keepdims=True)
        np.testing.assert_allclose(gate.cpu().numpy()[sure], want_gate, rtol=5e-5)


def test_full_router_agrees_with_low_rank_router_on_the_identity():
    """Same inputs through ``more_route_ex`` with R1 = I (r = h = 64, the largest the low-rank tensor path takes):
    the two GPU paths must pick the same experts."""
    import torch
    case = inputs.full_rank_case(512, 64, 1024, 8, 0, seed=3)
    X, R1, W = to_device(case)
    low = mr.route(X, R1, W, case.k, 0)
    idx = torch.empty((case.T, case.k), dtype=torch.int32, device="cuda")
    gate = torch.empty((case.T, case.k), dtype=torch.float32, device="cuda")
    counts = torch.empty((case.M,), dtype=torch.int32, device="cuda")
    mr.more_route_full(X, W, case.k, 0, idx, gate, counts)
    torch.cuda.synchronize()
    same = (torch.sort(idx, dim=1).values == torch.sort(low.idx, dim=1).values).all(dim=1)
    assert same.float().mean() > 0.999                       # near-ties may differ; the oracle test is the exact one
    assert int(counts.sum()) == case.T * case.k


def test_full_router_rejects_shapes_it_cannot_take():
    import torch
    X = torch.zeros((8, 12), dtype=torch.bfloat16, device="cuda")
    W = torch.zeros((12, 16), dtype=torch.bfloat16, device="cuda")
    idx = torch.empty((8, 2), dtype=torch.int32, device="cuda")
    gate = torch.empty((8, 2), dtype=torch.float32, device="cuda")
    counts = torch.empty((16,), dtype=torch.int32, device="cuda")
    with pytest.raises(mr.MoreRouteError):
        mr.more_route_full(X, W, 2, 0, idx, gate, counts)     # h = 12 is not a multiple of 8


def test_full_router_at_benchmark_size_sampled_rows():
    """A full-size launch (c2's shape with M = 4096: 147 token blocks of 224 tokens, split in two along the experts, two
    CTAs per SM), checked on sampled rows the oracle can compute one by one and on the whole-output properties."""
    import torch
    T, h, M, k = 32768, 512, 4096, 8
    case = inputs.full_rank_case(T, h, M, k, 0, seed=21)
    X, _, W = to_device(case)
    idx = torch.empty((T, k), dtype=torch.int32, device="cuda")
    gate = torch.empty((T, k), dtype=torch.float32, device="cuda")
    counts = torch.empty((M,), dtype=torch.int32, device="cuda")
    topval = torch.empty((T, k), dtype=torch.float32, device="cuda")
    lse = torch.empty((T,), dtype=torch.float32, device="cuda")
    mr.more_route_full(X, W, k, 0, idx, gate, counts, topval, lse)
    torch.cuda.synchronize()
    assert mr.more_route_status() == 0
    rows = np.unique(np.concatenate([np.arange(0, 64), np.arange(T - 64, T),
                                     np.random.default_rng(4).integers(0, T, 128)]))
    idx_np, gate_np = idx.cpu().numpy(), gate.cpu().numpy()
    check_rows(case, rows, idx_np[rows], gate_np[rows], topval.cpu().numpy()[rows], lse.cpu().numpy()[rows], gate_mode=0)
    check_counts(idx_np, counts.cpu().numpy(), M)
    srt = np.sort(idx_np, axis=1)
    assert idx_np.min() >= 0 and idx_np.max() < M and np.all(srt[:, 1:] != srt[:, :-1])
    np.testing.assert_allclose(gate_np.sum(axis=1), 1.0, atol=1e-5)
