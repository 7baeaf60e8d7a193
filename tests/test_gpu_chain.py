"""The chain projection -> sweep -> finish of the low-rank router, at the edges of its tiles: token blocks of 128, units of
128 experts, K-steps of 16 ranks, the three finishing kernels (few, up to 64 and more segments per token), lists that
overflow, equal logits, and a call that is cut into chunks of tokens."""
import numpy as np
import pytest

from paper_2609_36301_b200 import binding as mr
from paper_2609_36301_b200 import inputs

from helpers import check_counts, check_rows, to_device

pytestmark = pytest.mark.gpu


def _route_and_check(case, rows=None, launches=3):
    import torch
    X, R1, R2 = to_device(case)
    before = mr.launches()
    res = mr.route(X, R1, R2, case.k, case.gate_mode, want_topval=True, want_lse=case.gate_mode == 1)
    assert mr.launches() - before == launches, "this shape is not served by the chain"
    torch.cuda.synchronize()
    assert mr.more_route_status() == 0
    sel = slice(None) if rows is None else torch.from_numpy(rows).cuda()
    st = check_rows(case, rows, res.idx[sel].cpu().numpy(), res.gate[sel].cpu().numpy(), res.topval[sel].cpu().numpy(),
                    None if res.lse is None else res.lse[sel].cpu().numpy(), gate_mode=case.gate_mode, k=case.k)
    counts = res.counts.cpu().numpy()
    if rows is None:
        check_counts(res.idx.cpu().numpy(), counts, case.M, st["ref"].counts, bool(st["differs_mask"].any()))
    else:
        check_counts(res.idx.cpu().numpy(), counts, case.M)
    return st


@pytest.mark.parametrize("gate_mode", [0, 1])
@pytest.mark.parametrize("T,h,r,M,k", [
    (1, 8, 8, 512, 1),            # one token, one k-tile, four whole units
    (127, 72, 16, 520, 8),        # the last token row empty, a unit with eight live experts
    (129, 128, 24, 640, 9),       # a second block with one token, lists longer than 8
    (300, 200, 40, 1016, 16),     # three K-steps, the last unit short of eight experts
    (1000, 512, 48, 4104, 13),    # a unit with eight live experts, lists longer than 8
    (2000, 96, 56, 2000, 16),     # the longest lists
    (130, 1024, 32, 128, 16),     # a single unit
    (700, 512, 16, 264, 3),       # two whole units and eight experts
    (4100, 64, 64, 1024, 4),      # more token blocks than three per part: parts that begin inside a block
    (8500, 64, 32, 3072, 8),      # one or two segments per token: the finishing kernel with eight threads per token
    (40, 256, 64, 65536, 8),      # hundreds of segments per token: a CTA per token finishes
])
def test_edges(T, h, r, M, k, gate_mode):
    _route_and_check(inputs.gaussian_case(T, h, r, M, k, gate_mode, seed=T + M))


@pytest.mark.parametrize("k", [1, 3, 5, 8, 16])
@pytest.mark.parametrize("tail", [8, 24, 32, 40, 56, 64, 72, 120])
@pytest.mark.parametrize("T", [1, 130])
def test_a_part_of_few_experts(T, tail, k):
    """One unit per CTA, the last of fewer than 128 experts: the threshold of its tokens comes from those alone."""
    _route_and_check(inputs.gaussian_case(T, 128, 40, 1024 + tail, k, k & 1, seed=tail + k))


@pytest.mark.parametrize("T,h,r,M,k", [(300, 128, 32, 4096, 8), (64, 128, 64, 16384, 20), (20000, 64, 16, 512, 8), (45000, 64, 16, 512, 4)])
def test_the_plan_names_the_kernels_that_run(T, h, r, M, k):
    import torch
    plan = mr.more_route_plan_ex(T, h, r, M, k)
    X, R1, R2 = to_device(inputs.gaussian_case(T, h, r, M, k, 0, seed=2))
    before = mr.launches()
    mr.route(X, R1, R2, k, 0)
    torch.cuda.synchronize()
    assert mr.more_route_status() == 0
    assert mr.launches() - before == (3 if plan.chain else 1)


@pytest.mark.parametrize("k", [1, 8, 16])
@pytest.mark.parametrize("descending", [False, True])
def test_logits_that_rise_or_fall_with_the_expert_id(k, descending):
    """Every expert beats the threshold so far (the lists overflow again and again), or none does after the first."""
    case = inputs.gaussian_case(200, 64, 8, 4096, k, 0, seed=13)
    R1f = np.zeros((64, 8), dtype=np.float32)
    R1f[0, 0] = 1.0
    Xf = inputs.bf16_bits_to_f32(case.X)
    Xf[:, 0] = np.abs(Xf[:, 0]) + 0.5
    ramp = np.arange(4096, dtype=np.float32) / 512.0
    R2f = np.zeros((8, 4096), dtype=np.float32)
    R2f[0] = -ramp if descending else ramp
    case.X, case.R1, case.R2 = inputs.to_bf16_bits(Xf), inputs.to_bf16_bits(R1f), inputs.to_bf16_bits(R2f)
    _route_and_check(case)


@pytest.mark.parametrize("T,M", [(64, 2048), (3000, 1024), (8500, 3072)])
def test_all_logits_equal(T, M):
    """Nothing beats anything: the first k experts are selected."""
    import torch
    case = inputs.gaussian_case(T, 64, 16, M, 8, 0, seed=3)
    case.R2[:] = case.R2[:, :1]
    X, R1, R2 = to_device(case)
    res = mr.route(X, R1, R2, 8, 0)
    torch.cuda.synchronize()
    assert mr.more_route_status() == 0
    assert bool((res.idx == torch.arange(8, device="cuda", dtype=torch.int32)).all())
    assert int(res.counts[:8].sum()) == 8 * T and int(res.counts[8:].sum()) == 0


def test_more_tokens_than_one_chunk():
    T = 131072 + 130
    case = inputs.gaussian_case(T, 64, 8, 32768, 4, 0, seed=9)
    rows = np.concatenate([np.arange(64), np.arange(131072 - 64, T)])
    _route_and_check(case, rows, launches=6)


@pytest.mark.parametrize("T,M,k,msplit,sweeps", [
    (9000, 4096, 8, 16, 4),           # 71 token blocks, 18 per sweep
    (5000, 16384, 12, 64, 10),        # 40 token blocks, 4 per sweep
    (40000, 8192, 4, 1, 2),           # one CTA per token block, 296 of 313 blocks in the first sweep
    (131072 + 130, 8192, 4, 3, 12),   # two chunks: 98 token blocks per sweep, then two blocks
])
def test_a_forced_split_in_several_sweeps(T, M, k, msplit, sweeps):
    """More CTAs than are resident at once: as many sweeps as that takes, the same results as without a split."""
    import torch
    case = inputs.gaussian_case(T, 64, 8, M, k, 1, seed=T)
    X, R1, R2 = to_device(case)
    whole = mr.route(X, R1, R2, k, 1, want_topval=True, want_lse=True)
    before = mr.launches()
    res = mr.route(X, R1, R2, k, 1, want_topval=True, want_lse=True, msplit=msplit)
    assert mr.launches() - before == (2 if T > 131072 else 1) + 2 * sweeps
    torch.cuda.synchronize()
    assert mr.more_route_status() == 0 and mr.debug_scratch_guard() == 1
    for a, b in ((res.idx, whole.idx), (res.topval, whole.topval), (res.counts, whole.counts)):
        assert torch.equal(a, b)
    # (the sums of exponentials are added segment by segment: fp32 rounding of a few additions)
    assert float((res.lse - whole.lse).abs().max()) <= 1e-5
    np.testing.assert_allclose(res.gate.cpu().numpy(), whole.gate.cpu().numpy(), rtol=2e-5)
    rows = np.unique(np.concatenate([np.arange(32), np.arange(T // 2, T // 2 + 32), np.arange(T - 32, T)]))
    sel = torch.from_numpy(rows).cuda()
    check_rows(case, rows, res.idx[sel].cpu().numpy(), res.gate[sel].cpu().numpy(), res.topval[sel].cpu().numpy(),
               res.lse[sel].cpu().numpy(), gate_mode=1, k=k)


@pytest.mark.parametrize("k,gate_mode", [(8, 1), (12, 0)])
def test_long_segments(k, gate_mode):
    """More than 32 units per segment: the leading units are computed twice, the threshold rises on the way."""
    case = inputs.gaussian_case(4800, 64, 16, 36008, k, gate_mode, seed=17)
    _route_and_check(case, np.concatenate([np.arange(40), np.arange(2400, 2440), np.arange(4760, 4800)]))


@pytest.mark.parametrize("T,M,k", [(3, 256, 16), (40, 16384, 8), (300, 65536, 16), (3000, 4096, 8), (4100, 8192, 16), (4800, 36008, 8)])
def test_tokens_of_zeros(T, M, k):
    """Padding: every third token is zero, so all its logits are equal; the others are as ever."""
    case = inputs.gaussian_case(T, 512, 16, M, k, 1, seed=19)
    case.X[::3] = 0
    _route_and_check(case, None if T < 1000 else np.arange(T - 64, T))
    import torch
    res = mr.route(*to_device(case), k, 1)
    assert bool((res.idx[::3] == torch.arange(k, device="cuda", dtype=torch.int32)).all())


@pytest.mark.parametrize("zeros", [False, True])
@pytest.mark.parametrize("T,M,k", [
    (290, 2048, 8),        # 16 segments per token: CTAs of 512 threads
    (296, 2048, 16),       # the most tokens that they take
    (297, 2048, 16),       # 16 segments: CTAs of 128 threads
    (310, 4096, 8),
    (700, 8200, 16),       # 49 segments of one or two units
    (700, 6152, 16),       # 49 segments of one unit, the last of 8 experts
    (600, 1024, 16),       # 8 segments
    (700, 1024, 16),       # 8 segments: a warp per token, candidates in registers
    (1300, 4096, 4),       # 26 segments
    (1300, 512, 4),        # four segments: the short code
])
def test_finishing_by_the_number_of_segments(T, M, k, zeros):
    case = inputs.gaussian_case(T, 64, 16, M, k, 1, seed=23)
    if zeros:
        case.X[::5] = 0
    _route_and_check(case)


@pytest.mark.parametrize("gate_mode", [0, 1])
@pytest.mark.parametrize("T,M,k", [
    (300, 16384, 8),       # one or two units per segment
    (8000, 16384, 2),      # 27 units, the threshold final from the start
    (4800, 36008, 16),     # long segments of lists longer than 8
    (4800, 36008, 8),
    (40, 65536, 8),        # hundreds of segments per token
    (8500, 3072, 8),       # the finishing kernel with eight threads per token
])
def test_infinite_logits(T, M, k, gate_mode):
    """Finite inputs whose logits overflow: a token for which every second expert's logit is +inf, one with three such experts
    among equals.  They are logits like any other (the lists must not grow past their end), other tokens are unaffected."""
    import torch
    gen = torch.Generator(device="cuda").manual_seed(T + M + k)
    X = torch.randn((T, 64), generator=gen, device="cuda").to(torch.bfloat16)
    R1 = (torch.randn((64, 8), generator=gen, device="cuda") / 8).to(torch.bfloat16)
    R2 = torch.randn((8, M), generator=gen, device="cuda").to(torch.bfloat16)
    R1[0], R1[1] = 0, 0
    R1[0, 0] = R1[1, 1] = 1
    R2[0, ::2], R2[0, 1::2] = 4, 1
    R2[1], few = 0, torch.tensor([M // 3, M // 2, M - 1], device="cuda")
    R2[1, few] = 4
    half, three = torch.arange(5, T, 97, device="cuda"), torch.arange(6, T, 97, device="cuda")
    X[half], X[three] = 0, 0
    clean = mr.route(X, R1, R2, k, gate_mode, want_topval=True)
    X[half, 0], X[three, 1] = 2e38, 2e38
    res = mr.route(X, R1, R2, k, gate_mode, want_topval=True)
    assert mr.more_route_plan_ex(T, 64, 8, M, k, gate_mode).chain
    torch.cuda.synchronize()
    assert mr.more_route_status() == 0 and mr.debug_scratch_guard() == 1
    assert bool((res.idx[half] == 2 * torch.arange(k, device="cuda", dtype=torch.int32)).all())
    assert bool(torch.isinf(res.topval[half]).all())
    want = torch.cat([few.int(), torch.arange(k, device="cuda", dtype=torch.int32)])[:k]
    assert bool((res.idx[three] == want).all())
    others = torch.ones(T, dtype=torch.bool, device="cuda")
    others[half], others[three] = False, False
    assert torch.equal(res.idx[others], clean.idx[others]) and torch.equal(res.gate[others], clean.gate[others])
    check_counts(res.idx.cpu().numpy(), res.counts.cpu().numpy(), M)


@pytest.mark.parametrize("equals", [False, True])
@pytest.mark.parametrize("T,M,k", [(4800, 36008, 16), (4800, 36008, 8), (4800, 36008, 3), (2000, 131072, 8), (8000, 16384, 12)])
def test_lists_that_overflow_at_different_times(T, M, k, equals):
    """A warp makes room in all its lists when one overflows.  Eight kinds of tokens side by side, whose logits rise with the
    expert id up to an eighth, two eighths, ... of the experts and are low from there on, so that lists overflow in turn;
    with `equals`, tokens of zeros but for three experts stand between them."""
    import torch
    gen = torch.Generator(device="cuda").manual_seed(M + k)
    e = torch.arange(M, device="cuda")
    X = torch.zeros((T, 64), device="cuda")
    kind = torch.arange(T, device="cuda") % 8
    X[torch.arange(T, device="cuda"), kind] = 1 + torch.rand(T, generator=gen, device="cuda")
    R1 = torch.eye(64, device="cuda")[:, :8]
    R2 = torch.stack([torch.where(e < M * (j + 1) // 8, torch.exp2(20.0 * e / M), -1.0) for j in range(8)])
    if equals:
        R2[1::2] = 0
        R2[1::2, torch.tensor([M // 5, M // 3, M - 1], device="cuda")] = 3
    X, R1, R2 = X.to(torch.bfloat16), R1.to(torch.bfloat16).contiguous(), R2.to(torch.bfloat16)
    assert mr.more_route_plan_ex(T, 64, 8, M, k, 0).chain
    res = mr.route(X, R1, R2, k, 0, want_topval=True)
    torch.cuda.synchronize()
    assert mr.more_route_status() == 0 and mr.debug_scratch_guard() == 1
    # (z has one element that is not zero, and it is a bf16: the logits are exact in fp32)
    rows = torch.cat([torch.arange(i, i + 64, device="cuda") for i in range(0, T - 63, max(64, T // 12))])
    val, idx = (X[rows, :8].float() @ R2.float()).sort(dim=1, descending=True, stable=True)
    assert torch.equal(res.topval[rows], val[:, :k])
    assert torch.equal(res.idx[rows], idx[:, :k].int())
    check_counts(res.idx.cpu().numpy(), res.counts.cpu().numpy(), M)


def test_what_an_earlier_call_left_behind_the_last_token_is_not_swept():
    """Rows of z behind the last token are not written.  An earlier call leaves large values there, with which the weights of
    this one overflow to infinity: such rows must not be taken for tokens that beat every threshold (their lists would
    overflow all the time; the call took 20 times as long)."""
    import torch
    T, h, r, M, k = 57 * 128 - 12, 256, 8, 16384, 2              # two CTAs share a block's projection, and 25 units per sweep
    gen = torch.Generator(device="cuda").manual_seed(5)
    X, R1, R2 = (torch.randn(s, generator=gen, device="cuda").to(torch.bfloat16) for s in ((T, h), (h, r), (r, M)))
    R1 /= 16
    R2[0] = 8 + R2[0].abs()

    def timed(leftover):
        X0 = torch.zeros((T + 12, h), dtype=torch.bfloat16, device="cuda")
        R10 = torch.zeros((h, r), dtype=torch.bfloat16, device="cuda")
        X0[:, 0], R10[0, 0] = 1.0, leftover
        mr.route(X0, R10, torch.zeros_like(R2), k, 0)
        best = 1e9
        for _ in range(5):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            torch.cuda.synchronize()
            a.record()
            res = mr.route(X, R1, R2, k, 0, want_topval=True)
            b.record()
            b.synchronize()
            best = min(best, a.elapsed_time(b))
        assert mr.more_route_status() == 0
        return best, res

    assert mr.more_route_plan_ex(T, h, r, M, k).chain
    clean, res = timed(0.0)
    left, res2 = timed(1e38)
    assert torch.equal(res.idx, res2.idx) and torch.equal(res.topval, res2.topval)
    assert left < 2 * clean, f"{clean * 1e3:.0f} us with zeros behind the last token, {left * 1e3:.0f} us with large values"
