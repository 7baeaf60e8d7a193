"""Seeded random shapes through the C interface against the oracle: the low-rank router on whichever path the plan
picks (tensor-core for h, r, M multiples of 8 and r <= 64, CUDA-core otherwise), forced expert splits, and the fused
standard router.  The shapes are drawn once from a fixed seed, so the cases are the same on every run."""
import numpy as np
import pytest

from paper_2609_36301_b200 import binding as mr
from paper_2609_36301_b200 import inputs

from helpers import check_counts, check_rows, to_device

pytestmark = pytest.mark.gpu


def _cases(n, seed, tensor_core):
    rng = np.random.default_rng(seed)
    out = []
    for _ in range(n):
        if tensor_core:
            h = int(rng.integers(1, 40)) * 8
            r = int(rng.choice([8, 16, 24, 32, 40, 48, 64]))
            M = int(rng.integers(1, 300)) * 8
        else:
            h = int(rng.integers(3, 200))
            r = int(rng.integers(1, 70))
            M = int(rng.integers(2, 1500))
        T = int(rng.integers(1, 700))
        k = int(min(M, rng.choice([1, 2, 3, 4, 6, 8, 8, 8, 12, 16, 20, 32])))
        gate_mode = int(rng.integers(0, 2))
        msplit = int(rng.choice([0, 0, 0, 1, 2, 3, 5]))
        out.append((T, h, r, M, k, gate_mode, msplit))
    return out


def _route_and_check(case, path, msplit):
    import torch
    X, R1, R2 = to_device(case)
    res = mr.route(X, R1, R2, case.k, case.gate_mode, want_topval=True, want_lse=True, path=path, msplit=msplit)
    torch.cuda.synchronize()
    assert mr.more_route_status() == 0
    idx = res.idx.cpu().numpy()
    stats = check_rows(case, None, idx, res.gate.cpu().numpy(), res.topval.cpu().numpy(), res.lse.cpu().numpy())
    check_counts(idx, res.counts.cpu().numpy(), case.M, stats["ref"].counts, bool(stats["differs_mask"].any()))


@pytest.mark.parametrize("T,h,r,M,k,gate_mode,msplit", _cases(24, 2024, True))
def test_random_shapes_tensor_core_path(T, h, r, M, k, gate_mode, msplit):
    case = inputs.gaussian_case(T, h, r, M, k, gate_mode, seed=T + M)
    plan = mr.more_route_plan(T, h, r, M, k, gate_mode, mr.PATH_TCGEN05, msplit)
    assert plan.path == mr.PATH_TCGEN05
    _route_and_check(case, mr.PATH_TCGEN05, msplit)


@pytest.mark.parametrize("T,h,r,M,k,gate_mode,msplit", _cases(12, 77, False))
def test_random_shapes_any_path(T, h, r, M, k, gate_mode, msplit):
    case = inputs.gaussian_case(T, h, r, M, k, gate_mode, seed=T + M)
    _route_and_check(case, mr.PATH_AUTO, 0)


@pytest.mark.parametrize("T,h,r,M,k,gate_mode,msplit", _cases(12, 4242, True))
def test_random_shapes_standard_router(T, h, r, M, k, gate_mode, msplit):
    import torch
    h = min(h, 256)                                         # the oracle forms z = X I_h: keep the identity small
    case = inputs.full_rank_case(T, h, M, k, gate_mode, seed=T + M)
    X, _, W = to_device(case)
    idx = torch.empty((T, k), dtype=torch.int32, device="cuda")
    gate = torch.empty((T, k), dtype=torch.float32, device="cuda")
    counts = torch.empty((M,), dtype=torch.int32, device="cuda")
    topval = torch.empty((T, k), dtype=torch.float32, device="cuda")
    lse = torch.empty((T,), dtype=torch.float32, device="cuda")
    mr.more_route_full(X, W, k, gate_mode, idx, gate, counts, topval, lse, msplit)
    torch.cuda.synchronize()
    assert mr.more_route_status() == 0
    stats = check_rows(case, None, idx.cpu().numpy(), gate.cpu().numpy(), topval.cpu().numpy(), lse.cpu().numpy())
    check_counts(idx.cpu().numpy(), counts.cpu().numpy(), M, stats["ref"].counts, bool(stats["differs_mask"].any()))


def _pattern(rng, gen, M):
    """Logits of one kind of token: rising, falling, plateaus, few distinct values, a few spikes."""
    import torch
    e = torch.arange(M, device="cuda")
    cut = M * int(rng.integers(1, 9)) // 8
    what = int(rng.integers(0, 8))
    if what == 0:
        return torch.where(e < cut, torch.exp2(16.0 * e / M), -1.0)
    if what == 1:
        return torch.where(e < cut, torch.exp2(16.0 * (M - e) / M), -1.0)
    if what == 2:
        return -torch.exp2(16.0 * e / M)
    if what == 3:
        return torch.where((e // int(rng.choice([4, 32, 128, 1000]))) % 2 == 0, torch.exp2(10.0 * e / M), 0.0)
    if what == 4:
        return (e % int(rng.choice([3, 32, 128, 129]))).float()
    if what == 5:
        return torch.randn(M, generator=gen, device="cuda").round()
    if what == 6:
        v = torch.zeros(M, device="cuda")
        v[torch.randint(0, M, (12,), generator=gen, device="cuda")] = 3.0
        return v
    return torch.randn(M, generator=gen, device="cuda")


@pytest.mark.parametrize("seed", range(48))
def test_patterned_logits(seed):
    """Tokens with one element of z, so that the logits are exact and the whole result, ties included, is that of a stable
    sort: eight kinds of logits side by side, which overflow lists in turn and are full of equals.  Every third case has
    rows of infinities and NaN among them, which must not touch the others."""
    import torch
    rng, gen = np.random.default_rng(9000 + seed), torch.Generator(device="cuda").manual_seed(seed)
    k = int(rng.choice([1, 2, 4, 8, 8, 12, 16, 16, 20, 32]))
    M = 8 * int(2 ** rng.uniform(4, 13.5))
    T = int(2 ** rng.uniform(0, min(15.0, np.log2(3e8 / M))))
    h, gate_mode, msplit = int(rng.choice([8, 72, 512, 2048])), int(rng.integers(0, 2)), int(rng.choice([0, 0, 0, 1, 3, 64]))
    R2 = torch.stack([_pattern(rng, gen, M) for _ in range(8)]).to(torch.bfloat16)
    X = torch.zeros((T, h), device="cuda")
    X[torch.arange(T, device="cuda"), torch.randint(0, 8, (T,), generator=gen, device="cuda")] = \
        1 + torch.rand(T, generator=gen, device="cuda")
    X = X.to(torch.bfloat16)
    R1 = torch.eye(h, device="cuda")[:, :8].to(torch.bfloat16).contiguous()
    rows = torch.randint(0, T, (min(T, 256),), generator=gen, device="cuda")
    val, idx = (X[rows, :8].double() @ R2.double()).sort(dim=1, descending=True, stable=True)
    if seed % 3 == 0:
        bad = torch.randint(0, T, (max(1, T // 50),), generator=gen, device="cuda")
        X[bad, int(rng.integers(0, 8))] = float(rng.choice([2e38, np.inf, -np.inf, np.nan]))
        keep = ~torch.isin(rows, bad)
        rows, val, idx = rows[keep], val[keep], idx[keep]
    res = mr.route(X, R1, R2, k, gate_mode, want_topval=True, want_lse=True, path=mr.PATH_TCGEN05, msplit=msplit)
    torch.cuda.synchronize()
    assert mr.more_route_status() == 0 and mr.debug_scratch_guard() == 1
    assert torch.equal(res.idx[rows], idx[:, :k].int())
    assert torch.equal(res.topval[rows].double(), val[:, :k])
    lse = torch.logsumexp(val, 1)
    # (sums of exponentials of logits up to 2^17 in fp32: their difference from the maximum is rounded to 2^-24 of that)
    assert bool(((res.lse[rows].double() - lse).abs() <= 1e-4 * (1 + lse.abs())).all())
    valid = res.idx[(res.idx >= 0) & (res.idx < M)]
    assert torch.equal(torch.bincount(valid.long(), minlength=M).int(), res.counts)
