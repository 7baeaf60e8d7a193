"""Decode-sized batches and expert splits at their widest: a handful of tokens, tens of thousands of experts, the expert
range cut over tens to hundreds of CTAs per token block.  With k <= 16 the chain of three kernels serves them (automatic
plan and a split forced to 64); with more, the grouped kernel, whose ranges are also swept side by side inside a CTA and
whose partial top-k lists and (max, sum) pairs are merged by the CTA that finishes last.  Every token is compared with
the oracle, including the log-sum-exp."""
import numpy as np
import pytest

from paper_2609_36301_b200 import binding as mr
from paper_2609_36301_b200 import inputs

from helpers import check_counts, check_rows, to_device

pytestmark = pytest.mark.gpu

SHAPES = [(2048, 64, 16384, 8), (4096, 64, 131072, 16)]      # h, r, M, k


@pytest.mark.parametrize("h,r,M,k", SHAPES)
@pytest.mark.parametrize("T", [1, 64, 256])
@pytest.mark.parametrize("msplit", [0, 64])
@pytest.mark.parametrize("gate_mode", [0, 1])
def test_decode_shapes(T, h, r, M, k, msplit, gate_mode):
    import torch
    case = inputs.gaussian_case(T, h, r, M, k, gate_mode, seed=77)
    X, R1, R2 = to_device(case)
    plan = mr.more_route_plan_ex(T, h, r, M, k, gate_mode, True, mr.PATH_TCGEN05, msplit)
    if msplit == 0:
        assert plan.msplit * plan.expert_ranges >= 8, "a decode-sized batch must be spread along the expert axis"
    else:
        assert plan.msplit == 64
    assert plan.chain
    res = mr.route(X, R1, R2, k, gate_mode, want_topval=True, want_lse=True, path=mr.PATH_TCGEN05, msplit=msplit)
    torch.cuda.synchronize()
    assert mr.more_route_status() == 0
    idx, gate, counts = res.idx.cpu().numpy(), res.gate.cpu().numpy(), res.counts.cpu().numpy()
    st = check_rows(case, None, idx, gate, res.topval.cpu().numpy(), res.lse.cpu().numpy(), gate_mode=gate_mode, k=k)
    check_counts(idx, counts, M, st["ref"].counts, any_differs=bool(st["differs_mask"].any()))
    # the same without the extra outputs (the variant without the softmax sweep in top-k mode)
    res2 = mr.route(X, R1, R2, k, gate_mode, path=mr.PATH_TCGEN05, msplit=msplit)
    torch.cuda.synchronize()
    assert mr.more_route_status() == 0
    assert np.array_equal(np.sort(res2.idx.cpu().numpy(), 1), np.sort(idx, 1))
    np.testing.assert_allclose(res2.gate.cpu().numpy(), gate, rtol=1e-4, atol=1e-7)


@pytest.mark.parametrize("T,h,r,M,k,msplit,ctas_per_block", [
    (1, 2048, 64, 16384, 32, 0, 32),       # the automatic plans: every list of 32 entries is merged by up to 16 threads per token
    (64, 512, 64, 131072, 32, 0, 64),
    (64, 2048, 32, 16384, 20, 0, 32),
    (256, 256, 16, 32768, 17, 0, 32),
    (256, 512, 64, 16384, 32, 64, 64),     # forced: blocks of 128 tokens, four threads per token
    (512, 128, 16, 65536, 17, 64, 64),     # ... and of 256, two
    (130, 128, 16, 4096, 32, 8, 8),        # the fewest lists that are merged that way
    (130, 128, 16, 4096, 32, 5, 5),        # one thread per token
])
@pytest.mark.parametrize("gate_mode", [0, 1])
def test_lists_of_32_entries_over_many_ctas(T, h, r, M, k, msplit, ctas_per_block, gate_mode):
    import torch
    case = inputs.gaussian_case(T, h, r, M, k, gate_mode, seed=78)
    if T > 1:
        case.X[1::7] = 0                     # tokens whose logits are all equal: the first k experts, whichever list they are in
    X, R1, R2 = to_device(case)
    plan = mr.more_route_plan_ex(T, h, r, M, k, gate_mode, gate_mode == 1, mr.PATH_TCGEN05, msplit)
    assert not plan.chain and not plan.paired and plan.msplit == ctas_per_block
    res = mr.route(X, R1, R2, k, gate_mode, want_topval=True, want_lse=gate_mode == 1, path=mr.PATH_TCGEN05, msplit=msplit)
    torch.cuda.synchronize()
    assert mr.more_route_status() == 0 and mr.debug_scratch_guard() == 1
    idx = res.idx.cpu().numpy()
    st = check_rows(case, None, idx, res.gate.cpu().numpy(), res.topval.cpu().numpy(),
                    res.lse.cpu().numpy() if gate_mode == 1 else None, gate_mode=gate_mode, k=k)
    check_counts(idx, res.counts.cpu().numpy(), M, st["ref"].counts, any_differs=bool(st["differs_mask"].any()))
    if T > 1:
        assert bool((res.idx[1::7] == torch.arange(k, device="cuda", dtype=torch.int32)).all())
