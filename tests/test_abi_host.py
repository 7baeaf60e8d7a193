"""Host-side checks that need no GPU: the shared library loads, exports every symbol the header declares,
rejects bad arguments before touching a device, and plans launches sensibly."""
import ctypes
import os
import re

import numpy as np
import pytest

from paper_2609_36301_b200 import binding as mr
from paper_2609_36301_b200 import build as mr_build

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def declared_functions():
    text = open(os.path.join(ROOT, "include", "more_route.h")).read()
    text = re.sub(r"/\*.*?\*/", "", text, flags=re.S)
    return sorted(set(re.findall(r"\b(more_[a-z_0-9]+)\s*\(", text)))


def test_library_builds_and_exports_every_declared_symbol():
    mr_build.build()
    lib = mr.lib()
    names = declared_functions()
    assert {"more_route", "more_route_ex", "more_route_host", "more_route_plan", "more_route_status",
            "more_strerror", "more_version", "more_route_launches"} <= set(names)
    for n in names:
        assert hasattr(lib, n), f"{n} is declared in more_route.h but not exported"
    assert mr.version() >= 100
    assert "ok" == mr.strerror(0)


def test_bad_arguments_are_rejected_before_any_device_work():
    lib = mr.lib()
    buf = (ctypes.c_char * 4096)()
    p = ctypes.addressof(buf)
    p16 = (p + 15) & ~15
    def call(X=p16, R1=p16, R2=p16, T=4, h=8, r=8, M=8, k=2, mode=0, idx=p16, gate=p16, counts=p16):
        return lib.more_route(X, R1, R2, T, h, r, M, k, mode, idx, gate, counts, None)
    assert call(k=9) == -2            # k > M
    assert call(k=0) == -2
    assert call(T=-1) == -2
    assert call(M=40, k=33) == -2     # k > MORE_K_MAX
    assert call(r=2048) == -2         # r > MORE_R_MAX
    assert call(M=(1 << 30) + 8) == -2   # M > MORE_M_MAX
    assert call(mode=2) == -4
    assert call(X=None) == -1
    assert call(counts=None) == -1
    assert call(X=p16 + 2) == -3
    assert call(idx=p16 + 1) == -3
    assert lib.more_route_ex(p16, p16, p16, 4, 8, 8, 8, 2, 0, p16, p16, p16, None, None, 7, 0, None) == -4
    for code in range(-8, 1):
        assert len(mr.strerror(code)) > 1


def test_plan_picks_paths_and_splits():
    P = mr.more_route_plan
    assert P(256, 128, 8, 256, 2).path == mr.PATH_TCGEN05
    assert P(100, 20, 5, 33, 3).path == mr.PATH_GENERIC          # odd sizes
    assert P(64, 64, 96, 256, 4).path == mr.PATH_GENERIC         # r > 64
    assert P(64, 64, 8, 260, 4).path == mr.PATH_GENERIC          # M % 8 != 0
    with pytest.raises(mr.MoreRouteError):
        P(100, 20, 5, 33, 3, path=mr.PATH_TCGEN05)
    with pytest.raises(mr.MoreRouteError):
        P(300, 256, 32, 4096, 8, msplit=65)                      # more than 64 CTAs per token block
    PX = mr.more_route_plan_ex
    # few token blocks, many experts: the experts are split, inside a CTA and over CTAs, and one wave is not exceeded
    p = PX(8192, 4096, 64, 131072, 16, gate_mode=1)
    assert p.ctas % p.msplit == 0 and p.ctas <= (296 if p.chain else 148)
    assert p.msplit * p.expert_ranges >= 4 and p.token_groups * p.expert_ranges <= 4
    # many tokens: the kernel with 256-token CTAs, two per SM, in one wave
    p = PX(65536, 2048, 64, 16384, 8)
    assert p.ctas in range(256, 297) and p.msplit == 1
    # a decode-sized batch is spread over the SMs along the expert axis
    p = PX(64, 2048, 64, 16384, 8)
    assert p.ctas > 16 and p.ctas <= 148 and p.msplit > 1
    # never more CTAs per token block than 64-expert blocks
    assert PX(300, 256, 32, 256, 8, msplit=5).msplit * PX(300, 256, 32, 256, 8, msplit=5).expert_ranges <= 4
    assert P(300, 256, 32, 4096, 8, msplit=5).msplit == 5
    # asking for the log-sum-exp changes the kernel variant but is always accepted
    assert PX(32768, 512, 32, 16384, 8, want_lse=True).path == mr.PATH_TCGEN05


def test_plan_names_the_kernel_and_its_real_numbers():
    """The chain's plan is its sweep's: two CTAs per SM, 128 tokens each, one expert range per CTA."""
    PX = mr.more_route_plan_ex
    p = PX(8192, 4096, 64, 131072, 16, gate_mode=1)              # parts that begin anywhere: 296 of them for 64 token blocks
    assert p.chain and not p.paired
    assert (p.ctas, p.msplit, p.block_tokens, p.token_groups, p.expert_ranges) == (296, 4, 128, 1, 1)
    p = PX(1, 2048, 64, 16384, 8)                                # one CTA per unit of 128 experts
    assert p.chain and (p.ctas, p.msplit) == (128, 128)
    p = PX(300, 256, 32, 4096, 8, msplit=5)                      # forced
    assert p.chain and (p.ctas, p.msplit) == (15, 5)
    p = PX(9000, 64, 8, 4096, 8, msplit=64)                      # no more CTAs than the 32 units of 128 experts
    assert p.chain and (p.ctas, p.msplit) == (71 * 32, 32)
    p = PX(65536, 2048, 64, 16384, 8)
    assert p.paired and not p.chain
    p = PX(32768, 512, 32, 1024, 8)
    assert not p.paired and not p.chain and p.token_groups * p.expert_ranges <= 4 and p.ctas <= 148
    assert not PX(64, 2048, 64, 16384, 32).chain                 # more than 16: the chain does not take it
    assert not PX(100, 20, 5, 33, 3).chain


def test_choice_of_the_chain_has_no_holes():
    """More experts or fewer tokens never take a shape off the chain, nor does a smaller k within a class of buckets."""
    def chain(T, M, k, h, gate):
        return mr.more_route_plan_ex(T, h, 32, M, k, gate).chain

    Ts = [1, 1000, 3000, 5000, 8000, 11000, 14000, 16000, 18000, 25000, 34000, 36000, 45000, 50400, 55000, 65536, 200000]
    Ms = [64, 120, 128, 256, 512, 1016, 1024, 1536, 2048, 3072, 4096, 8192, 12000, 16384, 20000, 24576, 32768, 65536, 131072]
    for h in (128, 1024, 4096, 16384):
        for gate in (0, 1):
            for k in (1, 4, 5, 8, 9, 16):
                grid = [[chain(T, M, k, h, gate) for M in Ms] for T in Ts]
                for row in grid:
                    assert row == sorted(row), (h, gate, k)
                for column in zip(*grid):
                    assert list(column) == sorted(column, reverse=True), (h, gate, k)
                assert all(grid[0][2:]) or h < 512, "a single token is always served by the chain"
    for T, M in ((1, 128), (16000, 16384), (16000, 24576), (30000, 4096), (40000, 65536)):
        assert chain(T, M, 4, 2048, 0) == chain(T, M, 1, 2048, 0) and chain(T, M, 8, 2048, 0) == chain(T, M, 5, 2048, 0)


@pytest.mark.parametrize("T,h,r,M,k,gate,us_chain,us_one", [
    (15019, 2048, 64, 208, 4, 0, 48.8, 32.9), (16652, 2680, 16, 168, 3, 1, 54.2, 34.8), (25521, 3608, 48, 440, 4, 1, 82.7, 72.7),
    (9947, 3728, 40, 304, 15, 1, 84.7, 64.9), (14350, 1728, 40, 240, 3, 0, 38.2, 32.8), (1651, 136, 24, 144, 2, 1, 14.2, 23.4),
    (6229, 128, 16, 304, 2, 0, 14.2, 20.8), (23020, 512, 16, 504, 1, 0, 25.9, 39.2), (50540, 1024, 48, 6784, 6, 0, 148.0, 182.0),
    (45337, 584, 48, 8056, 5, 0, 125.9, 193.8), (54277, 136, 48, 9704, 7, 0, 161.7, 217.8), (36910, 2048, 64, 728, 12, 0, 120.4, 95.4),
])
def test_choice_of_the_quicker_kernel(T, h, r, M, k, gate, us_chain, us_one):
    """Shapes near the lines of the choice whose two sides were measured far apart (microseconds on B200)."""
    assert mr.more_route_plan_ex(T, h, r, M, k, gate).chain == (us_chain < us_one)


def test_shared_memory_plan_of_the_grouped_kernel_fits():
    """Every (rank, token groups, expert ranges) the planner may pick leaves room for at least two R2 stages and one
    phase-1 stage in the 208 KB ring (checked through the plans of shapes that exercise them)."""
    PX = mr.more_route_plan_ex
    for T in (1, 33, 128, 200, 300, 512, 5000, 20000):
        for r in (8, 16, 32, 64):
            for M in (8, 64, 256, 1000, 4096, 65536):
                for k in (1, 8, 16, 32):
                    if k > M:
                        continue
                    p = PX(T, 512, r, M - M % 8 if M >= 8 else 8, k)
                    assert p.path == mr.PATH_TCGEN05 and p.ctas >= 1
                    assert p.block_tokens % 32 == 0 and 32 <= p.block_tokens <= 512


def test_device_memory_of_a_routing_call_is_bounded():
    """The sweep's lists are sized for the CTAs that run at once (two per SM, 1 MiB each at most), whatever split of the
    experts is forced, and for the tokens and experts that a CTA has: T tokens of z, lists, candidates."""
    B = mr.debug_scratch_bytes
    MiB = 1 << 20

    def bound(T, r, M, k):
        blocks = -(-min(T, 131072) // 128)
        z = blocks * 128 * (128 if r <= 32 else 256)
        segments = 2 * 148 + 2 * blocks
        return z + 2 * 148 * MiB + segments * 128 * (4 * k * 8 + 12) + MiB

    for T, M, k in ((131072, 16384, 4), (65536, 65536, 4), (65536, 16384, 16), (4096, 131072, 16), (300000, 32768, 4), (300, 65536, 8)):
        for msplit in (0, 1, 2, 7, 64):
            assert B(T, 512, 64, M, k, 1, msplit=msplit) <= bound(T, 64, M, k), (T, M, k, msplit)
    # largest there is without a forced split
    assert B(131072, 512, 64, 131072, 16, 1) <= 512 * MiB
    # few tokens: only the rows that are there, and no longer lists than a CTA's experts can fill
    assert B(1, 2048, 64, 16384, 8) <= 9 * MiB
    assert B(64, 4096, 64, 131072, 16) <= 96 * MiB


def test_a_full_list_ends_inside_its_area():
    """The sweep advances the end of a list by adds to the low word of its address.  So whatever the scratch's address, no place of
    a list may lie behind a multiple of 2^32 bytes that the first one lies before, and the place behind the last entry that a
    CTA's units can add (eight each) has to be one of them.  (Lists of 64 places are cut at 56 and end at 60 at most.)"""
    shapes = [(T, M, k) for T in (1, 40, 128, 300, 1000, 2000, 4800) for M in (128, 1024, 5800, 16384, 40000, 131072) for k in (1, 8, 16)]
    shapes += [(131072, 8192, 4), (131072 + 130, 32768, 4), (20000, 16384, 16)]
    checked = set()
    for T, M, k in shapes:
        for msplit in (0, 1, 3, 16, 64):
            if not mr.more_route_plan_ex(T, 512, 64, M, k, msplit=msplit).chain:
                continue
            size = mr.debug_scratch_bytes(T, 512, 64, M, k, msplit=msplit)
            at, areas, places, step = mr.debug_chain_lists(T, 512, 64, M, k, msplit=msplit, scratch=1 << 40)
            # the largest part of the units: equal parts of all blocks, or of one block each
            blocks, units = -(-min(T, 131072) // 128), -(-M // 128)
            if T <= 131072:
                ctas = mr.more_route_plan_ex(T, 512, 64, M, k, msplit=msplit).ctas
                most = -(-blocks * units // ctas) if not msplit else -(-units // min(msplit, units))
            else:
                most = 64
            assert 8 * most < places or places == 64, (T, M, k, msplit)
            checked.add(places)
            area = places * step
            for where in (0, 256, area // 2, area - 256, area, area + 256, 2 * area - 16384, (areas - 1) * area + 512, areas * area - 256,
                          areas * area, (areas + 1) * area - 256, (areas + 1) * area):
                scratch = (9 << 32) - (at - (1 << 40)) - where // 256 * 256
                first = mr.debug_chain_lists(T, 512, 64, M, k, msplit=msplit, scratch=scratch)[0]
                assert first % 256 == 0 and scratch <= first and first + areas * area <= scratch + size
                for a in (first + i * area for i in range(areas)):
                    assert a >> 32 == a + area - 1 >> 32, (T, M, k, msplit, where)
                # as the kernel does it: the last thread's list, filled to its last entry
                for a in (first + i * area for i in range(areas)):
                    begin = a + step - 32
                    n = min(8 * most, 60)
                    end = begin & ~0xffffffff | begin + n * step & 0xffffffff
                    assert (end - begin) // step == n
    assert {9, 17, 33, 64} <= checked


@pytest.mark.parametrize("T,h,M,most,us,us_more", [
    (2737, 3800, 7136, 148, 51.4, 82.2), (1218, 3520, 15256, 148, 38.0, 54.7), (46814, 1008, 312, 200, 27.4, 34.0),
    (18993, 744, 184, 100, 18.9, 22.7), (1068, 2824, 29056, 148, 48.6, 73.0), (5902, 2872, 4304, 148, 41.4, 57.9),
])
def test_column_sums_take_no_more_ctas_than_pay(T, h, M, most, us, us_more):
    """Shapes with a large projection and few tiles for each CTA, which up to `most` CTAs finish in `us` and more of them in
    `us_more` (microseconds on B200)."""
    block, split = mr.debug_psum_plan(T, h, M)
    assert -(-T // block) * split <= most, (block, split, us, us_more)


def test_cut_of_the_column_sums_is_sound():
    for T in (1, 128, 129, 160, 161, 300, 1000, 5000, 40000, 47360, 47361, 65536, 1 << 20):
        for h in (8, 512, 4096):
            for M in (8, 128, 1000, 8192, 131072):
                block, split = mr.debug_psum_plan(T, h, M)
                tiles = -(-M // 128)
                assert block == 128 if T <= 128 else block in (160, 192, 224, 256)
                assert 1 <= split <= tiles and -(-T // block) * split <= max(296, -(-T // block))


def test_the_guard_begins_where_the_lists_end():
    """The sweep's lists are the last of the scratch, and what is written behind them is caught only in the guard behind it.  Only
    lists that move because of a multiple of 2^32 bytes may leave room there, less than an area."""
    for T, M, k in ((1, 1024, 8), (1, 131072, 16), (40, 1024, 3), (300, 5800, 8), (2000, 8192, 16), (20000, 16384, 16), (131202, 32768, 4)):
        size = mr.debug_scratch_bytes(T, 512, 64, M, k)
        at, areas, places, step = mr.debug_chain_lists(T, 512, 64, M, k, scratch=1 << 40)
        end = at + areas * places * step
        assert end == (1 << 40) + size and size % 256 == 0
        for before in (0, 256, 16384, places * step, areas * places * step - 256):      # the multiple, so far in front of the end
            scratch = (9 << 32) + before - size
            at = mr.debug_chain_lists(T, 512, 64, M, k, scratch=scratch)[0]
            slack = scratch + size - (at + areas * places * step)
            assert 0 <= slack < places * step and (slack == 0 or before % (places * step))


def test_extension_module_of_another_torch_is_not_used(monkeypatch):
    """The module is compiled against torch's C++ headers: after an upgrade it is built again, and until then refused."""
    import torch
    mr_build.build_binding()
    assert mr_build.binding_is_current()
    monkeypatch.setattr(torch, "__version__", "0.0.1+other")
    assert not mr_build.binding_is_current()
    monkeypatch.setattr(mr, "_fast_module", None)
    with pytest.raises(ImportError, match="was not built for torch 0.0.1"):
        mr._fast()


def test_committed_counters_are_of_the_kernels_that_run():
    """Every entry of profiles/counters.json was captured on a kernel of the plan that serves its workload, and bench.py
    would not attach it otherwise."""
    import json

    import bench
    from paper_2609_36301_b200 import inputs
    counters = json.load(open(os.path.join(ROOT, "profiles", "counters.json")))
    assert counters
    for key, entry in counters.items():
        name, gate_mode = key.split("/mode")
        c = inputs.CONFIGS[name]
        plan = mr.more_route_plan_ex(c["T"], c["h"], c["r"], c["M"], c["k"], int(gate_mode))
        assert bench.counters_of(counters, name, int(gate_mode), plan) == entry, f"{key} was captured on {entry['kernel']}"
        assert os.path.exists(os.path.join(ROOT, re.search(r"profiles/\S+\.md", entry["source"]).group()))
        other = mr.more_route_plan_ex(2000, 64, 16, 64, 2)                 # too few experts for the chain, too few tokens for pairs
        assert bench.counters_of(counters, name, int(gate_mode), other) == {}


@pytest.mark.parametrize("name,kernel,other", [("c2_M16384/mode0", "sweep_kernel<8, 0, 0>", "sweep_kernel<8, 0>"),
                                               ("c3/mode1", "sweep_kernel<8, 1, 0>", "sweep_kernel<16, 1, 0>"),
                                               ("c3/mode0", "route_tcgen05_kernel<64, 8, 0, 0, 0>", "route_tcgen05_kernel<32, 8, 0, 0, 0>")])
def test_counters_of_another_instantiation_are_not_used(name, kernel, other):
    import bench
    from paper_2609_36301_b200 import inputs
    config, gate_mode = name.split("/mode")
    c = inputs.CONFIGS[config]
    plan = mr.more_route_plan_ex(c["T"], c["h"], c["r"], c["M"], c["k"], int(gate_mode))
    for k in (kernel, other):
        entry = {"kernel": k, "dram_bytes": 1}
        assert bench.counters_of({name: entry}, config, int(gate_mode), plan) == (entry if k == kernel else {})
