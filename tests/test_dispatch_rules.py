"""Rules by which launches choose their kernels (csrc/wash_internal.h), compiled for the host and evaluated over their ranges."""
import ctypes
import os
import subprocess

import pytest

from paper_2405_17517_b200 import build

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def rules(tmp_path_factory):
    lib = str(tmp_path_factory.mktemp("rules") / "rules.so")
    cuda = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(build._nvcc()))), "include")
    subprocess.run(["g++", "-std=c++17", "-O1", "-fPIC", "-shared", "-I", build.CSRC, "-I", cuda, os.path.join(HERE, "dispatch_rules.cpp"), "-o", lib], check=True)
    return ctypes.CDLL(lib)


@pytest.mark.parametrize("bytes_a,bytes_b", [(4, 0), (2, 0), (4, 4), (2, 4), (4, 2), (2, 2)])
@pytest.mark.parametrize("N", [17, 24, 32, 40, 48, 56, 60, 64])
def test_bulk_copies_only_where_they_can_be_reported_and_fit(rules, N, bytes_a, bytes_b):
    """A launch without a status word never takes copies whose wait can be given up; neither do odd ranges or padded images, whose
    bytes are no multiples of 16 or not contiguous.  Where they fit, a larger selection or a larger block never turns them off, and the
    stacks' order does not matter."""
    def bulk(has_status=1, pad=0, lo=0, hi=1 << 26, groups=32, share=0.5, a=bytes_a, b=bytes_b):
        return rules.rule_copies_in_bulk(has_status, pad, lo, hi, groups, N, a, b, ctypes.c_float(share))
    for share in (0.005, 0.1, 0.5, 1.0):
        assert not bulk(has_status=0, share=share) and not bulk(has_status=0, groups=64, share=share)
        assert not bulk(pad=4, share=share) and not bulk(lo=3, share=share) and not bulk(hi=999, share=share) and bulk(hi=1000, share=share)
        assert bulk(groups=32, share=share) <= bulk(groups=64, share=share)
        if bytes_b:
            assert bulk(share=share) == bulk(share=share, a=bytes_b, b=bytes_a)
    taken = [bulk(share=s) for s in (0.003, 0.01, 0.05, 0.1, 0.19, 0.21, 0.6, 1.0)]
    assert taken == sorted(taken) and taken[-1] == 1


@pytest.mark.parametrize("tile", [256, 512], ids=["two groups a lane", "four"])
def test_no_slot_is_reported_more_than_its_fields_hold(rules, tile):
    """The resident-warp kernel's packed report (8 bits of blocks, 26 of selected coordinates) on devices of 1 to 592 SMs, from one
    block an SM on, for rows up to the longest there are and everything selected; blocks take the tiles round-robin."""
    rules.rule_report_grid.argtypes = [ctypes.c_ulonglong, ctypes.c_ulonglong]
    slots = rules.rule_stat_slots()
    for n_tiles in (1, slots - 1, slots, slots + 1, 4736, 1 << 20, (1 << 33) // tile):
        for resident in [sms * blocks for sms in (1, 2, 7, 16, 37, 74, 148, 296, 592) for blocks in range(1, 33)]:
            grid = rules.rule_report_grid(n_tiles, resident)
            assert 1 <= grid <= n_tiles and grid >= min(resident, n_tiles)
            blocks = range(0, grid, slots)            # of the fullest slot: its first block takes every grid-th tile from 0 on
            assert len(blocks) < 256
            coordinates = sum((n_tiles - b + grid - 1) // grid for b in blocks) * tile
            assert coordinates < 1 << 26 and 16 * coordinates < 1 << 30


def test_half_lines_are_asked_for_alike_in_either_order_of_the_stacks(rules):
    """Both stacks of a launch take one form of load, so bf16 weights with fp32 momentum and fp32 weights with bf16 momentum
    get the same one; a single stack in [P][N], whose loads never gained, and rare values get the plain load."""
    def half(layout, N, share, a, b, by_warps=0):
        return rules.rule_fetch_half_lines(layout, N, ctypes.c_float(share), by_warps, a, b)
    shares = [10.0 ** (-4 + 0.05 * k) for k in range(81)]
    for layout in (0, 1):
        for N in range(2, 65):
            for by_warps in (0, 1):
                assert [half(layout, N, s, 2, 4, by_warps) for s in shares] == [half(layout, N, s, 4, 2, by_warps) for s in shares]
            assert not any(half(1, N, s, e, 0) for s in shares for e in (2, 4))
            assert not any(half(layout, N, s, a, b) for s in shares if s * N < 0.03 for a, b in ((4, 0), (2, 0), (4, 4), (2, 4)))
    assert half(0, 8, 0.005, 2, 4) and half(0, 5, 0.025, 4, 0)


def test_half_a_wave_only_where_it_does_not_lose_more_than_it_gains(rules):
    """0.4 of a wave's values and 16 tiles a warp (1184 resident blocks); with more than 32 models few values a block."""
    def half(N, by_load, n_wtiles, layout=0, stacks=1, expected=0.0):
        return rules.rule_half_wave_serves(layout, N, stacks, ctypes.c_double(expected), ctypes.c_double(by_load), 1184, n_wtiles)
    assert half(5, 374.0, 21_914, stacks=2, expected=11_220.0) and half(32, 0.0, 37_888, expected=1e6)
    assert not half(5, 474.0, 21_914) and not half(5, 1.0, 37_889)
    assert half(64, 200.0, 6_000, expected=937.0) and half(64, 10.0, 6_000, layout=1, expected=3_125.0)
    assert not half(48, 333.0, 4_069, expected=2_083.0) and not half(48, 21.0, 4_069, layout=1, expected=6_250.0) and not half(64, 200.0, 6_000, stacks=2, expected=937.0)


def test_which_populations_store_neighbouring_values_together(rules):
    """[P][N]: four models' values where the population is a multiple of four, two where it is even, up to 16 models, but not two
    models; the kernels' code paths, WASH_MODE_AUTO's table and the early flavour all go by this."""
    assert rules.rule_stored_together(1, 2) == 1
    for N in range(3, 65):
        want = 4 if N % 4 == 0 else 2 if N % 2 == 0 and N <= 16 else 1
        assert rules.rule_stored_together(1, N) == want and rules.rule_stored_together(0, N) == 1


def test_tensors_are_served_densely_late_or_never_in_even_populations(rules):
    """A threshold of up to 2^32 (half of it is compared) is reached (by everything selected at the latest) or none is: populations of a multiple of four from 12
    models on in one stack, from 8 on in two."""
    rules.rule_dense_threshold.restype = ctypes.c_uint32
    for N in range(2, 17, 2):
        for two_stacks in (0, 1):
            for all_f32 in (0, 1):
                at = rules.rule_dense_threshold(N, two_stacks, all_f32) / 2.0 ** 31
                never = N % 4 == 0 and (N >= 12 or (two_stacks and (N >= 8 or all_f32)))
                assert at > 1.0 if never else 0.5 < at < 0.9
