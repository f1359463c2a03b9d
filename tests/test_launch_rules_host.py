"""Rules on the shape of the bounding launches (csrc/ivb_launch.h), compiled for
the CPU as they are."""
from __future__ import annotations

import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2507_20769_gb300", "csrc")


@pytest.fixture(scope="module")
def rows(tmp_path_factory):
    """run C++ statements against the header; each printed line as a list of integers"""
    if shutil.which("g++") is None:
        pytest.skip("needs g++")
    where = tmp_path_factory.mktemp("launch")

    def run(body: str):
        src, exe = str(where / "rules.cpp"), str(where / "rules")
        with open(src, "w") as fh:
            fh.write('#include <cstdio>\n#include <initializer_list>\n#include "ivb_launch.h"\nusing namespace ivb;\nint main() {' + body + "}\n")
        subprocess.run(["g++", "-std=c++17", "-Wall", "-Werror", "-I", CSRC, src, "-o", exe], check=True)
        out = subprocess.run([exe], check=True, capture_output=True, text=True).stdout
        return [[int(x) for x in line.split()] for line in out.splitlines()]
    return run


def test_groups_of_a_block_are_whole_warps(rows):
    """threads per subdomain: what was asked for where that leaves whole warps, else 1"""
    got = rows('for (int b = 32; b <= 1024; b += 32) for (int t : {1, 2, 4}) '
               'std::printf("%d %d %d\\n", b, t, block_tpsub(b, t));')
    assert len(got) == 96
    for block, wanted, t in got:
        assert block % t == 0 and (block // t) % 32 == 0, (block, wanted, t)
        assert t == (wanted if block % (32 * wanted) == 0 else 1), (block, wanted, t)
    assert [96, 2, 1] in got and [192, 2, 2] in got and [192, 4, 1] in got


def test_blocks_of_a_range_all_get_work(rows):
    """as many blocks as there are warps of subdomains, of the resident ones"""
    counts = (1, 31, 32, 33, 64, 65, 19455, 19456, 19457, 50003, 1 << 24)
    got = rows("for (long long c : {%s}) std::printf(\"%%lld %%d\\n\", c, range_blocks(c, 608));"
               % ", ".join(f"{c}LL" for c in counts))
    assert got == [[c, min(608, -(-c // 32))] for c in counts]


def test_frames_when_memory_is_short(rows):
    """a failing allocation halves the blocks until one succeeds, and gives up after one block"""
    got = rows("for (int most : {0, 1, 2, 37, 303, 304, 607, 608, 5000}) { int calls = 0; "
               "const int b = blocks_that_fit(608, [&](int g) { ++calls; return g <= most; }); "
               'std::printf("%d %d %d\\n", most, b, calls); }')
    for most, blocks, calls in got:
        want = [b for b in (608, 304, 152, 76, 38, 19, 9, 4, 2, 1) if b <= most]
        assert blocks == (want[0] if want else 0)
        assert calls == 11 - max(1, len(want)), (most, calls)


def test_default_shapes_keep_their_frames_small(rows):
    """1024 threads per SM up to a sixteenth of the device's memory"""
    mib = 284_208
    got = rows("for (long long u : {1LL, 1680LL, 14000LL, 15000LL, 15500LL, 262000LL}) "
               'std::printf("%%lld %%d\\n", u, (int)wide_frames_fit((size_t)u * 8, 152, (size_t)%dLL << 20));' % mib)
    for units, wide in got:
        assert wide == (units * 8 * 1024 * 152 <= (mib << 20) // 16), units
    assert {w for _, w in got} == {0, 1}


def test_block_of_a_register_budget_fits_an_sm(rows):
    got = rows('for (int r = 64; r <= 255; ++r) std::printf("%d %d\\n", r, seg_block_max(r));')
    assert len(got) == 192
    for regs, block in got:
        per = -(-regs // 8) * 8
        assert block % 128 == 0 and 256 <= block <= 1024 and block * per <= 65536, (regs, block)
        assert block == 1024 or (block + 128) * per > 65536, (regs, block)


def test_register_budget_follows_a_fixed_shape(rows):
    """64 for the library's shapes; fixed ones get their threads' share of an SM, 64 to 128"""
    got = {tuple(r[:3]): r[3] for r in rows(
        'for (int s : {0, 100}) for (int b = 0; b <= 1024; b += 32) for (int k = 0; k <= 8; ++k) '
        'std::printf("%d %d %d %d\\n", s, b, k, seg_registers(s, b, k));')}
    for (seg_regs, block, per_sm), regs in got.items():
        if seg_regs:
            assert regs == seg_regs
        elif block == 0:
            assert regs == 64
        else:
            threads = block * (per_sm or max(1, 512 // block))
            assert regs % 8 == 0 and 64 <= regs <= 128
            assert regs == 64 or regs * threads <= 65536
            assert regs == 128 or (regs + 8) * threads > 65536
    # blocks up to 256 as before: two of 256, four of 128 at 128 registers
    assert all(got[0, b, 0] == 128 for b in range(32, 257, 32))
    assert got[0, 256, 2] == 128 and got[0, 256, 4] == 64 and got[0, 1024, 0] == 64 and got[0, 1024, 1] == 64


def test_segmented_kernel_is_built_for_the_block_asked_for(rows):
    got = rows('for (int b = 0; b <= 1024; b += 32) for (int k = 0; k <= 8; ++k) { const int r = seg_budget(0, b, k); '
               'std::printf("%d %d %d %d %d\\n", b, k, r, seg_block_max(r), seg_registers(0, b, k)); }')
    for block, per_sm, regs, most, wanted in got:
        assert block <= most and 64 <= regs <= wanted, (block, per_sm)
        assert regs == wanted or -(-block // 128) * 128 * (regs + 8) > 65536, (block, per_sm)


@pytest.mark.parametrize("opts,big_tape,most", [
    (dict(specialize=0), True, 512), (dict(specialize=1), True, 256), (dict(specialize=2), False, 256),
    (dict(specialize=3), True, 1024), (dict(specialize=3), False, 1024), (dict(specialize=-1), True, 1024),
    (dict(specialize=-1), False, 512), (dict(specialize=-1, grad_mode="forward"), True, 512),
    (dict(specialize=3, seg_regs=128), True, 512), (dict(specialize=3, seg_regs=100), True, 512),
    (dict(specialize=3, seg_regs=255), True, 256)])
def test_largest_block_that_options_can_ask_for(opts, big_tape, most):
    """every shape that the autotuner can report is accepted, and nothing a kernel is not built for
    (invalid options are refused before the device is touched: no GPU needed)"""
    from paper_2507_20769_gb300 import build as B
    from paper_2507_20769_gb300 import workloads as W
    B.build()
    from paper_2507_20769_gb300 import ivb
    t = W.random_problem(2, 40 if big_tape else 6, 2 if big_tape else 0, W.OPS_RATIONAL, [[-2, 2]] * 2, 7, "blocks")

    def refused(block):
        try:
            ivb.Problem(t, block_threads=block, **opts).destroy()
        except ivb.IvbError as e:
            return e.status == ivb.IVB_EINVAL
        return False
    assert not refused(most) and not refused(32)
    assert refused(most + 32) and refused(most - 1) and refused(-32)


def test_emulated_sums_of_large_tapes_are_called_out_of_line(rows):
    got = rows('for (int o = -1; o <= 2; ++o) for (int e = 0; e < 16; ++e) for (long long k : {1LL, 1024LL, 1025LL, 99999LL}) '
               'std::printf("%d %d %lld %d\\n", o, e, k, seg_outline_for(o, e, k));')
    assert len(got) == 256
    for option, emulate, ops, out in got:
        assert out == (option if option >= 0 else 1 if emulate >= 4 and ops > 1024 else 2)
