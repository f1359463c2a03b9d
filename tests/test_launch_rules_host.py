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
