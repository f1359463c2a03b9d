"""The fixed-point primitives of the kernels (csrc/ivb_fixed.cuh), compiled for
the CPU: reciprocal, quotient and square root equal the directed IEEE results on
every operand (exact results, powers of two and their neighbours among them);
exp and log enclose the binary128 value within three steps per end, at the ends
of the table intervals too, and log hands over next to 1."""
from __future__ import annotations

import os
import platform
import shutil
import subprocess

import pytest

SRC = os.path.join(os.path.dirname(os.path.abspath(__file__)), "mirror", "fixed_check.cpp")


@pytest.fixture(scope="module")
def counts(tmp_path_factory):
    if shutil.which("g++") is None:
        pytest.skip("needs g++")
    exe = str(tmp_path_factory.mktemp("fixed") / "fixed_check")
    cmd = ["g++", "-O2", "-std=gnu++17", "-frounding-math", "-ffp-contract=off", "-Wno-unknown-pragmas", SRC, "-o", exe]
    if platform.machine() in ("x86_64", "AMD64", "i686"):
        cmd.append("-lquadmath")
    subprocess.run(cmd, check=True)
    out = subprocess.run([exe, "1000000"], check=True, capture_output=True, text=True).stdout
    return {k: int(v) for k, v in (kv.split("=") for kv in out.split())}


@pytest.mark.parametrize("name", ["rcp", "div", "sqrt", "exp", "log"])
def test_fixed_point_primitive(counts, name):
    assert counts[name] == 0


def test_the_edge_cases_were_met(counts):
    assert counts["exact"] > 10_000 and counts["small"] > 10_000
