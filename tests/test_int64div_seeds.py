"""The integer-pipe division and root with seeds at both ends of their bound,
1 - 2^-22 and 1 + 2^-22 times the true value in every operand class: a high
seed is the side that the estimates must stay below."""
import os
import subprocess

import pytest

from test_int64div import ROOT, SRC


@pytest.fixture(scope="module")
def prog(tmp_path_factory):
    d = tmp_path_factory.mktemp("int64div_seeds")
    a, b = SRC.index("    if (i % 500 == 0) off ="), SRC.index("    uint64_t a = rnd(), b = rnd();")
    src = SRC[:a] + "    off = (rnd() & 1 ? 1.0 : -1.0) * 0x1p-22;\n" + SRC[b:]
    # divisors whose bits beyond the seed's 23 are all ones
    ones = "    if (i % 4 == 1) mb |= (1ull << 29) - 1;\n"
    c = src.index("    if (mode == 1)")
    (d / "t.cpp").write_text(src[:c] + ones + src[c:])
    exe = str(d / "t")
    subprocess.run(["g++", "-O2", "-std=c++17", "-I" + os.path.join(ROOT, "paper_1112_1710_gb300", "csrc"), str(d / "t.cpp"),
                    "-o", exe], check=True)
    return exe


@pytest.mark.parametrize("mode", range(7))
def test_seeds_at_both_ends(prog, mode):
    r = subprocess.run([prog, str(mode)], capture_output=True, text=True)
    assert r.returncode == 0 and r.stdout.strip() == "0", r.stdout
