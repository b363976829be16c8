"""The rule that lets a kernel access a host array (one page-locked allocation holds all of it, under its own address), compiled for the
host: an array that reaches beyond its registration, on either side, is left to the copy engine."""
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2609_22441_b200", "csrc")
START, SIZE, TOP = 0x7000_0000_0000, 1 << 20, (1 << 64) - 1


@pytest.fixture(scope="module")
def rule(tmp_path_factory):
    d = tmp_path_factory.mktemp("rule")
    src, exe = d / "rule.cpp", d / "rule"
    src.write_text('#include "ccr_hostrange.h"\n#include <cstdlib>\n'
                   "int main(int, char** v) { auto u = [&](int i) { return strtoull(v[i], nullptr, 0); };\n"
                   "return ccr::pinned_range_holds(u(1), u(2), u(3), u(4), u(5), u(6), u(7)) ? 10 : 20; }\n")
    subprocess.run(["g++", "-std=c++17", "-Wall", "-Werror", "-I", CSRC, "-o", str(exe), str(src)], check=True)
    return lambda *a: {10: True, 20: False}[subprocess.run([str(exe)] + [str(int(x)) for x in a]).returncode]


@pytest.mark.parametrize("host,managed,device,start,size,p,n,want", [
    (1, 0, START, START, SIZE, START, SIZE, True),                         # all of it
    (1, 0, START + 16, START, SIZE, START + 16, SIZE - 16, True),          # up to its end
    (1, 0, START + 16, START, SIZE, START + 16, SIZE - 15, False),         # one byte beyond
    (1, 0, START, START, SIZE, START, SIZE + 1, False),
    (1, 0, START + SIZE - 1, START, SIZE, START + SIZE - 1, 1, True),
    (1, 0, START - 16, START, SIZE, START - 16, 32, False),                # begins in front of the registration
    (1, 0, START, START, SIZE, START, TOP, False),                         # no wrap-around
    (1, 0, TOP - 15, TOP - 15, 16, TOP - 15, 17, False),
    (0, 0, START, START, SIZE, START, 64, False),                          # not page-locked
    (1, 1, START, START, SIZE, START, 64, False),                          # managed
    (1, 0, START + 4096, START, SIZE, START, 64, False),                   # another address on the device
    (1, 0, START, 0, 0, START, 64, False),                                 # no range reported
])
def test_the_rule(rule, host, managed, device, start, size, p, n, want):
    assert rule(host, managed, device, start, size, p, n) is want
