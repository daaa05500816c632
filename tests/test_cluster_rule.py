"""The blocks of a batch's coarse-level clusters (csrc/cluster_rule.h), on the CPU: a size that the device does
not run, or whose blocks do not hold the levels, gives way to another one."""
import ctypes as ct
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2603_21869_gb300", "csrc")


@pytest.fixture(scope="module")
def blocks(tmp_path_factory):
    d = tmp_path_factory.mktemp("rule")
    (d / "rule.cpp").write_text('#include "cluster_rule.h"\n'
                                'extern "C" int rule(int preferred, int most, int usable) {\n'
                                '    return cluster_blocks(preferred, most, [&](int S) { return (usable & S) != 0; });\n}\n')
    subprocess.run(["g++", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, str(d / "rule.cpp"), "-o", str(d / "rule.so")],
                   check=True)
    return ct.CDLL(str(d / "rule.so")).rule


@pytest.mark.parametrize("preferred,usable,want", [
    (16, 31, 16), (8, 31, 8), (1, 31, 1),     # the preferred size
    (16, 15, 8), (8, 7, 4), (16, 1, 1),       # the device holds smaller clusters only
    (2, 28, 4), (1, 16, 16),                  # the levels need more blocks
    (8, 6, 4), (8, 18, 16),                   # larger sizes before smaller ones
    (16, 0, 0),
])
def test_cluster_blocks(blocks, preferred, usable, want):
    assert blocks(preferred, 16, usable) == want
