"""The rules for host buffers that a kernel stores into directly (csrc/host_buffer.h), on the CPU."""
import ctypes as ct
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2603_21869_gb300", "csrc")


def rule(tmp_path, name, arguments):
    """One of the header's functions, compiled alone: arguments as C declarations."""
    src, lib = tmp_path / "rule.cpp", tmp_path / "rule.so"
    names = ", ".join(a.split()[-1] for a in arguments)
    src.write_text('#include "host_buffer.h"\n'
                   f'extern "C" int rule({", ".join(arguments)}) {{ return {name}({names}); }}\n')
    subprocess.run(["g++", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, str(src), "-o", str(lib)], check=True)
    f = ct.CDLL(str(lib)).rule
    f.argtypes = [ct.c_size_t] * len(arguments)
    return f


def test_only_aligned_doubles_are_stored_directly(tmp_path):
    aligned = rule(tmp_path, "doubles_aligned", ["uintptr_t at"])
    assert [bool(aligned(0x7f0000001000 + o)) for o in range(9)] == [True] + 7 * [False] + [True]


def test_only_buffers_within_one_allocation_are_stored_directly(tmp_path):
    holds = rule(tmp_path, "allocation_holds", ["uintptr_t start", "size_t size", "uintptr_t at", "size_t bytes"])
    start, size = 0x7f0000001000, 0x10000
    assert holds(start, size, start, size) and holds(start, size, start + 8, size - 8)
    assert not holds(start, size, start, size + 8)               # past the end: the next range is another one's
    assert not holds(start, size, start + 8, size)
    assert not holds(start, size, start - 8, 16)
    assert not holds(start, size, start + 4 * size, 8)           # a gap after the range
    assert not holds(start, size, start + 8, 2**64 - 8)          # no wrapping round
