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
