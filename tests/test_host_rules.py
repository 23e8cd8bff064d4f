"""The rules of csrc/lbm_host_rules.h, compiled by the host compiler (no GPU)."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1412_7228_gb300", "csrc")


def ask(tmp_path, body):
    """The numbers that a program with this body of main() prints."""
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    src = tmp_path / "ask.cpp"
    src.write_text('#include <cstdio>\n#include <initializer_list>\n#include "lbm_host_rules.h"\nint main() {\n%s\nreturn 0; }\n' % body)
    exe = tmp_path / "ask"
    r = subprocess.run([cxx, "-std=c++17", "-Wall", "-Werror", "-I", CSRC, str(src), "-o", str(exe)], capture_output=True,
                       text=True)
    assert r.returncode == 0, r.stderr
    out = subprocess.run([str(exe)], capture_output=True, text=True, check=True).stdout
    return [int(v) for v in out.split()]


def test_arrays_off_their_values_alignment_are_left_to_the_copies(tmp_path):
    got = ask(tmp_path, """
        for (size_t size : {4, 8})
            for (uintptr_t off = 0; off < 17; ++off) printf("%d ", lbm::in_place({0x7f0000001000 + off, 100 * size}, size));
    """)
    assert got == [int(off % size == 0) for size in (4, 8) for off in range(17)]
