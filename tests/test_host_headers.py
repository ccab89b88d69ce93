"""The parts of the CUDA path's headers that compile for the host too, built with
g++ and checked without a GPU."""

import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2109_01329_gb300", "csrc")


def _build(path, code, *flags):
    """Compiles C++ source text against the headers; the path of what it makes."""
    src, out = str(path / "t.cpp"), str(path / "t.bin")
    with open(src, "w") as f:
        f.write(code)
    subprocess.run(["g++", "-std=c++17", "-O2", "-ffp-contract=off", "-I", CSRC, src, "-o", out, *flags],
                   check=True, timeout=300)
    return out


def test_jump_table_is_aligned_for_16_byte_loads(tmp_path):
    """The kernels read the table of jump matrices in 16-byte pieces: the type, not
    the order in which a linker lays globals, has to place every row and second
    matrix on such a boundary."""
    exe = _build(tmp_path, """
#include <cstdio>
#include "mrg_tables.h"
int main() { std::printf("%zu %zu", alignof(grng::mrg::DigitTable), sizeof(grng::mrg::DigitTable::row[0])); }
""")
    align, row = map(int, subprocess.run([exe], check=True, capture_output=True, text=True).stdout.split())
    assert align % 16 == 0 and row % 16 == 0
