"""Rules and tables on the host that no entry point shows, through a small
program linked against the library (no GPU needed)."""
import os
import subprocess

import pytest

from paper_1412_7789_gb300 import build


def run_cpp(tmp_path, source: str, *args: str) -> str:
    """Compile a program against the internal header and the library; its output."""
    lib = build.build()
    src, exe = tmp_path / "prog.cpp", tmp_path / "prog"
    src.write_text(source)
    subprocess.run([build._nvcc(), "-O1", "-std=c++17", "-I", build.INCLUDE, "-I", build.CSRC, str(src), "-o", str(exe),
                    lib, "-Xlinker", "-rpath=" + os.path.dirname(lib)], check=True)
    return subprocess.run([str(exe), *args], capture_output=True, text=True, check=True).stdout


def test_full_counts_fit_32_bits(tmp_path):
    """Full output goes tile by tile (2,048 results) while 2,048 results with
    the set's longest chain fit 32 bits, by half tiles while 1,024 do."""
    out = run_cpp(tmp_path, r'''
#include <cstdio>
#include "pfac_internal.h"
int main() {
    for (unsigned c : {1u, (1u << 21) - 1, 1u << 21, (1u << 22) - 1, 1u << 22, 0xFFFFFFFFu})
        std::printf("%d%d ", pfac::full_fits(c, pfac::kStreamTile), pfac::full_fits(c, pfac::kDenseStride));
}''')
    assert out.split() == ["11", "11", "01", "01", "00", "00"]
