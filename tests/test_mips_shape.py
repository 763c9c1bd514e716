"""Shared memory of the batched queries' draw blocks (host arithmetic of
csrc/mips_shape.h): what the draw kernels opt in to holds every accepted
shape, those above the 48 KB default included, and fits an SM."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1506_03872_gb300", "csrc")

PROGRAM = r"""
#include <cstdio>
#include <cstdlib>
#include "mips_shape.h"
int main(int argc, char** argv) {
  std::printf("%zu\n", mad::kDrawSmemMax);
  for (int a = 1; a + 2 < argc; a += 3)
    std::printf("%zu\n", mad::draw_smem_bytes(std::atoi(argv[a]), (uint32_t)std::atoi(argv[a + 1]),
                                              std::atoi(argv[a + 2])));
}
"""


def test_draw_blocks_fit_what_the_kernels_ask_for(tmp_path):
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("no C++ compiler")
    src, exe = tmp_path / "shape.cpp", tmp_path / "shape"
    src.write_text(PROGRAM)
    subprocess.run([cxx, "-std=c++17", "-I", CSRC, "-o", str(exe), str(src)], check=True)
    shapes = [(chunk, parts, d) for chunk in (256, 512, 1024, 2048)
              for parts in (1, 1015, 1016, 2047, 2048) for d in (1, 765, 766, 1024)]
    out = subprocess.run([str(exe), *[str(v) for s in shapes for v in s]], check=True,
                         capture_output=True, text=True).stdout.split()
    most, sizes = int(out[0]), dict(zip(shapes, map(int, out[1:])))
    # records 8, part and rank 4, source 2 bytes a diamond; counts, two rows and pairs
    for (chunk, parts, d), b in sizes.items():
        assert b == 14 * chunk + 4 * (parts + 1) + 16 * d
        assert b <= most
    assert sizes[2048, 1015, 1024] + 32 <= 48 * 1024 < sizes[2048, 1016, 1024] + 32
    assert most <= 227 * 1024 - 1024
    # Both kernels opt in to it, and nothing follows a draw that did not launch.
    text = open(os.path.join(CSRC, "mips.cu")).read()
    for kernel in ("k_mips_draw<true>", "k_mips_draw<false>"):
        at = text.index(f"cudaFuncSetAttribute({kernel}")
        assert "kDrawSmemMax" in text[at:at + 200]
    run = text[text.index("mad_status mad_mips_run"):]
    assert "cudaGetLastError" in run[run.index("k_mips_draw<false><<<"):run.index("k_mips_parts<<<")]
