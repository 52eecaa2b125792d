"""How many matrices the rotation into natural spinors takes at a time: what fits
the scratch beside the packed spinors, and one where these alone do not fit (an
unsigned difference would wrap).  Compiles a small host program against the
library's header (no GPU)."""

import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
NVCC = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"

PROGRAM = r"""
#include "common.cuh"
using namespace cvs;
int main() {
  const size_t G = (size_t)1 << 30;
  int bad = 0;
  bad += block_within(1000, G / 8, G / 1000, G / 2) != 375;  // (1/2 - 1/8) 1000
  bad += block_within(7, G / 8, G / 1000, G / 2) != 7;
  bad += block_within(7, G, G, 2 * G) != 1;
  bad += block_within(7, G, G, 2 * G - 1) != 1;  // not one fits
  bad += block_within(7, G, G, G) != 1;
  bad += block_within(7, G + 1, G, G) != 1;
  bad += block_within(1 << 20, 2 * G, 1, G) != 1;
  bad += block_within(1, 0, G, 8 * G) != 1;
  return bad;
}
"""


@pytest.mark.skipif(not os.path.exists(NVCC), reason="needs nvcc")
def test_block_within(tmp_path):
    src = tmp_path / "block.cu"
    src.write_text(PROGRAM)
    exe = str(tmp_path / "block")
    subprocess.run([NVCC, "-std=c++17", "-I" + os.path.join(ROOT, "paper_2604_27451_gb300", "csrc"),
                    "-I" + os.path.join(ROOT, "include"), "-gencode",
                    "arch=compute_103a,code=sm_103a", "-o", exe, str(src)], check=True)
    assert subprocess.run([exe]).returncode == 0
