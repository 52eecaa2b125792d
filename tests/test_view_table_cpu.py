"""The host's range check of matrix views whose inner columns lie at offsets
from a table: the largest of them counts, before and after a transposition.
Compiles a small host program against the library's header (no GPU)."""

import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
NVCC = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"

PROGRAM = r"""
#include "common.cuh"
using namespace cvs;
// does the check accept a rows x cols view?
static bool ok(const View& v, int64_t rows, int64_t cols) {
  try {
    check_view(v, rows, cols, 1, "v");
  } catch (const Error&) {
    return false;
  }
  return true;
}
int main() {
  // [c < 4][k < o][b < v][l < o] over the pairs k < l, rows b
  const int64_t o = 5, v = 7, vo = v * o, ovo = o * vo;
  const int pairs = o * (o - 1) / 2;
  static const int tab[1] = {0};  // the host looks at its largest entry only
  const int64_t last = (o - 2) * vo + o - 1;
  const int64_t need = 3 * ovo + last + (v - 1) * o + 1;
  int bad = 0;
  for (int64_t ext = need - 2; ext <= need + 2; ++ext) {
    View t = cols_table(view(nullptr, o, 0, ext), ovo, tab, last, pairs);
    bad += ok(t, v, 4 * pairs) != (ext >= need);
    bad += ok(trans(t), 4 * pairs, v) != (ext >= need);
    bad += ok(trans(trans(t)), v, 4 * pairs) != (ext >= need);
  }
  // whole inner columns only are read of a part of the last block
  View t = cols_table(view(nullptr, o, 0, need), ovo, tab, last, pairs);
  bad += !ok(t, v, 3 * pairs + 1);
  bad += ok(t, v, 4 * pairs + 1);
  // without a table as before
  bad += !ok(cols2(view(nullptr, o, 0, 3 * ovo + 35), ovo, 1, pairs), 1, 4 * pairs);
  return bad;
}
"""


@pytest.mark.skipif(not os.path.exists(NVCC), reason="needs nvcc")
def test_table_offsets_are_in_range(tmp_path):
    src = tmp_path / "view.cu"
    src.write_text(PROGRAM)
    exe = str(tmp_path / "view")
    inc = os.path.join(ROOT, "paper_2604_27451_gb300", "csrc")
    subprocess.run([NVCC, "-std=c++17", "-I" + inc, "-I" + os.path.join(ROOT, "include"),
                    "-gencode", "arch=compute_103a,code=sm_103a", "-o", exe, str(src)], check=True)
    assert subprocess.run([exe]).returncode == 0
