"""The leaf batches of closest hits and sun rays (one option sets both): the
option's default value gives the default pair, every value a batch of 1 to 32
lanes.  Checked at compile time on the library's own header."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_1912_04000_gb300", "csrc")

SOURCE = """
#include "rt_internal.h"
using namespace srt;
static_assert(kDefaultLeafBatch == 16 && shadow_leaf_batch(kDefaultLeafBatch) == 26);
constexpr bool in_range() {
  for (int l = 1; l <= 32; ++l)
    if (shadow_leaf_batch(l) < 1 || shadow_leaf_batch(l) > 32) return false;
  return true;
}
static_assert(in_range());
"""


def test_leaf_batch_pairs(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    cxx = shutil.which("g++") or shutil.which("c++")
    include = os.path.join(os.path.dirname(os.path.dirname(nvcc)), "include")
    if cxx is None or not os.path.exists(os.path.join(include, "cuda_runtime.h")):
        pytest.skip("no C++ compiler or no CUDA headers")
    src = tmp_path / "leaf.cpp"
    src.write_text(SOURCE)
    subprocess.run([cxx, "-std=c++17", "-fsyntax-only", "-I", CSRC, "-I", include, str(src)], check=True)
