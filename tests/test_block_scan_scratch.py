"""The block-wide scan writes 33 elements of its scratch whatever the block's size, so scratch of any other size has to be refused by
the compiler: an array sized by the block's warps is written past its end by the scan's first warp."""
import os
import subprocess

import pytest

from paper_2609_12299_b200 import build

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SOURCE = """#include "argus_common.cuh"
__global__ void k(u32* out) {
  __shared__ u64 scratch[%s];
  u64 total;
  out[threadIdx.x] = (u32)argus_block_exclusive_scan<u64>(threadIdx.x, %s, &total);
}
"""


@pytest.mark.parametrize("size,arg,fits", [("33", "scratch", True), ("9", "scratch", False), ("32", "scratch", False), ("2][9", "scratch[0]", False)])
def test_scratch_size_is_checked(tmp_path, size, arg, fits):
    src = tmp_path / "k.cu"
    src.write_text(SOURCE % (size, arg))
    r = subprocess.run([build.NVCC, *build.ARCH, "-std=c++17", "-I", os.path.join(ROOT, "include"), "-I", os.path.join(ROOT, "paper_2609_12299_b200", "csrc"),
                        "-c", "-o", os.devnull, str(src)], capture_output=True, text=True)
    assert (r.returncode == 0) == fits, r.stderr
    assert fits or "static assertion failed" in r.stderr
