"""The rounds in which a stream's markers are counted cover it exactly and end, also for the longest streams that are allowed: the
index arithmetic of the kernel, run on the CPU."""
import os
import subprocess

from paper_2609_12299_b200 import build

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SOURCE = """#include <stdio.h>
#include "argus_pair_common.cuh"
int main() {
  const u32 most = 0xffffffffu, sizes[] = {0, 1, kRecountStep - 1, kRecountStep, kRecountStep + 1, 1u << 31, most - kRecountStep, most - kRecountStep + 1,
                                           most - kRecountStep + 2, most - 1, most};
  for (u32 n : sizes) {
    const u32 rounds = argus_recount_rounds(n);
    u64 next = 0;  // the marker that has to come next
    for (u32 round = 0; round < rounds; ++round) {
      const u32 have = argus_recount_markers(n, round);
      if (have == 0 || have > kRecountStep || (u64)round * kRecountStep != next || next + have > n) { printf("%u: round %u\\n", n, round); return 1; }
      next += have;
    }
    if (next != n || rounds > (1u << 17)) { printf("%u: %llu in %u rounds\\n", n, next, rounds); return 1; }
  }
  return 0;
}
"""


def test_rounds_cover_a_stream(tmp_path):
    src, exe = tmp_path / "rounds.cu", tmp_path / "rounds"
    src.write_text(SOURCE)
    subprocess.check_call([build.NVCC, *build.ARCH, "-std=c++17", "-I", os.path.join(ROOT, "include"), "-I", os.path.join(ROOT, "paper_2609_12299_b200", "csrc"),
                           "-o", str(exe), str(src)])
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout
