"""The lines of a list range that a warp prefetches (CPU): the library's own
loop (csrc/ctb_internal.cuh) on ranges at the start, in the middle and at the
very end of a list buffer of 2^32 entries, where the end of the last list is
0 modulo 2^32 and the next line's word past it wraps."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)

# the callback leaves a loop that does not end by an exception
PROGRAM = r"""
#include <cstdio>
#include <cstdlib>
#include "ctb_internal.cuh"
int main(int argc, char** argv) {
  for (int i = 1; i + 1 < argc; i += 2) {
    const uint32_t off = (uint32_t)strtoull(argv[i], nullptr, 10), end = (uint32_t)strtoull(argv[i + 1], nullptr, 10);
    unsigned long long lines = 0, sum = 0;
    try {
      for (uint32_t lane = 0; lane < 32; ++lane)
        ctb::each_list_line(off, end, lane, [&](uint32_t w) {
          if (++lines > 1000000ull) throw 1;
          sum += w;
        });
    } catch (int) {
      sum = 0;
    }
    printf("%llu %llu\n", lines, sum);
  }
  return 0;
}
"""


def test_list_lines_end_at_the_top_of_the_buffer(tmp_path):
    nvcc = shutil.which("nvcc") or ("/usr/local/cuda/bin/nvcc" if os.path.exists("/usr/local/cuda/bin/nvcc") else None)
    if nvcc is None:
        pytest.skip("nvcc not available")
    src = tmp_path / "lines.cu"
    src.write_text(PROGRAM)
    exe = tmp_path / "lines"
    r = subprocess.run([nvcc, "-std=c++17", "--expt-relaxed-constexpr", "-I",
                        os.path.join(ROOT, "paper_2604_08855_gb300", "csrc"), str(src), "-o", str(exe)],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    top = 1 << 32
    ranges = [(0, 0), (0, 1), (5, 1029), (7, 1032), (123456, 123456 + 99999), (top - 1, top), (top - 33, top),
              (top - 1024, top), (top - 1025, top), (top - 5000, top - 1), (top - 1000, top - 999),
              (top - 700, top - 10), (top - 5000, top - 1100), (top - 40, top - 40)]
    args = [str(v % top) for r in ranges for v in r]
    out = subprocess.run([str(exe), *args], capture_output=True, text=True, timeout=60).stdout.split()
    got = [(int(out[2 * i]), int(out[2 * i + 1])) for i in range(len(ranges))]
    want = []
    for off, end in ranges:
        words = range(off, end, 32)
        want.append((len(words), sum(words)))
    assert got == want
