"""Workspace layouts, on the CPU: a per-vertex run that is short of memory takes
a lean layout, which is no larger than that of a run without per-vertex counts
(the size that per-vertex runs had before they kept bitmaps and streams)."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1503_00576_gb300", "csrc")
CUDA = "/usr/local/cuda/include"

PROGRAM = """
#include <algorithm>
#include <cstdio>
#include <tc_common.cuh>
using namespace tc;
int main() {
  const long long pairs[] = {1, 8191, 131072, 700000, 16777216, 20971520, 20971521, 33554431,
                             33554432, 180000000, 2147482000};
  const int vertices[] = {1, 1000, 16384, 131071, 131072, 1 << 20, (1 << 24) + 1};
  for (long long m : pairs)
    for (int n : vertices) {
      const Layout t = make_layout(m, n, true), v = make_layout(m, n, true, kHubSize, false, true),
                   l = make_layout(m, n, true, kHubSize, false, true, true);
      std::printf("%lld %d %zu %zu %zu %d %d\\n", m, n, t.total, v.total, l.total,
                  (int)l.has_bits, (int)l.has_desc);
    }
}
"""


@pytest.mark.skipif(shutil.which("g++") is None or not os.path.isdir(CUDA),
                    reason="needs g++ and the CUDA headers")
def test_lean_layout_is_no_larger_than_without_counts(tmp_path):
    src = tmp_path / "layout.cpp"
    src.write_text(PROGRAM)
    exe = str(tmp_path / "layout")
    subprocess.run(["g++", "-std=c++17", "-I", CSRC, "-I", CUDA, str(src), "-o", exe], check=True)
    rows = [[int(x) for x in line.split()]
            for line in subprocess.run([exe], check=True, capture_output=True,
                                       text=True).stdout.splitlines()]
    assert len(rows) == 77
    for m, n, total_only, per_vertex, lean, bits, desc in rows:
        assert lean == total_only <= per_vertex, (m, n)
        assert bits == 0 and desc == 0
        counting = m <= 20 << 20 and (m <= 1 << 18 or m <= 768 * n)
        if n <= m // 64 and (counting or m >= 1 << 25):
            assert per_vertex > lean, (m, n)
