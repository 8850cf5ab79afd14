"""The operand rows that a thread of the shared-memory tiles (block_kernel) loads:
as many as it computes, for every tile shape and residues per entry.  The
function is compiled for the host with array-bounds checks (no GPU needed) and
must leave what lies behind its array alone and read only staged entries."""
import os
import shutil
import subprocess

import pytest

from paper_1805_00475_gb300 import build as tnc_build

SRC = r"""
#include <cstdio>
#include <cstring>
#include "steps.cuh"
using namespace tnc_dev;
template <int N, int RG>
int check(uint32_t staged) {  // N of `staged` entries, evenly apart, from each thread's first one on
  static uint4 entries[64];   // 64 rows of at most 16 bytes, aligned as entries are
  uint32_t* e = reinterpret_cast<uint32_t*>(entries);
  for (uint32_t i = 0; i < 64 * 4; i++) e[i] = i < staged * RG ? i + 1 : 0xBADu;
  int bad = 0;
  for (uint32_t first = 0; first < staged / N; first++) {
    struct {
      uint32_t v[N][RG], behind[16];
    } x;
    std::memset(&x, 0xA5, sizeof(x));
    load_rows(e + first * RG, staged / N, x.v);
    for (int i = 0; i < N; i++)
      for (int r = 0; r < RG; r++) bad += x.v[i][r] != (first + i * (staged / N)) * RG + r + 1;
    for (uint32_t w : x.behind) bad += w != 0xA5A5A5A5u;
  }
  return bad;
}
template <int SHAPE, int RG>
int shape() {
  using B = Blk<SHAPE>;
  return check<1 << B::RA, RG>(1u << B::LA) + check<1 << B::RB, RG>(1u << B::LB);
}
template <int SHAPE>
int residues() { return shape<SHAPE, 1>() + shape<SHAPE, 2>() + shape<SHAPE, 4>(); }
int main() {
  const int bad[3] = {residues<0>(), residues<1>(), residues<2>()};
  std::printf("%d %d %d\n", bad[0], bad[1], bad[2]);
  return bad[0] + bad[1] + bad[2] != 0;
}
"""


def test_block_kernel_loads_the_rows_it_computes(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    csrc = os.path.join(os.path.dirname(tnc_build.__file__), "csrc")
    (tmp_path / "rows.cu").write_text(SRC)
    exe = str(tmp_path / "rows")
    r = subprocess.run([nvcc, "-std=c++17", "-O1", *tnc_build.ARCH, "-I", csrc, "-I", os.path.join(csrc, "..", "..", "include"),
                        "-Xcompiler", "-fsanitize=bounds",
                        "-Xcompiler", "-fno-sanitize-recover=bounds", str(tmp_path / "rows.cu"), "-o", exe],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    r = subprocess.run([exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout + r.stderr
