"""The rule that keeps the tensor-core CTAs of one SM within its 512 columns of tensor memory
(csrc/tmem_share.h), over every set of CTAs that fit in the SM's shared memory together."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2606_05893_gb300", "csrc")
SOURCE = r"""
#include <cstdio>
#include "tmem_share.h"
using namespace unet;
static int most = 0;
static void add(uint32_t top, size_t bytes, int cols) {  // CTAs of at most `top` columns beside the ones counted
  if (cols > most) most = cols;
  for (uint32_t c = 32; c <= top; c *= 2) {
    const size_t b = smem_floor(0, c) + kSmemReserved;
    if (bytes + b <= kSmemPerSM) add(c, bytes + b, cols + (int)c);
  }
}
int main() {
  add(512, 0, 0);
  for (uint32_t c = 32; c <= 512; c *= 2) {
    const size_t b = smem_floor(0, c);
    if (b > kSmemMax || kSmemPerSM / (b + kSmemReserved) != 512 / c || smem_floor(kSmemMax, c) != kSmemMax) return 1;
  }
  printf("%d\n", most);
}
"""


@pytest.mark.skipif(shutil.which("g++") is None, reason="no host compiler")
def test_columns_of_any_ctas_that_fit_together(tmp_path):
    src = tmp_path / "t.cpp"
    src.write_text(SOURCE)
    exe = tmp_path / "t"
    subprocess.run(["g++", "-std=c++17", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    out = subprocess.run([str(exe)], capture_output=True, text=True, check=True).stdout
    assert int(out) == 512
