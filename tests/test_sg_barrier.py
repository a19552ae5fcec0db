"""The barrier between same-generation iterations compares a running 32-bit count
of arrivals with the count that ends an iteration; both wrap after 2^32
arrivals.  On the host: a CTA waits exactly until the last CTA of its iteration
has arrived, also where the count or the target wraps."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2607_17571_gb300", "csrc")
PROGRAM = r'''
#include "wg_device.cuh"
int main() {
  const uint32_t grids[] = {1, 3, 152, 2432};
  const uint64_t top = 1ull << 32;
  for (uint32_t g : grids) {
    const uint64_t k0[] = {0, 1, top / g - 2, top / g - 1, top / g, top / g + 1, 3 * (top / g)};
    for (uint64_t k : k0)
      // iteration k: the arrivals run from k * g (all of the iteration before) to
      // (k + 2) * g (a CTA may still poll when the others have arrived once more)
      for (uint64_t a = k * g; a <= (k + 2) * g; ++a)
        if (wg::sg_arrived((uint32_t)a, (uint32_t)((k + 1) * g)) != (a >= (k + 1) * g)) return 1;
  }
  return 0;
}
'''


def test_count_and_target_wrap(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("needs nvcc")
    src, exe = tmp_path / "barrier.cu", tmp_path / "barrier"
    src.write_text(PROGRAM)
    subprocess.run([nvcc, "-std=c++17", "-I", CSRC, "-gencode", "arch=compute_103a,code=sm_103a",
                    str(src), "-o", str(exe)], check=True, capture_output=True)
    assert subprocess.run([str(exe)]).returncode == 0
