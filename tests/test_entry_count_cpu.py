"""The work entries of an expert: the device function's quotient is exact for
every number of selections that a call can have (2^20 tokens of up to 32)."""
import subprocess

from paper_2609_34117_gb300 import build

SOURCE = r"""
#include <cstdio>
#include "common.cuh"
int main() {
  for (int chunk = 16; chunk <= slimwise::kMaxTokTile; chunk += 16) {
    const float inv = 1.0f / (float)chunk;
    for (int n = 0; n <= (1 << 25); ++n)
      if (slimwise::entry_count(n, chunk, inv) != (n + chunk - 1) / chunk) {
        std::printf("n %d chunk %d\n", n, chunk);
        return 1;
      }
  }
  return 0;
}
"""


def test_entry_count_is_exact(tmp_path):
    src, exe = tmp_path / "count.cu", tmp_path / "count"
    src.write_text(SOURCE)
    subprocess.run([build._nvcc(), *build.ARCH, "-O2", "-std=c++17", "-I", build.INCLUDE, "-I",
                    build.CSRC, str(src), "-o", str(exe)], check=True, capture_output=True, text=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
