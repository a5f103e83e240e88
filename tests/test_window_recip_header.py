"""CPU check of the library's own window reciprocal (mf_internal.h, compiled for the host): the quotient that the filter
kernels form is n / window at the first and the last sample of every window of every length."""

import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CUDA = os.environ.get("CUDA_HOME", "/usr/local/cuda")

SOURCE = r"""
#include "mf_internal.h"
#include <cstdio>
int main() {
  for (int64_t w = 1; w <= mf::kMaxN; ++w) {
    const uint64_t r = mf::window_recip(w);
    auto right = [&](int64_t n, int64_t quotient) {
      const unsigned __int128 full = (unsigned __int128)n * r;
      return full >> 64 == 0 && (int64_t)((uint64_t)n * r >> mf::kRecipBits) == quotient;
    };
    for (int64_t q = 0; q * w < mf::kMaxN; ++q) {
      const int64_t last = q * w + w - 1 < mf::kMaxN ? q * w + w - 1 : mf::kMaxN - 1;
      if (!right(q * w, q) || !right(last, q)) return std::printf("window %lld, %lld\n", (long long)w, (long long)q), 1;
    }
  }
  return 0;
}
"""


@pytest.mark.skipif(not shutil.which("g++") or not os.path.exists(f"{CUDA}/include/cuda.h"), reason="no host compiler")
def test_every_window_length(tmp_path):
    src, exe = tmp_path / "recip.cc", tmp_path / "recip"
    src.write_text(SOURCE)
    subprocess.run(["g++", "-std=c++17", "-O2", f"-I{CUDA}/include", f"-I{ROOT}/include",
                    f"-I{ROOT}/paper_2309_00019_gb300/csrc", str(src), "-o", str(exe)], check=True)
    run = subprocess.run([str(exe)], capture_output=True, text=True)
    assert run.returncode == 0, run.stdout
