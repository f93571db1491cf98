"""Host rules of the launches (csrc/erem_internal.h), compiled and walked on the
CPU."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
HEAD = """
#include <cstdio>
#include "erem_internal.h"
using namespace erem;
"""


def run_cpp(tmp_path, program):
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    cxx = shutil.which(os.environ.get("CXX", "g++"))
    if not cxx or not os.path.exists(os.path.join(cuda, "include", "cuda_runtime.h")):
        pytest.skip("needs a C++ compiler and the CUDA headers")
    src, exe = tmp_path / "rule.cpp", tmp_path / "rule"
    src.write_text(HEAD + program)
    subprocess.run([cxx, "-std=c++17", "-I", os.path.join(cuda, "include"), "-I",
                    os.path.join(ROOT, "paper_1209_5553_gb300", "csrc"), str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout


def test_resident_launches_renumber_between_interpolations_only(tmp_path):
    # the messages are cleared with the numbers, and a launch that continues an
    # interpolation takes the last two partial sums of the one before
    run_cpp(tmp_path, r"""
int main() {
  for (unsigned start = kResBaseTop - 5000; start < kResBaseTop + 5000; ++start)
    for (int last : {3, 240, 242, 500, 2100, kMaxTerms + kResLag}) {
      unsigned base = start;
      for (int rep = 0; rep < 3; ++rep)
        for (int m0 = 1; m0 <= last;) {
          const int m1 = leja_chunk_end(m0, kResTerms, last, 0);
          if (res_renumbers(base, m0)) {
            if (m0 > 1) return std::printf("base %u: cleared before term %d\n", base, m0), 1;
            base = 0;
          }
          if (base + (unsigned)m1 < base) return std::printf("base %u wraps\n", base), 1;
          base += (unsigned)m1 + 1u;
          m0 = m1 + 1;
        }
      if (base > kResBaseTop + 200000u) return std::printf("never renumbered from %u\n", start), 1;
    }
  return 0;
}
""")
