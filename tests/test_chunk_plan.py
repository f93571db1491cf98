"""Host rule that splits an interpolation's terms into launches (leja_chunk_end,
csrc/erem_internal.h), compiled and walked on the CPU over every forced degree:
a launch whose last vectors are kept never goes past the tape slots of a forced
degree (q_0 .. q_forced)."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
PROGRAM = r"""
#include <cstdio>
#include "erem_internal.h"
int main() {
  using namespace erem;
  for (int forced = 1; forced <= kMaxTerms; ++forced) {
    const int last = forced + kResLag;
    int m = 1, launches = 0;
    while (true) {
      const int end = leja_chunk_end(m, kResTerms, last, forced);
      ++launches;
      if (end < m || end > last || end - m >= kResTerms) return std::printf("degree %d: terms %d to %d\n", forced, m, end), 1;
      if (end == last) break;
      if (end > forced) return std::printf("degree %d: a kept launch ends at %d\n", forced, end), 1;
      m = end + 1;
    }
    if (launches > (forced + kResLag) / kResTerms + 2) return std::printf("degree %d: %d launches\n", forced, launches), 1;
  }
  // free interpolations, and forms without vectors past the degree, as before
  for (int last = 1; last < 600; ++last)
    for (int m = 1; m <= last; ++m)
      for (int chunk : {4, 8, 48, kResTerms}) {
        const int want = m + chunk - 1 < last ? m + chunk - 1 : last;
        if (leja_chunk_end(m, chunk, last, 0) != want || leja_chunk_end(m, chunk, last, last) != want) return 1;
      }
  return 0;
}
"""


def test_launches_stay_inside_the_slots_of_a_forced_degree(tmp_path):
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    cxx = shutil.which(os.environ.get("CXX", "g++"))
    if not cxx or not os.path.exists(os.path.join(cuda, "include", "cuda_runtime.h")):
        pytest.skip("needs a C++ compiler and the CUDA headers")
    src, exe = tmp_path / "plan.cpp", tmp_path / "plan"
    src.write_text(PROGRAM)
    subprocess.run([cxx, "-std=c++17", "-I", os.path.join(cuda, "include"), "-I",
                    os.path.join(ROOT, "paper_1209_5553_gb300", "csrc"), str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
