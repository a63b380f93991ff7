"""The multiply-and-shift division of hga_common.cuh (the kernels' index arithmetic) against the host's own division: every small
divisor, powers of two and their neighbours, random ones and the largest, at the multiples where a wrong multiplier shows."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
PROGRAM = r"""
#include <cstdio>
#include <random>
#include "hga_common.cuh"
int main() {
  const uint32_t top = 0x7fffffffu;
  std::mt19937 rng(1);
  long bad = 0, n_div = 0;
  auto check = [&](uint32_t d) {
    const hga::Div by((int)d);
    auto at = [&](uint64_t n) { if (n <= top && (uint32_t)by((int)n) != (uint32_t)n / d) ++bad; };
    ++n_div;
    for (uint64_t n : {0u, 1u, 2u, top - 1, top}) at(n);
    const uint32_t q_max = top / d;
    for (int i = 0; i < 64; ++i) {          // multiples, one below and one above; the largest among them
      const uint64_t q = i < 2 ? q_max - (q_max ? i : 0) : i < 8 ? i : rng() % (q_max + 1ull), m = q * d;
      at(m); at(m + 1); at(m + d - 1);
      if (m) at(m - 1);
    }
  };
  for (uint32_t d = 1; d <= 4096; ++d) check(d);
  for (int s = 1; s < 31; ++s)
    for (int e = -1; e <= 1; ++e) check((1u << s) + e);
  for (int i = 0; i < 100000; ++i) { const uint32_t d = rng() >> (1 + rng() % 31); check(d ? d : 1); }
  check(top); check(top - 1);
  printf("%ld %ld\n", n_div, bad);
  return bad != 0;
}
"""


def test_division_is_exact_below_2_31(tmp_path):
    cuda = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "include")
    if shutil.which("g++") is None or not os.path.exists(os.path.join(cuda, "cuda_runtime.h")):
        pytest.skip("needs g++ and the CUDA headers")
    src, exe = tmp_path / "div.cpp", tmp_path / "div"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-O2", "-w", "-I", os.path.join(ROOT, "include"), "-I", os.path.join(ROOT, "paper_2607_15105_b200", "csrc"),
                    "-I", cuda, str(src), "-o", str(exe)], check=True)
    out = subprocess.run([str(exe)], capture_output=True, text=True)
    assert out.returncode == 0, out.stdout
