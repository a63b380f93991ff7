"""The diagnostic build's record of a wait that gave up holds the line of that wait, also where a role waits by a call of its own: a
small program around hga_bwd_sm100.cuh whose one warp waits for a barrier that nothing completes."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
NVCC = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
PROGRAM = r"""
#include <cstdio>
#include "hga_common.cuh"
#include "hga_bwd_sm100.cuh"
using namespace hga;
__global__ void k_give_up(int which, int* out) {
  __shared__ uint64_t never;               // one arrival expected, none ever made
  __shared__ int flag;
  if (threadIdx.x == 0) {
    sm100::mbar_init(&never, 1);
    flag = 0;
    sm100::fence_barrier_init();
    g_dbg_fail[0] = 0;
  }
  __syncwarp();
  volatile int* abort = &flag;
  bool ok = true;
  auto by_call = [&](uint64_t* bar, uint32_t parity, int line = __builtin_LINE()) { return ok = wait_out_of_line(bar, parity, abort, line); };
  int expected = 0;
  if (which == 0) { by_call(&never, 0); expected = __LINE__; }
  if (which == 1) { by_call(&never, 0); expected = __LINE__; }
  if (which == 2) { wait_out_of_line(&never, 0, abort); expected = __LINE__; }
  if (which == 3) { ok = bwd_wait(&never, 0, abort); expected = __LINE__; }
  __syncwarp();
  if (threadIdx.x == 0) { out[0] = g_dbg_fail[0] & 0xffff; out[1] = expected; out[2] = flag; out[3] = ok; }
}
int main() {
  int* out;
  int h[4];
  if (cudaMallocManaged(&out, sizeof h) != cudaSuccess) return 2;
  for (int which = 0; which < 4; ++which) {
    k_give_up<<<1, 32>>>(which, out);
    if (cudaDeviceSynchronize() != cudaSuccess) return 3;
    printf("%d %d %d\n", out[0], out[1], out[2]);
  }
  return 0;
}
"""


def build(tmp_path):
    src, exe = tmp_path / "lines.cu", tmp_path / "lines"
    src.write_text(PROGRAM)
    subprocess.run([NVCC, "-gencode", "arch=compute_100a,code=sm_100a", "-O2", "-std=c++17", "--expt-relaxed-constexpr", "-DHGA_DEBUG_WAIT", "-w",
                    "-I", os.path.join(ROOT, "include"), "-I", os.path.join(ROOT, "paper_2607_15105_b200", "csrc"), str(src), "-o", str(exe)], check=True)
    return str(exe)


@pytest.mark.gpu
def test_a_wait_that_gives_up_records_its_line(tmp_path):
    if not os.path.exists(NVCC):
        pytest.skip("needs nvcc")
    out = subprocess.run([build(tmp_path)], capture_output=True, text=True, timeout=60)
    assert out.returncode == 0, out.stderr
    rows = [tuple(int(x) for x in line.split()) for line in out.stdout.splitlines()]
    assert len(rows) == 4 and len({r[1] for r in rows}) == 4
    for recorded, expected, flag in rows:
        assert recorded == expected == flag, rows
