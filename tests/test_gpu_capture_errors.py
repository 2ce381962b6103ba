"""A kernel launch that the runtime refuses during a capture (here for its shared memory, which no GPU has) is an error
of the capture: no graph that leaves the kernel out."""
import os
import subprocess

import pytest

from paper_1211_0585_gb300 import build as B

pytestmark = pytest.mark.gpu

SOURCE = r"""
#include "wf_internal.h"
#include <cstdio>
namespace wfk { wf_status cuda_status(cudaError_t e, const char *) { return e == cudaSuccess ? WF_OK : WF_ECUDA; } }
__global__ void one(int *p) { *p += 1; }
int main() {
  int *p, h = -1;
  cudaStream_t s;
  if (cudaMalloc(&p, sizeof(int)) || cudaMemset(p, 0, sizeof(int)) || cudaStreamCreate(&s)) return 1;
  cudaGraphExec_t bad = nullptr, good = nullptr;
  const int refused = wfk::capture_graph(s, 2, &bad, "refused", [&] { one<<<1, 1, 16 << 20, s>>>(p); });
  const int taken = wfk::capture_graph(s, 3, &good, "taken", [&] { one<<<1, 1, 0, s>>>(p); });
  if (!taken) cudaGraphLaunch(good, s);
  cudaMemcpyAsync(&h, p, sizeof(int), cudaMemcpyDeviceToHost, s);
  if (cudaStreamSynchronize(s)) return 2;
  std::printf("%d %d %d %d\n", refused == WF_ECUDA, bad == nullptr, taken, h);
}
"""


def test_refused_launch_fails_the_capture(tmp_path):
    src, exe = str(tmp_path / "t.cu"), str(tmp_path / "t")
    with open(src, "w") as f:
        f.write(SOURCE)
    subprocess.check_call([B.nvcc(), *B.ARCH, "-std=c++17", "-I", B.INCLUDE, "-I", B.CSRC, src, "-o", exe])
    assert subprocess.check_output([exe], text=True, env=dict(os.environ)).split() == ["1", "1", "0", "3"]
