"""What hydra_prefill and hydra_verify make of the runtime's answer to "is this stream being captured", on the CPU with made-up answers: a failure of something else is
reported under its own name, not as a call under capture."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
PKG = os.path.join(ROOT, "paper_2402_05109_b200")

PROGRAM = r"""
#include "launch.h"
#include <cstdio>
#include <cstring>
#include <initializer_list>
using namespace hydra;
int main() {
  bool c = true;
  if (capture_answer(cudaSuccess, cudaStreamCaptureStatusNone, &c) != HYDRA_OK || c) return 1;
  for (auto s : {cudaStreamCaptureStatusActive, cudaStreamCaptureStatusInvalidated})
    if (c = false, capture_answer(cudaSuccess, s, &c) != HYDRA_OK || !c) return 2;
  if (c = false, capture_answer(cudaErrorStreamCaptureImplicit, cudaStreamCaptureStatusNone, &c) != HYDRA_OK || !c) return 3;
  for (cudaError_t e : {cudaErrorInvalidResourceHandle, cudaErrorLaunchFailure, cudaErrorContextIsDestroyed}) {
    if (capture_answer(e, cudaStreamCaptureStatusNone, &c) != HYDRA_ERR_CUDA) return 4;
    if (!strstr(hydra_last_error(), cudaGetErrorString(e)) || strstr(hydra_last_error(), "under capture")) return printf("%s\n", hydra_last_error()), 5;
  }
  return 0;
}
"""


def test_answers(tmp_path):
    from paper_2402_05109_b200.build import build
    build()
    src, exe = tmp_path / "answers.cu", tmp_path / "answers"
    src.write_text(PROGRAM)
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    subprocess.run([nvcc, "-gencode", "arch=compute_100a,code=sm_100a", "-std=c++17", "-O2", "-I", os.path.join(PKG, "csrc"), str(src), "-o", str(exe),
                    "-L", PKG, "-lhydra", "-Xlinker", "-rpath=" + PKG], check=True, capture_output=True, text=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, (r.returncode, r.stdout)
