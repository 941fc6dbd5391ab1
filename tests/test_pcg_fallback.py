"""CPU check of what nk_pcg_solve does when the cooperative launch of its resident
CG run is refused (csrc/pcg_resident.h, compiled with the host C++ compiler, with
fakes of the launch and of the graph-replayed run): the replayed form takes over
at once and for the rest of the solve, every other error is passed on."""

import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2303_05420_gb300", "csrc")

PROGRAM = r"""
#include <cstdio>
#include "pcg_resident.h"
static int res, rep;
static double seen;
static cudaError_t run(bool* r, cudaError_t launch) {
  return nk_cg_either(r, 1e-3, 3e-2, [&](double t) { ++res; seen = t; return launch; },
                      [&](double t) { ++rep; seen = t; return cudaSuccess; });
}
#define CHECK(x) if (!(x)) { std::printf("FAIL line %d\n", __LINE__); return 1; }
int main() {
  bool r = true;
  CHECK(run(&r, cudaSuccess) == cudaSuccess && r && res == 1 && rep == 0 && seen == 1e-3);
  // refused: the replayed form, at its own tolerance, and no further attempt
  for (cudaError_t e : {cudaErrorCooperativeLaunchTooLarge, cudaErrorLaunchOutOfResources, cudaErrorNotSupported}) {
    r = true;
    res = rep = 0;
    CHECK(run(&r, e) == cudaSuccess && !r && res == 1 && rep == 1 && seen == 3e-2);
    CHECK(run(&r, e) == cudaSuccess && !r && res == 1 && rep == 2 && seen == 1e-3);
  }
  // errors of a run that did start stay errors
  for (cudaError_t e : {cudaErrorLaunchTimeout, cudaErrorLaunchFailure, cudaErrorIllegalAddress}) {
    r = true;
    res = rep = 0;
    CHECK(run(&r, e) == e && r && res == 1 && rep == 0);
  }
  std::printf("ok\n");
  return 0;
}
"""


def test_refused_launch_falls_back(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    include = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nvcc))), "include")
    if cxx is None or not os.path.exists(os.path.join(include, "cuda_runtime.h")):
        pytest.skip("no host C++ compiler or no CUDA headers")
    src, exe = tmp_path / "fallback.cpp", str(tmp_path / "fallback")
    src.write_text(PROGRAM)
    subprocess.run([cxx, "-O1", "-std=c++17", "-I", CSRC, "-I", include, str(src), "-o", exe], check=True)
    out = subprocess.run([exe], capture_output=True, text=True, timeout=60)
    assert out.returncode == 0 and out.stdout.strip() == "ok", out.stdout + out.stderr
