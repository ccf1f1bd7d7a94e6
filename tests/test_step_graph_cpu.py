"""Blocks of solver iterations as graphs, on the CPU against a fake of the CUDA calls: a capture that is refused
(at any of its calls) is launched one by one on the legacy default stream, and ends the solve on the caller's own
stream; an accepted one is captured once and replayed."""
import os
import shutil
import subprocess

import pytest

from paper_1403_0968_gb300 import build

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CUDA = os.path.dirname(os.path.dirname(shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"))

PROGRAM = r"""
#include "sem_graph.h"
#include <cstdio>
#include <cstdlib>

static int fail_at, launches, destroyed, streams;
static cudaError_t at(int call) { return call == fail_at ? cudaErrorStreamCaptureUnsupported : cudaSuccess; }
sem_status sem_fail(sem_status s, const std::string &) { return s; }
extern "C" {
cudaError_t cudaStreamCreateWithFlags(cudaStream_t *s, unsigned int) {
  if (at(1) != cudaSuccess) return at(1);
  *s = reinterpret_cast<cudaStream_t>(64);
  ++streams;
  return cudaSuccess;
}
cudaError_t cudaStreamDestroy(cudaStream_t) { return --streams, cudaSuccess; }
cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode) { return at(2); }
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t *g) {
  *g = at(4) == cudaSuccess ? reinterpret_cast<cudaGraph_t>(8) : nullptr;
  return at(4);
}
cudaError_t cudaGraphInstantiate(cudaGraphExec_t *e, cudaGraph_t, unsigned long long) {
  *e = reinterpret_cast<cudaGraphExec_t>(8);  // (also on failure: nothing may be destroyed then)
  return at(5);
}
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) { return ++launches, at(6); }
cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return ++destroyed, cudaSuccess; }
cudaError_t cudaGetLastError(void) { return cudaSuccess; }
const char *cudaGetErrorString(cudaError_t) { return ""; }
}

int main(int, char **argv) {
  fail_at = atoi(argv[1]);
  cudaStream_t st = reinterpret_cast<cudaStream_t>((size_t)atoi(argv[2]));
  int eager = 0, captured = 0, status = SEM_OK;
  {
    StepGraph g;
    for (int i = 0; i < 3 && status == SEM_OK; ++i)
      status = replay(st, &g, [&](cudaStream_t on) {
        const bool capturing = !eager && !captured && !g.refused;
        ++(capturing ? captured : eager);
        if (!capturing && on != st) return SEM_ERR_INVALID;
        return capturing && fail_at == 3 ? SEM_ERR_CUDA : SEM_OK;
      });
  }
  printf("%d %d %d %d %d %d\n", status == SEM_OK, captured, eager, launches, destroyed, streams);
}
"""


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    if shutil.which("g++") is None or not os.path.exists(os.path.join(CUDA, "include", "cuda_runtime.h")):
        pytest.skip("needs a host C++ compiler and the CUDA headers")
    d = tmp_path_factory.mktemp("graph")
    (d / "g.cpp").write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-w", "-I", build.CSRC, "-I", os.path.join(CUDA, "include"), "-o", str(d / "g"),
                    str(d / "g.cpp")], check=True)
    return lambda fail, stream: [int(v) for v in subprocess.run(
        [str(d / "g"), str(fail), str(stream)], check=True, capture_output=True, text=True).stdout.split()]


@pytest.mark.parametrize("stream", [0, 32])
def test_captured_once_and_replayed(program, stream):
    assert program(0, stream) == [1, 1, 0, 3, 1, 0]


# 1 stream creation (only for the default stream), 2 begin, 3 a launch while capturing, 4 end, 5 instantiation
@pytest.mark.parametrize("fail", [1, 2, 3, 4, 5])
def test_refused_capture_on_the_default_stream_runs_eagerly(program, fail):
    ok, captured, eager, launches, destroyed, streams = program(fail, 0)
    assert (ok, eager, launches, destroyed, streams) == (1, 3, 0, 0, 0) and captured == (1 if fail >= 3 else 0)


@pytest.mark.parametrize("fail", [2, 3, 4, 5])
def test_refused_capture_on_the_callers_stream_is_an_error(program, fail):
    ok, captured, eager, launches, destroyed, streams = program(fail, 32)
    assert (ok, eager, launches, destroyed, streams) == (0, 0, 0, 0, 0) and captured == (1 if fail >= 3 else 0)


def test_failed_launch_is_an_error(program):
    assert program(6, 0)[0] == 0
