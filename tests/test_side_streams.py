"""Segments over side streams (CPU): csrc/side_streams.cpp compiled as plain
C++ against fakes of the runtime calls and of the kernel launch. Whatever call
fails, a side stream that may hold work is joined back, and the first error is
the one returned."""
from __future__ import annotations

import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2605_02224_gb300", "csrc")
CUDA = os.path.dirname(os.path.dirname(shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"))

PROGRAM = r"""
#include <cstdio>
#include <cstdlib>
#include <map>
#include <set>
#include "batch.h"
static int calls = 0, fail_at = -1, fail_code = 0;
static char mem[64];
static int made = 0;
static cudaError_t step() { return calls++ == fail_at ? (cudaError_t)fail_code : cudaSuccess; }
static std::map<cudaEvent_t, cudaStream_t> recorded;
static std::set<cudaStream_t> busy, joined;
static cudaStream_t const own = (cudaStream_t)(mem + 63);
extern "C" {
cudaError_t cudaGetLastError() { return cudaSuccess; }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) { *s = (cudaStream_t)(mem + made++); return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* s, unsigned) { *s = (cudaEvent_t)(mem + made++); return cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t s) {
  const cudaError_t r = step();
  if (r == cudaSuccess) recorded[e] = s;
  return r;
}
cudaError_t cudaStreamWaitEvent(cudaStream_t s, cudaEvent_t e, unsigned) {
  const cudaError_t r = step();
  if (r == cudaSuccess && s == own) joined.insert(recorded[e]);
  return r;
}
}
namespace mknn {
cudaError_t launch_batch_kernel(const ReqDev*, const Item*, int, uint32_t, unsigned*,
                                const BatchLaunch&, cudaStream_t s) {
  const cudaError_t r = step();
  if (r == cudaSuccess) busy.insert(s);
  return r;
}
}
int main(int argc, char** argv) {  // segments, call that fails, its code
  mknn::SideStreams side;
  if (!side.create()) return 2;
  std::vector<mknn::Segment> segs(std::atoi(argv[1]));
  fail_at = std::atoi(argv[2]);
  fail_code = std::atoi(argv[3]);
  const cudaError_t e = mknn::launch_segments(nullptr, nullptr, nullptr, segs, own, side, 1000);
  busy.erase(own);
  int loose = 0;
  for (cudaStream_t s : busy) loose += joined.count(s) ? 0 : 1;
  std::printf("%d %d %d %d\n", (int)e, calls, (int)busy.size(), loose);
}
"""


@pytest.mark.skipif(
    shutil.which("g++") is None or not os.path.exists(os.path.join(CUDA, "include/cuda_runtime.h")),
    reason="needs g++ and the CUDA headers")
def test_side_streams_are_joined_after_a_failure(tmp_path):
    src = tmp_path / "t.cpp"
    src.write_text(PROGRAM)
    exe = tmp_path / "t"
    subprocess.run(["g++", "-std=c++17", "-O1", "-w", f"-I{CSRC}", f"-I{CUDA}/include", str(src),
                    os.path.join(CSRC, "side_streams.cpp"), "-o", str(exe)], check=True)

    def run(segments, fail_at):
        out = subprocess.run([str(exe), str(segments), str(fail_at), "700"], check=True,
                             capture_output=True, text=True).stdout
        return [int(x) for x in out.split()]

    for segments in (1, 2, 4, 7):
        side = min(3, segments - 1)
        error, calls, busy, loose = run(segments, -1)
        forks = 1 + side if side else 0
        assert (error, calls, busy, loose) == (0, forks + segments + 2 * side, side, 0)
        for at in range(forks + segments):          # a fork or a launch fails
            error, _, _, loose = run(segments, at)
            assert error == 700 and loose == 0, (segments, at)
        for at in range(forks + segments, calls):   # a join fails: the others are made
            error, made, _, loose = run(segments, at)
            assert error == 700 and made >= calls - 1 and loose == 1, (segments, at)
