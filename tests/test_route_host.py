"""Which kernel a call takes and what scratch it touches (CPU): csrc/capi.cu
and csrc/lane_rule.cpp compiled as plain C++ against fakes of the CUDA runtime
and of the launches, on a cloud that claims to have box trees."""
from __future__ import annotations

import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2605_02224_gb300", "csrc")
CUDA = os.path.dirname(os.path.dirname(shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"))

pytestmark = pytest.mark.skipif(
    shutil.which("g++") is None or not os.path.exists(os.path.join(CUDA, "include/cuda_runtime.h")),
    reason="needs g++ and the CUDA headers")

FAKES = r"""
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include "../../include/mknn.h"
#include "batch.h"
#include "cloud.h"

static int allocs = 0;         // cudaMalloc and cudaStreamSynchronize calls
static size_t largest = 0;     // device memory: a larger allocation fails
static bool capturing = false;
static cudaError_t last = cudaSuccess;  // what cudaGetLastError returns and clears
static mknn::PlainLaunch L;             // the last launch
static mknn::Mode tuned{0, 0};

extern "C" {
cudaError_t cudaGetDevice(int* d) { *d = 0; return cudaSuccess; }
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaGetLastError() { const cudaError_t e = last; last = cudaSuccess; return e; }
const char* cudaGetErrorString(cudaError_t) { return "error"; }
cudaError_t cudaMalloc(void** p, size_t n) {
  ++allocs;
  if (capturing) return last = cudaErrorStreamCaptureUnsupported;
  if (n > largest) return last = cudaErrorMemoryAllocation;
  *p = malloc(n);
  return cudaSuccess;
}
cudaError_t cudaFree(void* p) { free(p); return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { ++allocs; return cudaSuccess; }
cudaError_t cudaStreamIsCapturing(cudaStream_t, cudaStreamCaptureStatus* st) {
  *st = capturing ? cudaStreamCaptureStatusActive : cudaStreamCaptureStatusNone;
  return cudaSuccess;
}
cudaError_t cudaDeviceSynchronize() { return cudaSuccess; }
cudaError_t cudaMemcpy(void* d, const void* s, size_t n, cudaMemcpyKind) { memcpy(d, s, n); return cudaSuccess; }
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind, cudaStream_t) { memcpy(d, s, n); return cudaSuccess; }
cudaError_t cudaMemset(void* d, int v, size_t n) { memset(d, v, n); return cudaSuccess; }
cudaError_t cudaMemsetAsync(void* d, int v, size_t n, cudaStream_t) { memset(d, v, n); return cudaSuccess; }
}

namespace mknn {
Mode tuned_mode(int, int64_t, int) { return tuned; }
int default_lanes(int k) { return k >= kWarpMinK ? 32 : 1; }
int default_placement(int, int lanes) { return lanes == 1 || lanes == 32 ? 2 : 1; }
int plain_max_k(int lanes) { return lanes == 4 || lanes == 8 ? 64 : 128; }
static int sms = 152;
int num_sms() { return sms; }
size_t sort_workspace_bytes(int64_t nq) { return kSortHistBytes + (((size_t)nq * 4 + 255) & ~(size_t)255); }
static cudaError_t launched() { return cudaGetLastError(); }  // as the launchers return it
cudaError_t launch_query_sort(const CloudDevHost&, const float*, int32_t, int64_t, void*, int32_t*, cudaStream_t) { return launched(); }
cudaError_t launch_query_sort_any(const CloudDevHost&, const float*, int32_t, int64_t, void*, int32_t*, int32_t*, cudaStream_t) { return launched(); }
cudaError_t launch_gather_sites(const CloudDevHost&, const int32_t*, int64_t, const int32_t*, int32_t, float4*, int32_t*, cudaStream_t) { return launched(); }
cudaError_t launch_fill_entries(const void*, const int32_t*, int64_t, void*, cudaStream_t) { return launched(); }
cudaError_t launch_knn_plain(const CloudDevHost&, const PlainLaunch& l, cudaStream_t) { L = l; return launched(); }
}  // namespace mknn

static char dev[1 << 12];
static mknn_cloud* cloud(int hub, int64_t longest) {
  mknn_cloud* c = new mknn_cloud;
  c->n = 200000;
  c->device = 0;
  c->d_pts = dev;
  c->d_hub_of = (int32_t*)dev;
  c->hub_longest = longest;
  c->hub_ = hub;
  return c;
}
#define CHECK(c) do { if (!(c)) { std::printf("line %d: %s (k %d, lanes %d)\n", __LINE__, #c, L.k, L.lanes); std::exit(1); } } while (0)
"""

MAIN_ROOM = r"""
int main() {
  const int64_t nq = 1 << 20;  // above every one-lane line below k = 48
  static float q[4], d2[4];
  static int32_t idx[4], order[4];
  uintptr_t stream = 1;  // library scratch is kept per stream: a new one each time
  for (int hub : {14, 17})
    for (int k : {1, 8, 16, 32, 40, 47, 48, 100}) {
      mknn_cloud* c = cloud(hub, int64_t(1) << hub);
      const bool one = k < 48;  // the trees serve every k
      auto run = [&](mknn_knn_opts o, uintptr_t s) {
        allocs = 0;
        L = mknn::PlainLaunch{};
        return mknn_knn_ex(c, q, nq, 3, k, nullptr, 0, idx, d2, &o, (mknn_stream_t)s);
      };
      mknn_knn_opts sorted{}, ordered{};
      ordered.order = order;
      const size_t full = mknn_knn_workspace_size(nq, nullptr);
      const size_t sort_only = full - mknn::defer_bytes(nq);
      // caller workspace: with room for the hand-over, and without
      largest = 0;
      mknn_knn_opts o = sorted;
      o.workspace = dev;
      o.workspace_bytes = full;
      CHECK(run(o, ++stream) == MKNN_OK && L.lanes == (one ? 1 : 32) && !!L.defer == one && !allocs);
      o.workspace_bytes = full - 1;
      CHECK(run(o, ++stream) == MKNN_OK && L.lanes == 32 && L.placement == 2 && !L.defer && !allocs);
      o.workspace_bytes = sort_only;
      CHECK(run(o, ++stream) == MKNN_OK && L.lanes == 32 && !L.defer);
      o.lanes = 1;  // asked for: one lane reads the lists through
      o.placement = 2;
      CHECK(run(o, ++stream) == MKNN_OK && L.lanes == 1 && !L.defer);
      o.workspace_bytes = sort_only - 1;
      CHECK(run(o, ++stream) == MKNN_EINVAL);
      // library scratch, no device memory: an order given needs none
      CHECK(run(ordered, ++stream) == MKNN_OK && L.lanes == 32 && !L.defer);
      CHECK(run(sorted, ++stream) == MKNN_ENOMEM);
      cudaGetLastError();
      largest = sort_only;  // room for the sort only
      CHECK(run(sorted, ++stream) == MKNN_OK && L.lanes == 32 && !L.defer);
      largest = size_t(1) << 40;
      CHECK(run(ordered, ++stream) == MKNN_OK && L.lanes == (one ? 1 : 32) && !!L.defer == one);
      // captured: no allocation, no wait, and no scratch without a sort
      capturing = true;
      CHECK(run(ordered, stream) == MKNN_OK && L.lanes == 32 && !L.defer && !allocs);
      CHECK(run(ordered, ++stream) == MKNN_OK && L.lanes == 32 && !L.defer && !allocs);
      capturing = false;
      CHECK(run(sorted, ++stream) == MKNN_OK && L.lanes == (one ? 1 : 32) && !!L.defer == one);
      capturing = true;  // the scratch is there from the call before
      CHECK(run(sorted, stream) == MKNN_OK && L.lanes == (one ? 1 : 32) && !!L.defer == one && !allocs);
      capturing = false;
      o = sorted;  // room for the sort only
      o.lanes = 32;
      CHECK(run(o, ++stream) == MKNN_OK && L.lanes == 32);
      capturing = true;
      CHECK(run(sorted, stream) == MKNN_OK && L.lanes == 32 && !L.defer && !allocs);
      capturing = false;
      // the longer the lists, the more queries it takes until one lane that
      // reads them through is the faster
      if (one) {
        const int64_t line = 102400 + 1100 * k + (int64_t(90) << hub);
        CHECK(mknn::choose_mode(k, c->n, hub, line - 1, true, false).lanes == 32);
        CHECK(mknn::choose_mode(k, c->n, hub, line, true, false).lanes == 1);
        CHECK(mknn::choose_mode(k, c->n, 11, 200000, true, false).lanes == 32);
        CHECK(mknn::choose_mode(k, c->n, 11, nq, true, false).lanes == 1);
      }
      if (one) {  // a tuned lane per query follows the same rule
        tuned = mknn::Mode{1, 2};
        o = sorted;
        o.workspace = dev;
        o.workspace_bytes = full;
        CHECK(run(o, ++stream) == MKNN_OK && L.lanes == 1 && L.defer);
        o.workspace_bytes = sort_only;
        CHECK(run(o, ++stream) == MKNN_OK && L.lanes == 32 && !L.defer);
        tuned = mknn::Mode{0, 0};
      }
      CHECK(cudaGetLastError() == cudaSuccess);
    }
  std::printf("ok\n");
}
"""


def _run(tmp_path, main):
    src = tmp_path / "t.cpp"
    src.write_text(FAKES + main)
    exe = tmp_path / "t"
    cpp = [os.path.join(CSRC, f) for f in ("lane_rule.cpp", "builder.cpp", "predicates.cpp",
                                           "hub_index.cpp")]
    subprocess.run(["g++", "-std=c++17", "-O1", "-w", f"-I{CSRC}", f"-I{CUDA}/include", str(src),
                    *cpp, "-x", "c++", os.path.join(CSRC, "capi.cu"), "-o", str(exe),
                    "-lpthread"], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0 and r.stdout.strip().endswith("ok"), r.stdout + r.stderr[-4000:]


def test_no_room_for_the_handover_means_one_warp_per_query(tmp_path):
    _run(tmp_path, MAIN_ROOM)


MAIN_TUNED = r"""
int main() {
  // a tuned width below 32 lanes serves large launches; small ones take one
  // warp per query
  for (int lanes : {1, 4, 8, 16})
    for (int k : {1, 8, 16}) {
      tuned = mknn::Mode{lanes, lanes == 1 ? 2 : 1};
      for (int64_t nq : {1, 64, 1000, 10000, 40000}) {
        const mknn::Mode m = mknn::choose_mode(k, 100000, 8, nq, false);
        L.k = k;
        L.lanes = m.lanes;
        CHECK(m.lanes == 32 && m.placement == 2);
      }
      const mknn::Mode m = mknn::choose_mode(k, 100000, 8, 1 << 20, false);
      CHECK(m.lanes == tuned.lanes && m.placement == tuned.placement);
    }
  tuned = mknn::Mode{32, 1};  // registers, when tuned so, at every size
  for (int64_t nq : {64, 1 << 20}) {
    const mknn::Mode m = mknn::choose_mode(8, 100000, 8, nq, false);
    CHECK(m.lanes == 32 && m.placement == 1);
  }
  std::printf("ok\n");
}
"""


def test_tuned_widths_of_small_launches(tmp_path):
    _run(tmp_path, MAIN_TUNED)


MAIN_SMS = r"""
int main() {
  // the number of queries from which one lane is the default, on a GPU and on
  // half of one: 40,960 + 1,100 k, more with long lists and above k = 32
  for (int part : {1, 2})
    for (int k : {1, 16, 32, 33, 47})
      for (int hub : {8, 9, 12}) {
        mknn::sms = 152 / part;
        const bool trees = hub == 12;
        const int64_t line = (40960 + 1100 * k + (k > 32 ? 32768 * (k - 32) : 0) +
                              (hub >= 9 ? 81920 : 0)) / part;
        L.k = k;
        CHECK(mknn::choose_mode(k, 100000, hub, line - 1, trees).lanes == 32);
        CHECK(mknn::choose_mode(k, 100000, hub, line, trees).lanes == 1);
      }
  std::printf("ok\n");
}
"""


def test_one_lane_line_follows_the_number_of_sms(tmp_path):
    _run(tmp_path, MAIN_SMS)
