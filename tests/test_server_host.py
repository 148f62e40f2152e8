"""The serving loop's host side (CPU): csrc/server.cu compiled as plain C++
against fakes of the CUDA runtime calls and of the launches it makes, so that
a launch can fail without a GPU."""
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

# Copies run at once, on the calling thread; events have always happened. The
# faked launch answers every query of a pack with the request's k, or fails.
FAKES = r"""
#include <atomic>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <thread>
#include "../../include/mknn.h"
#include "batch.h"
#include "cloud.h"

std::atomic<int> syncs{0}, forks{0};
std::atomic<bool> fail_launch{false}, fail_sort{false};
static char handles[64];

extern "C" {
cudaError_t cudaGetDevice(int* d) { *d = 0; return cudaSuccess; }
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
cudaError_t cudaMalloc(void** p, size_t n) { *p = calloc(1, n); return cudaSuccess; }
cudaError_t cudaMallocHost(void** p, size_t n) { *p = calloc(1, n); return cudaSuccess; }
cudaError_t cudaFree(void* p) { free(p); return cudaSuccess; }
cudaError_t cudaFreeHost(void* p) { free(p); return cudaSuccess; }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) { *s = (cudaStream_t)handles; return cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { ++syncs; return cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t* e) { *e = (cudaEvent_t)handles; return cudaSuccess; }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventQuery(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) { *ms = 1.f; return cudaSuccess; }
cudaError_t cudaPointerGetAttributes(cudaPointerAttributes* a, const void*) {
  a->type = cudaMemoryTypeHost;
  return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind, cudaStream_t) {
  memcpy(d, s, n);
  return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void* d, int v, size_t n, cudaStream_t) { memset(d, v, n); return cudaSuccess; }
mknn_status mknn_cloud_upload(mknn_cloud*, mknn_stream_t) { return MKNN_OK; }
mknn_status mknn_knn_ex(const mknn_cloud*, const float*, int64_t nq, int32_t, int32_t k,
                        const int32_t*, int32_t, int32_t* idx, float* d2, const mknn_knn_opts* o,
                        mknn_stream_t) {
  if (o->lanes == 4 && k > 64) return MKNN_EINVAL;
  for (int64_t i = 0; i < nq * k; ++i) { idx[i] = k; d2[i] = (float)k; }
  return MKNN_OK;
}
}

namespace mknn {
void set_error(const std::string&) {}
Mode choose_mode(int, int64_t, int, int64_t, bool, bool) { return Mode{32, 2}; }
int default_placement(int, int lanes) { return lanes == 4 ? 1 : 2; }
int variant_index(int lanes, int k, int) { return lanes == 4 ? (k <= 64 ? 2 : -1) : 16; }
std::vector<Segment> make_segments(std::vector<Item>& items, int, const std::vector<int>&) {
  if (items.empty()) return {};
  Segment g;
  g.count = (int)items.size();
  g.units = 1;
  return {g};
}
bool SideStreams::create() { return true; }
void SideStreams::destroy() {}
cudaError_t launch_query_sort_any(const CloudDevHost&, const float*, int32_t, int64_t, void*,
                                  int32_t*, int32_t*, cudaStream_t) {
  return fail_sort ? cudaErrorLaunchFailure : cudaSuccess;
}
cudaError_t launch_segments(const ReqDev* reqs, const Item* items, unsigned*,
                            const std::vector<Segment>& segs, cudaStream_t, const SideStreams&,
                            int64_t) {
  if (fail_launch) return cudaErrorLaunchFailure;
  for (const Segment& g : segs)
    for (int i = g.begin; i < g.begin + g.count; ++i) {
      const ReqDev& R = reqs[items[i].req];
      for (int64_t j = 0; j < (int64_t)items[i].nq * R.k; ++j) {
        R.out_idx[j] = R.k;
        R.out_d2[j] = (float)R.k;
      }
    }
  return cudaSuccess;
}
cudaError_t launch_handover(const ReqDev*, Handover*, int, int, cudaStream_t) { return cudaSuccess; }
int handover_grid(int) { return 1; }
}  // namespace mknn

#define CHECK(c) do { if (!(c)) { std::printf("line %d: %s\n", __LINE__, #c); std::exit(1); } } while (0)

struct Req {
  std::vector<float> q, d2;
  std::vector<int32_t> idx;
  uint64_t ticket = 0;
  int k = 0;
};
static void submit(mknn_server* s, Req& r, int nq, int k, int cloud = 0) {
  r.k = k;
  r.q.assign(3 * nq, 0.f);
  r.idx.assign((size_t)nq * k, -9);
  r.d2.assign((size_t)nq * k, -9.f);
  mknn_request m{};
  m.cloud = cloud;
  m.k = k;
  m.q = r.q.data();
  m.nq = nq;
  m.out_idx = r.idx.data();
  m.out_d2 = r.d2.data();
  CHECK(mknn_server_submit(s, &m, &r.ticket) == MKNN_OK);
}
static bool all(const Req& r, int v) {
  for (int32_t x : r.idx) if (x != v) return false;
  for (float x : r.d2) if (x != (float)v) return false;
  return true;
}
static int state(mknn_server* s, const Req& r) {
  int32_t st = 0;
  CHECK(mknn_server_poll(s, r.ticket, &st) == MKNN_OK);
  return st;
}
static mknn_server* server(mknn_cloud* c, int plain, int lanes) {
  mknn_server_opts o{};
  o.plain = plain;
  o.lanes = lanes;
  o.mem_budget = 64 << 20;
  mknn_server* s = nullptr;
  CHECK(mknn_server_create(&o, &s) == MKNN_OK);
  int32_t id;
  CHECK(mknn_server_add_cloud(s, c, &id) == MKNN_OK);
  return s;
}
"""

MAIN_ERRORS = r"""
int main() {
  mknn_cloud c;
  c.n = 1000;
  c.rowp.assign(1001, 0);
  for (int plain = 0; plain < 2; ++plain) {
    // a k that the server's lanes cannot hold fails alone, its rows untouched
    mknn_server* s = server(&c, plain, 4);
    Req a, b, d;
    submit(s, a, 100, 8);
    submit(s, b, 100, 100);
    submit(s, d, 5000, 64);
    CHECK(mknn_server_drain(s, 10.0) == MKNN_OK);
    CHECK(state(s, a) == 1 && all(a, 8));
    CHECK(state(s, d) == 1 && all(d, 64));
    CHECK(state(s, b) == -(int)MKNN_EINVAL && all(b, -9));
    mknn_serving_stats st;
    CHECK(mknn_server_stats(s, &st) == MKNN_OK && st.completed == 2 && st.failed == 1);
    CHECK(mknn_server_destroy(s, 10.0) == MKNN_OK);
  }
  // a launch that fails: every request of it fails, none is reported done,
  // and the streams are waited for before its memory is given back
  for (int sort = 0; sort < 2; ++sort) {
    mknn_server* s = server(&c, 0, 0);
    Req a, b;
    (sort ? fail_sort : fail_launch) = true;
    syncs = 0;
    submit(s, a, 5000, 8);
    CHECK(mknn_server_drain(s, 10.0) == MKNN_OK);
    CHECK(state(s, a) == -(int)MKNN_ECUDA);
    CHECK(syncs >= 1 + mknn::kSideStreams);
    fail_sort = fail_launch = false;
    submit(s, b, 5000, 8);  // the server goes on
    CHECK(mknn_server_drain(s, 10.0) == MKNN_OK);
    CHECK(state(s, b) == 1 && all(b, 8));
    mknn_serving_stats st;
    CHECK(mknn_server_stats(s, &st) == MKNN_OK && st.completed == 1 && st.failed == 1);
    CHECK(mknn_server_destroy(s, 10.0) == MKNN_OK);
  }
  std::printf("ok\n");
}
"""


def _run(tmp_path, main, *flags):
    src = tmp_path / "t.cpp"
    src.write_text(FAKES + main)
    exe = tmp_path / "t"
    subprocess.run(["g++", "-std=c++17", "-O1", "-w", *flags, f"-I{CSRC}", f"-I{CUDA}/include",
                    str(src), "-x", "c++", os.path.join(CSRC, "server.cu"),
                    os.path.join(CSRC, "builder.cpp"), os.path.join(CSRC, "predicates.cpp"),
                    "-o", str(exe), "-lpthread"], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0 and r.stdout.strip().endswith("ok"), r.stdout + r.stderr[-4000:]


def test_requests_of_a_failed_launch_fail(tmp_path):
    _run(tmp_path, MAIN_ERRORS)


MAIN_THREADS = r"""
int main() {
  mknn_cloud c;
  c.n = 1000;
  c.rowp.assign(1001, 0);
  for (int plain = 0; plain < 2; ++plain) {
    mknn_server* s = server(&c, plain, 0);
    std::vector<std::vector<Req>> reqs(3, std::vector<Req>(400));
    std::vector<std::thread> th;
    for (int t = 0; t < 3; ++t)
      th.emplace_back([&, t] {
        for (int i = 0; i < 400; ++i) {
          int32_t id = 0;
          if (t == 0 && i % 4 == 0) CHECK(mknn_server_add_cloud(s, &c, &id) == MKNN_OK);
          submit(s, reqs[t][i], 1 + i % 7, 1 + (i + t) % 32, id);
        }
      });
    for (auto& t : th) t.join();
    CHECK(mknn_server_drain(s, 60.0) == MKNN_OK);
    for (auto& v : reqs)
      for (Req& r : v) CHECK(state(s, r) == 1 && all(r, r.k));
    CHECK(mknn_server_destroy(s, 10.0) == MKNN_OK);
  }
  std::printf("ok\n");
}
"""


def test_submitting_while_packs_are_launched(tmp_path):
    """Threads that submit requests and add clouds while the scheduler thread
    launches packs: no data race (ThreadSanitizer) and every row is right."""
    probe = tmp_path / "p.cpp"
    probe.write_text("int main() {}")
    built = subprocess.run(["g++", "-fsanitize=thread", str(probe), "-o", str(tmp_path / "p")],
                           capture_output=True)
    if built.returncode or subprocess.run([str(tmp_path / "p")], capture_output=True).returncode:
        pytest.skip("no ThreadSanitizer")
    _run(tmp_path, MAIN_THREADS, "-fsanitize=thread", "-g")
