// Streams beside a launch's own, and the order of a plan's or pack's segments
// over them.
#include "batch.h"

namespace mknn {

bool SideStreams::create() {
  bool ok = cudaEventCreateWithFlags(&fork, cudaEventDisableTiming) == cudaSuccess;
  for (int i = 0; i < kSideStreams && ok; ++i)
    ok = cudaStreamCreateWithFlags(&s[i], cudaStreamNonBlocking) == cudaSuccess &&
         cudaEventCreateWithFlags(&join[i], cudaEventDisableTiming) == cudaSuccess;
  if (!ok) cudaGetLastError();
  return ok;
}

void SideStreams::destroy() {
  if (fork) cudaEventDestroy(fork);
  for (int i = 0; i < kSideStreams; ++i) {
    if (join[i]) cudaEventDestroy(join[i]);
    if (s[i]) cudaStreamDestroy(s[i]);
  }
  *this = SideStreams{};
}

cudaError_t SideStreams::fork_from(cudaStream_t from, int n) const {
  cudaError_t e = cudaEventRecord(fork, from);
  for (int i = 0; i < n && e == cudaSuccess; ++i) e = cudaStreamWaitEvent(s[i], fork, 0);
  return e;
}

cudaError_t SideStreams::join_to(cudaStream_t from, int n) const {
  cudaError_t first = cudaSuccess;
  for (int i = 0; i < n; ++i) {
    cudaError_t e = cudaEventRecord(join[i], s[i]);
    if (e == cudaSuccess) e = cudaStreamWaitEvent(from, join[i], 0);
    if (first == cudaSuccess) first = e;
  }
  return first;
}

cudaError_t launch_segments(const ReqDev* d_reqs, const Item* d_items, unsigned* d_next,
                            const std::vector<Segment>& segs, cudaStream_t s,
                            const SideStreams& side, int64_t queries) {
  const bool split = segs.size() > 1 && side.fork && queries <= kSplitMaxQueries;
  const int nside = split ? (int)std::min<size_t>(kSideStreams, segs.size() - 1) : 0;
  return side.beside(s, nside, [&]() {
    cudaError_t e = cudaSuccess;
    for (size_t i = 0; i < segs.size() && e == cudaSuccess; ++i) {
      const Segment& g = segs[i];
      const int on = (int)(i % (size_t)(nside + 1));
      e = launch_batch_kernel(d_reqs, d_items + g.begin, g.count, g.units, d_next + i, g.launch,
                              on ? side.s[on - 1] : s);
    }
    return e;
  });
}

}  // namespace mknn
