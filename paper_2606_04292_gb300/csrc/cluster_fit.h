// How big a thread-block cluster a launch takes: host rules without CUDA, so
// that they can be checked without a device.
#pragma once
#include <atomic>

namespace rich {

constexpr int CLUSTER_MAX = 16;        // blocks; more than 8 need the kernel's consent (a non-portable size)

// For one kernel on one device and each size (1, 2, 4, 8, 16 blocks): one more
// than the clusters the device holds at once; 0 until it has been asked.
struct ClusterFit {
  std::atomic<int> known[5] = {};
};

// The clusters of 2^k blocks the device holds at once.  Api: pending() says
// whether an earlier error waits to be reported, consent() allows the
// non-portable size, held(blocks) asks the device (negative: the query
// failed), clear() takes back the error of a query that failed.  The answer
// is fixed per kernel and device and kept: a launch outside a graph otherwise
// pays the two runtime calls each time.  While an error is pending nothing is
// asked, so that a failing query cannot take its place: portable sizes then
// count as placeable.
template <typename Api>
inline int clusters_held(ClusterFit& fit, int k, Api&& api) {
  const int kept = fit.known[k].load(std::memory_order_relaxed);
  if (kept > 0) return kept - 1;
  const bool portable = k < 4;
  if (api.pending()) return portable ? 1 : 0;
  const int n = portable || api.consent() ? api.held(1 << k) : -1;
  if (n < 0) {
    api.clear();
    return portable ? 1 : 0;
  }
  fit.known[k].store(n + 1, std::memory_order_relaxed);
  return n;
}

// The blocks per cluster: the largest power of two up to `blocks` of which the
// device holds `clusters` clusters at once (1 if it holds that many of none).
template <typename Api>
inline int fit_blocks(ClusterFit& fit, int blocks, int clusters, Api&& api) {
  for (int k = 4; k > 0; --k)
    if ((1 << k) <= blocks && clusters_held(fit, k, api) >= clusters) return 1 << k;
  return 1;
}

}  // namespace rich
