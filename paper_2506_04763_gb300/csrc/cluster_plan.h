// cluster_plan.h — the cluster size a kernel is launched with whose CTAs take
// most of an SM's shared memory (k_lu_cluster, k_vcycle_cl).  Host code only,
// the CUDA calls behind `Api`.
//
// Api (of one kernel, on the current device):
//   int device()                          its number, < 0: the query failed
//   size_t smem_optin()                   shared memory a CTA may ask for, 0: failed
//   bool allow(size_t cap)                sets the kernel's non-portable cluster size and shared-memory cap
//   int clusters(int cs, size_t smem)     how many such clusters can run at once, < 0: failed
#pragma once
#include <array>
#include <cstddef>
#include <map>
#include <mutex>
#include <vector>

namespace rf {

// Whether clusters of a kernel can run, by device, kernel, size and bytes: asked
// once per process (the query takes longer than a launch).  A query that failed is
// asked again.
class ClusterAnswers {
 public:
  template <class Ask>
  bool fits(const std::array<long long, 4>& key, Ask ask) {
    std::lock_guard<std::mutex> lk(mu_);
    const auto it = known_.find(key);
    if (it != known_.end()) return it->second;
    const int n = ask();
    if (n < 0) return false;
    return known_[key] = n > 0;
  }

 private:
  std::mutex mu_;
  std::map<std::array<long long, 4>, bool> known_;
};

// The first of `sizes` whose CTAs' shared memory (smem(cs)) fits the device and of
// which a cluster can run; 0: none, the caller takes a kernel without a cluster.
// Function attributes belong to a device, so they are set on each one that asks,
// before its first query.
template <class Api, class Smem>
int choose_cluster(Api&& api, ClusterAnswers& known, int kernel, const std::vector<int>& sizes, Smem smem) {
  const int dev = api.device();
  const size_t cap = dev < 0 ? 0 : api.smem_optin();
  if (cap == 0) return 0;
  for (const int cs : sizes) {
    const size_t bytes = smem(cs);
    if (bytes <= cap && known.fits({dev, kernel, cs, (long long)bytes},
                                   [&] { return api.allow(cap) ? api.clusters(cs, bytes) : -1; }))
      return cs;
  }
  return 0;
}

}  // namespace rf
