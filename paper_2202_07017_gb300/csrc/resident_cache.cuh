// Resident blocks per SM of a kernel, asked once per launch configuration.
#pragma once

#include <cstddef>
#include <map>
#include <mutex>
#include <tuple>

namespace sv {

// The grids of persistent kernels follow from it, and so does the order in which a
// reduction's parts meet: every quantity that the answer depends on is in the key
// (passes of different slice sizes may ask for the same shared memory with different
// block sizes), so that a call's grid never depends on the calls before it.
class ResidentCache {
 public:
  // query() if the configuration is new; it may be called by several threads at once.
  template <typename Query>
  int get(const void* kernel, int device, int threads, size_t smem, const Query& query) {
    std::lock_guard<std::mutex> lk(mu_);
    int& blocks = known_[std::make_tuple(kernel, device, threads, smem)];
    if (!blocks) blocks = query();
    return blocks;
  }

 private:
  std::mutex mu_;
  std::map<std::tuple<const void*, int, int, size_t>, int> known_;
};

}  // namespace sv
