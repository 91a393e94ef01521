// Dynamic shared memory beyond the 48 KB default that kernels have been granted.  The limit is an attribute of a
// kernel on one device, shared by every solver that launches it there, so it only ever grows, and a second device of
// a process needs a grant of its own.
#pragma once
#include <cstddef>
#include <map>
#include <mutex>
#include <utility>

class SmemGrants {
 public:
  // Calls set() where kernel has been granted fewer than bytes on device; returns its error (0: none, and the
  // grant is remembered).
  template <typename Set>
  auto grant(int device, const void* kernel, size_t bytes, Set set) -> decltype(set()) {
    std::lock_guard<std::mutex> lock(mu_);
    size_t& have = have_[{device, kernel}];
    if (bytes <= have) return {};
    const auto e = set();
    if (e == decltype(set()){}) have = bytes;
    return e;
  }

 private:
  std::mutex mu_;
  std::map<std::pair<int, const void*>, size_t> have_;
};
