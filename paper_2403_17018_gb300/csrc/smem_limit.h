// Dynamic shared-memory limits of kernels (host code without CUDA headers).
#pragma once

#include <cstddef>
#include <map>
#include <mutex>
#include <utility>

namespace henry {

// The limit of a kernel is an attribute of the function in one device's
// context, shared by every solver of the process on that device: it is only
// ever raised, to the largest size any solver needs there, so that no
// solver's graph capture can meet a limit lowered by another solver. A
// context on another GPU has to raise its own, hence the key.
class SmemLimits {
 public:
  // set(fn, bytes) changes the current device's limit and returns an error code,
  // zero for success; it is called when `bytes` is above both what every
  // launch may use (48 KB) and what this device's limit was raised to.
  template <typename Set>
  auto raise(int device, const void* fn, std::size_t bytes, Set set) -> decltype(set(fn, bytes)) {
    std::lock_guard<std::mutex> lock(mu_);
    std::size_t& c = cur_[{device, fn}];
    if (bytes <= c || bytes <= 48 * 1024) return {};
    const auto e = set(fn, bytes);
    if (e == decltype(set(fn, bytes)){}) c = bytes;
    return e;
  }

 private:
  std::mutex mu_;
  std::map<std::pair<int, const void*>, std::size_t> cur_;
};

}  // namespace henry
