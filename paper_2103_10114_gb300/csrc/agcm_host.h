// agcm_host.h — host-side helpers of the library that need no CUDA.
#pragma once
#include <cstddef>
#include <cstdint>
#include <map>
#include <mutex>
#include <unordered_map>
#include <utility>

namespace agcm {

// Memory from a caller's hook, which may return any alignment, while kernels
// read tables and workspaces by loads and copies of 16 bytes: a block that is
// not aligned is given back, a larger one is taken and its first aligned
// address used.
class AlignedBlocks {
 public:
  static constexpr uintptr_t kAlign = 256;  // as cudaMalloc's
  template <class Take, class Give>
  void* take(size_t bytes, Take take, Give give) {
    void* p = take(bytes);
    if (!p || ((uintptr_t)p & 15) == 0) return p;
    give(p);
    if (!(p = take(bytes + kAlign - 1))) return nullptr;
    void* const q = (void*)(((uintptr_t)p + kAlign - 1) & ~(kAlign - 1));
    if (q != p) {
      std::lock_guard<std::mutex> lk(mu_);
      hook_[q] = p;
    }
    return q;
  }
  // The hook's own address of a block.
  void* release(void* q) {
    std::lock_guard<std::mutex> lk(mu_);
    const auto it = hook_.find(q);
    if (it == hook_.end()) return q;
    void* const p = it->second;
    hook_.erase(it);
    return p;
  }

 private:
  std::mutex mu_;
  std::unordered_map<void*, void*> hook_;
};

// The dynamic shared memory each kernel may be launched with, which is set per
// device and must hold for every thread that is about to launch: it is only
// ever raised, by one thread at a time.
class SharedLimits {
 public:
  // set(bytes) makes the limit `bytes` on device dev and returns 0 if it could.
  template <class Set>
  auto raise(int dev, const void* kernel, size_t bytes, Set set) -> decltype(set(bytes)) {
    std::lock_guard<std::mutex> lk(mu_);
    size_t& now = size_[{dev, kernel}];
    if (now >= bytes) return {};
    const auto rc = set(bytes);
    if (rc == decltype(set(bytes)){}) now = bytes;
    return rc;
  }

 private:
  std::mutex mu_;
  std::map<std::pair<int, const void*>, size_t> size_;
};

}  // namespace agcm
