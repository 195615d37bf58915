// agcm_host.h — host-side helpers of the library that need no CUDA.
#pragma once
#include <cstddef>
#include <cstdint>
#include <mutex>
#include <unordered_map>

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

}  // namespace agcm
