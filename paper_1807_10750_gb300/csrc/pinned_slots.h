// Small pieces of pinned host memory for what a handle's synchronising calls read.
//
// Pinning a page costs a process 130 us and unpinning it 170, as much as all the
// rest of a small graph's ising_create and ising_destroy, so the handles share pages of
// 64 slots. A page is unpinned when its last slot comes back, but for one, which
// stays for the next handle: 4 KB a process. Safe from any thread.
#pragma once

#include <cuda_runtime.h>

#include <cstddef>
#include <cstdint>
#include <mutex>
#include <new>
#include <vector>

namespace isingx {

class PinnedSlots {
 public:
  static constexpr size_t kSlotBytes = 64;
  static constexpr int kSlots = 64;

  // Memory of its own for the caller, on any device; null without room for it.
  void* take() {
    std::lock_guard<std::mutex> lock(mutex_);
    for (size_t i = 0; i < pages_.size();) {
      Page& p = pages_[i];
      cudaPointerAttributes attr{};
      if (cudaPointerGetAttributes(&attr, p.base) != cudaSuccess || attr.type != cudaMemoryTypeHost) {
        cudaGetLastError();  // a device reset has taken the page: its handles are gone, too
        pages_.erase(pages_.begin() + static_cast<std::ptrdiff_t>(i));
        continue;
      }
      for (int s = 0; s < kSlots; ++s)
        if (!((p.used >> s) & 1u)) {
          p.used |= uint64_t(1) << s;
          return p.base + static_cast<size_t>(s) * kSlotBytes;
        }
      ++i;
    }
    void* base = nullptr;
    if (cudaHostAlloc(&base, kSlots * kSlotBytes, cudaHostAllocPortable) != cudaSuccess) {
      cudaGetLastError();
      return nullptr;
    }
    try {
      pages_.push_back({static_cast<unsigned char*>(base), 1u});
    } catch (const std::bad_alloc&) {
      cudaFreeHost(base);
      return nullptr;
    }
    return base;
  }

  void give(void* slot) {
    if (slot == nullptr) return;
    std::lock_guard<std::mutex> lock(mutex_);
    const unsigned char* at = static_cast<unsigned char*>(slot);
    bool spare = false;
    for (const Page& p : pages_) spare = spare || p.used == 0u;
    for (size_t i = 0; i < pages_.size(); ++i) {
      Page& p = pages_[i];
      if (at < p.base || at >= p.base + kSlots * kSlotBytes) continue;
      p.used &= ~(uint64_t(1) << ((at - p.base) / kSlotBytes));
      if (p.used == 0u && spare) {
        cudaFreeHost(p.base);
        pages_.erase(pages_.begin() + static_cast<std::ptrdiff_t>(i));
      }
      return;
    }
  }

 private:
  struct Page {
    unsigned char* base;
    uint64_t used;
  };
  std::mutex mutex_;
  std::vector<Page> pages_;
};

// The process's slots; never destroyed, since handles may outlive static objects.
inline PinnedSlots& pinned_slots() {
  static PinnedSlots* slots = new PinnedSlots();
  return *slots;
}

}  // namespace isingx
