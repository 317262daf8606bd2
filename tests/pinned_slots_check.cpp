// The pinned slots (csrc/pinned_slots.h) on the host, with stand-ins for the
// CUDA calls: slots that are out never overlap, pages come and go with them, at
// most one empty page stays, and a page that a device reset took is not used again.
#include <cstdio>
#include <cstdlib>
#include <random>
#include <set>
#include <thread>

#include "pinned_slots.h"

static std::mutex mu;
static std::set<void*> pinned;  // live pages
static int pins = 0;
static bool full = false;

extern "C" {
cudaError_t cudaHostAlloc(void** p, size_t bytes, unsigned flags) {
  std::lock_guard<std::mutex> lock(mu);
  if (full) return cudaErrorMemoryAllocation;
  if (flags != cudaHostAllocPortable) std::abort();
  *p = std::malloc(bytes);
  pinned.insert(*p);
  ++pins;
  return cudaSuccess;
}
cudaError_t cudaFreeHost(void* p) {
  std::lock_guard<std::mutex> lock(mu);
  if (!pinned.erase(p)) std::abort();
  std::free(p);
  return cudaSuccess;
}
cudaError_t cudaGetLastError() { return cudaSuccess; }
cudaError_t cudaPointerGetAttributes(cudaPointerAttributes* attr, const void* p) {
  std::lock_guard<std::mutex> lock(mu);
  attr->type = pinned.count(const_cast<void*>(p)) ? cudaMemoryTypeHost : cudaMemoryTypeUnregistered;
  return cudaSuccess;
}
}

#define CHECK(x)                                    \
  do {                                              \
    if (!(x)) {                                     \
      std::printf("line %d: %s\n", __LINE__, #x);   \
      return 1;                                     \
    }                                               \
  } while (0)

int main() {
  isingx::PinnedSlots slots;
  std::mt19937 rng(1);
  std::set<void*> out;
  for (int step = 0; step < 20000; ++step) {
    const size_t want = (step / 1000) % 2 ? 10 : 300;
    if (out.size() < want) {
      void* p = slots.take();
      CHECK(p != nullptr && out.insert(p).second && reinterpret_cast<uintptr_t>(p) % 16 == 0);
      *static_cast<char*>(p) = 1, static_cast<char*>(p)[isingx::PinnedSlots::kSlotBytes - 1] = 1;
    } else {
      auto it = out.begin();
      std::advance(it, rng() % out.size());
      slots.give(*it);
      out.erase(it);
    }
    CHECK(out.empty() || pinned.size() >= (out.size() + 63) / 64);
  }
  for (void* p : out) slots.give(p);
  CHECK(pinned.size() == 1);
  out.clear();
  const int before = pins;
  for (int i = 0; i < 100; ++i) slots.give(slots.take());
  CHECK(pins == before);  // one handle after another: the page stays
  // without room for another page
  full = true;
  for (int i = 0; i < 64; ++i) out.insert(slots.take());
  CHECK(out.size() == 64 && !out.count(nullptr) && slots.take() == nullptr);
  full = false;
  for (void* p : out) slots.give(p);
  // a device reset takes the pages; what handles of before give back is ignored
  void* old = slots.take();
  void* page = *pinned.begin();
  pinned.clear();
  void* now = slots.take();
  CHECK(now != nullptr && pinned.size() == 1 && pinned.count(now));
  slots.give(old);
  CHECK(pinned.size() == 1);
  slots.give(now);
  std::free(page);
  // several threads
  std::thread threads[4];
  bool ok[4];
  for (int t = 0; t < 4; ++t)
    threads[t] = std::thread([&, t] {
      ok[t] = true;
      for (int i = 0; i < 2000; ++i) {
        int* a = static_cast<int*>(slots.take());
        int* b = static_cast<int*>(slots.take());
        *a = t, *b = t + 100;
        std::this_thread::yield();
        ok[t] = ok[t] && *a == t && *b == t + 100;
        slots.give(a);
        slots.give(b);
      }
    });
  for (auto& t : threads) t.join();
  CHECK(ok[0] && ok[1] && ok[2] && ok[3] && pinned.size() == 1);
  return 0;
}
