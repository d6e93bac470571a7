// host_slots.h -- small slots of pinned host memory, shared out of pages.
#pragma once
#include <cstddef>
#include <cstdint>
#include <mutex>
#include <vector>

namespace dsdna {

// Slots of 64 bytes, 64 to a page of 4096.  A page comes from `get` (null when
// out of memory) when no page has a free slot and goes back to `put` with its
// last slot.  Safe with several threads.
class HostSlots {
 public:
  HostSlots(void* (*get)(), void (*put)(void*)) : get_(get), put_(put) {}

  double* take() {
    std::lock_guard<std::mutex> lock(mutex_);
    Page* page = nullptr;
    for (Page& p : pages_)
      if (~p.used) page = &p;
    if (!page) {
      Page p;
      p.mem = (char*)get_();
      if (!p.mem) return nullptr;
      pages_.push_back(p);
      page = &pages_.back();
    }
    int k = 0;
    while ((page->used >> k) & 1u) ++k;
    page->used |= 1ull << k;
    return (double*)(page->mem + 64 * k);
  }

  void give(double* slot) {
    std::lock_guard<std::mutex> lock(mutex_);
    for (size_t i = 0; i < pages_.size(); ++i) {
      Page& p = pages_[i];
      const ptrdiff_t at = (char*)slot - p.mem;
      if (at < 0 || at >= 4096) continue;
      p.used &= ~(1ull << (at / 64));
      if (!p.used) {
        put_(p.mem);
        pages_.erase(pages_.begin() + (ptrdiff_t)i);
      }
      return;
    }
  }

 private:
  struct Page {
    char* mem = nullptr;
    uint64_t used = 0;
  };
  void* (*get_)();
  void (*put_)(void*);
  std::mutex mutex_;
  std::vector<Page> pages_;
};

// The process's slots, never destroyed: contexts may be destroyed as late as by
// exit handlers and static destructors of the program.
template <void* (*get)(), void (*put)(void*)>
HostSlots& host_slots() {
  static HostSlots* s = new HostSlots(get, put);
  return *s;
}

}  // namespace dsdna
