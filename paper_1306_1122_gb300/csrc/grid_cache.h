// grid_cache.h -- persistent grid sizes by kernel and device (host code, no CUDA calls).
#pragma once
#include <mutex>
#include <vector>

namespace dbie {

// A kernel's resident CTAs and its opt-in to more than 48 KB of shared memory belong to a device:
// an entry of one device says nothing about another.  Safe with several host threads.
class GridCache {
 public:
  // Grid size kept for (fn, dev), or 0.
  int find(const void* fn, int dev) {
    std::lock_guard<std::mutex> lk(mu_);
    for (const Entry& e : entries_)
      if (e.fn == fn && e.dev == dev) return e.grid;
    return 0;
  }
  void put(const void* fn, int dev, int grid) {
    std::lock_guard<std::mutex> lk(mu_);
    for (const Entry& e : entries_)
      if (e.fn == fn && e.dev == dev) return;
    entries_.push_back(Entry{fn, dev, grid});
  }

 private:
  struct Entry {
    const void* fn;
    int dev, grid;
  };
  std::mutex mu_;
  std::vector<Entry> entries_;
};

}  // namespace dbie
