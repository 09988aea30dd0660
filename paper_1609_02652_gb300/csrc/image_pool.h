// Device fields that an owner keeps to save recomputing them, when there is room: kPer fields
// per entry, entries 0 .. n-1 present for some n up to what was asked for.  Host code without
// CUDA calls of its own (the allocator is a parameter).
//
// Room is a 16th of the device's memory at most, and a quarter of what is free when the entries
// are first asked for: an owner of this kind leaves three quarters of the free memory to
// whoever comes later, and what does not fit, or whose allocation fails all the same, is
// simply absent.  Each size is asked for once, so that the calls after the first one allocate
// nothing and take the same route.
#pragma once
#include <algorithm>
#include <cstddef>
#include <vector>

namespace pfmp {

struct ImagePool {
  static constexpr int kPer = 3;
  std::vector<void*> f;
  int asked = 0;

  int entries() const { return (int)f.size() / kPer; }
  void* field(int entry, int k) const { return f[(size_t)kPer * entry + k]; }
  static size_t room(size_t free_bytes, size_t total_bytes, size_t held) {
    return std::min(total_bytes / 16, held + free_bytes / 4);
  }
  // the number of entries present out of n.  mem(free, total) reports the device's memory,
  // alloc(bytes) returns null when there is none left, release(p) gives a field back
  template <class Mem, class Alloc, class Release>
  int reserve(int n, size_t field_bytes, Mem mem, Alloc alloc, Release release) {
    if (n > asked) {
      asked = n;
      size_t free_bytes = 0, total_bytes = 0;
      mem(&free_bytes, &total_bytes);
      const size_t bound = room(free_bytes, total_bytes, f.size() * field_bytes);
      while (entries() < n && (f.size() + kPer) * field_bytes <= bound) {
        const size_t before = f.size();
        f.reserve(before + kPer);  // no exception between an allocation and its place in f
        while (f.size() < before + kPer) {
          void* p = alloc(field_bytes);
          if (!p) break;
          f.push_back(p);
        }
        if (f.size() < before + kPer) {
          for (size_t i = before; i < f.size(); ++i) release(f[i]);
          f.resize(before);
          break;
        }
      }
    }
    return std::min(n, entries());
  }
};

}  // namespace pfmp
