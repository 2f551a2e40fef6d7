// Buffers that a faster path wants and a context can do without (host side):
// all of them or none, so that a context without memory for the last one
// keeps none of the others and goes on as before.
#pragma once

#include <algorithm>
#include <cstddef>
#include <initializer_list>

namespace vcsgc {

struct Wanted {
  void** p;
  size_t bytes;
};

template <typename T>
inline Wanted wanted(T** p, size_t count) {
  return {reinterpret_cast<void**>(p), sizeof(T) * std::max<size_t>(count, 1)};
}

// get(bytes): an address or null; put(address): gives it back.  On failure every
// pointer is null.
template <typename Get, typename Put>
inline bool get_all(std::initializer_list<Wanted> list, Get get, Put put) {
  bool ok = true;
  for (const Wanted& w : list) {
    *w.p = ok ? get(w.bytes) : nullptr;
    ok = ok && *w.p;
  }
  if (!ok)
    for (const Wanted& w : list) {
      if (*w.p) put(*w.p);
      *w.p = nullptr;
    }
  return ok;
}

}  // namespace vcsgc
