// A host copy of a device array, made on first need and kept.
#pragma once

#include <cstddef>
#include <mutex>
#include <new>
#include <vector>

#include "../../include/gramsci_gb300.h"

namespace gs {

// *out = kept.data() with `count` entries, which fetch(dst) brings in when they
// are not there yet. fetch returns a status; what a failed fetch left behind is
// not kept: the caller gets the status, the next call fetches again.
template <class T, class Fetch>
int host_copy(std::mutex& mu, std::vector<T>& kept, size_t count, Fetch&& fetch, const T** out) {
  std::lock_guard<std::mutex> lock(mu);
  if (kept.size() != count) {
    try {
      std::vector<T> v(count);
      const int st = fetch(v.data());
      if (st) return st;
      kept.swap(v);
    } catch (const std::bad_alloc&) {
      return GS_ENOMEM;
    }
  }
  *out = kept.data();
  return GS_OK;
}

}  // namespace gs
