// Host-side facts that hold for one CUDA context only: attributes set on kernels, co-resident blocks, SM
// counts, memory pools, pinned words. A process has a context per device, and cudaDeviceReset ends one and
// starts another on the same device, so such facts are kept by the context's id, which is never reused.
#pragma once

#include <stdint.h>

#include <map>
#include <mutex>

namespace fpeps {

uint64_t context_id();   // of the calling thread's current context; the device's, made current, if there is none

// One T (a small value) per context, made on its first use there. Safe with several threads; make() may
// throw and is then called again by the next use.
template <class T>
class PerContext {
 public:
  template <class Make>
  T get(Make&& make, uint64_t id = context_id()) {
    std::lock_guard<std::mutex> lk(mu_);
    auto it = made_.find(id);
    if (it == made_.end()) it = made_.emplace(id, make()).first;
    return it->second;
  }
  // the current context's, if it has been made
  bool peek(T& out) {
    const uint64_t id = context_id();
    std::lock_guard<std::mutex> lk(mu_);
    auto it = made_.find(id);
    if (it == made_.end()) return false;
    out = it->second;
    return true;
  }

 private:
  std::mutex mu_;
  std::map<uint64_t, T> made_;
};

}  // namespace fpeps
