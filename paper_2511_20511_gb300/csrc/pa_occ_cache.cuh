// pa_occ_cache.cuh -- resident blocks per SM by (kernel, device, threads, shared
// memory), host code without CUDA calls of its own.
//
// A process that evaluates many shapes asks for many keys: a lane-per-chromosome
// kernel for each number of columns, and a shared-memory size for each shape.  The
// table grows with them (a fixed one of 256 keys, once full, had every further
// shape repeat the queries on each call: several microseconds under the lock).
#pragma once

#include <cstddef>
#include <cstdint>
#include <mutex>
#include <unordered_map>
#include <unordered_set>

namespace pa {

struct OccKey {
  const void* fn;
  int dev, threads;
  size_t smem;
  bool operator==(const OccKey& o) const {
    return fn == o.fn && dev == o.dev && threads == o.threads && smem == o.smem;
  }
};
struct OccHash {
  size_t operator()(const OccKey& k) const {
    uint64_t h = (uint64_t)reinterpret_cast<uintptr_t>(k.fn);
    for (uint64_t v : {(uint64_t)k.dev, (uint64_t)k.threads, (uint64_t)k.smem})
      h = (h ^ v) * 0x9e3779b97f4a7c15ULL;
    return (size_t)(h ^ (h >> 32));
  }
};

// prepare(): once per (kernel, device); query(&value): the value of a new key.
// Both return 0 on success; what they return otherwise is returned, and nothing is
// kept.  Safe from several threads.
class OccCache {
 public:
  template <typename Prepare, typename Query>
  int get(const OccKey& key, int* value, Prepare prepare, Query query) {
    std::lock_guard<std::mutex> lock(mu_);
    const auto it = values_.find(key);
    if (it != values_.end()) {
      *value = it->second;
      return 0;
    }
    const OccKey kernel{key.fn, key.dev, 0, 0};
    if (!prepared_.count(kernel)) {
      const int e = prepare();
      if (e) return e;
      keep([&] { prepared_.insert(kernel); });
    }
    const int e = query(value);
    if (e) return e;
    keep([&] { values_.emplace(key, *value); });
    return 0;
  }

 private:
  // a key that finds no memory is asked for again
  template <typename F>
  static void keep(F f) {
    try {
      f();
    } catch (...) {
    }
  }
  std::mutex mu_;
  std::unordered_map<OccKey, int, OccHash> values_;
  std::unordered_set<OccKey, OccHash> prepared_;
};

}  // namespace pa
