// Scratch memory that the library owns: one buffer per (device, stream), since
// work on one stream is ordered and a stream's solves can share one.  Host code
// only.
#pragma once

#include <cstddef>
#include <mutex>
#include <vector>

#include "apsp_internal.h"

namespace apsp {

class Workspaces {
 public:
  // forget(p): called before the buffer p is freed
  explicit Workspaces(void (*forget)(void *)) : forget_(forget) {}

  // At least `bytes` bytes for work on `stream` (*got of them), or nullptr if
  // there is no memory (the caller then runs kernels that need less or none) or
  // the stream is being captured and has no buffer of that size yet.
  void *get(int dev, cudaStream_t stream, size_t bytes, bool capturing, size_t *got) {
    std::lock_guard<std::mutex> lk(mu_);
    for (size_t i = 0; i < entries_.size(); ++i) {
      Entry &e = entries_[i];
      if (e.dev != dev || e.stream != stream) continue;
      if (e.bytes >= bytes) {
        *got = e.bytes;
        return e.p;
      }
      if (capturing) return nullptr;
      drop(i);
      break;
    }
    if (capturing) return nullptr;
    if (entries_.size() >= kMaxEntries) drop(0);
    void *p = nullptr;
    if (!got_memory(cudaMalloc(&p, bytes))) return nullptr;
    entries_.push_back({dev, stream, p, bytes});
    *got = bytes;
    return p;
  }

 private:
  struct Entry {
    int dev;
    cudaStream_t stream;
    void *p;
    size_t bytes;
  };
  static constexpr size_t kMaxEntries = 16;
  void drop(size_t i) {
    cudaDeviceSynchronize();
    forget_(entries_[i].p);
    cudaFree(entries_[i].p);
    entries_.erase(entries_.begin() + i);
  }
  void (*forget_)(void *);
  std::mutex mu_;
  std::vector<Entry> entries_;
};

}  // namespace apsp
