// Scratch memory that the library owns: one buffer per (device, stream), since
// work on one stream is ordered and a stream's solves can share one.  Host code
// only.
#pragma once

#include <cstddef>
#include <memory>
#include <mutex>
#include <utility>
#include <vector>

#include "apsp_internal.h"

namespace apsp {

// Device memory in stream order, from one pool per device.  Memory above
// `keep` bytes goes back to the device when nothing uses it.
class StreamPool {
 public:
  explicit StreamPool(uint64_t keep) : keep_(keep) {}
  void *alloc(int dev, size_t bytes, cudaStream_t stream) {
    const cudaMemPool_t pool = of(dev);
    void *p = nullptr;
    return pool && got_memory(cudaMallocFromPoolAsync(&p, bytes, pool, stream)) ? p : nullptr;
  }

 private:
  static constexpr int kMaxDev = 64;
  cudaMemPool_t of(int dev) {
    std::lock_guard<std::mutex> lk(mu_);
    if (!pool_[dev]) {
      cudaMemPoolProps props{};
      props.allocType = cudaMemAllocationTypePinned;
      props.location.type = cudaMemLocationTypeDevice;
      props.location.id = dev;
      cudaMemPool_t pool = nullptr;
      if (!got_memory(cudaMemPoolCreate(&pool, &props)) ||
          !got_memory(cudaMemPoolSetAttribute(pool, cudaMemPoolAttrReleaseThreshold, &keep_)))
        return nullptr;
      pool_[dev] = pool;
    }
    return pool_[dev];
  }
  uint64_t keep_;
  std::mutex mu_;
  cudaMemPool_t pool_[kMaxDev] = {};
};

class Workspaces {
  struct Entry {
    int dev;
    cudaStream_t stream;
    std::mutex mu;  // held from take() until the work that uses the buffer is enqueued
    void *p = nullptr;
    size_t bytes = 0;
  };

 public:
  // A buffer for the work that its holder enqueues before it lets go: until
  // then no other thread gets, frees or replaces the buffer of that stream.
  class Lease {
   public:
    Lease() = default;
    Lease(Lease &&o) noexcept
        : p(std::exchange(o.p, nullptr)),
          bytes(std::exchange(o.bytes, 0)),
          entry_(std::move(o.entry_)),
          lk_(std::move(o.lk_)),
          stream_(o.stream_) {}
    Lease &operator=(Lease &&o) noexcept {
      release();
      p = std::exchange(o.p, nullptr);
      bytes = std::exchange(o.bytes, 0);
      entry_ = std::move(o.entry_);
      lk_ = std::move(o.lk_);
      stream_ = o.stream_;
      return *this;
    }
    ~Lease() { release(); }
    void release() {
      if (p && !entry_) cudaFreeAsync(p, stream_);
      p = nullptr;
      bytes = 0;
      if (lk_.owns_lock()) lk_.unlock();
      entry_.reset();
    }
    explicit operator bool() const { return p != nullptr; }
    void *p = nullptr;
    size_t bytes = 0;

   private:
    friend class Workspaces;
    std::shared_ptr<Entry> entry_;  // empty: the buffer is this lease's alone
    std::unique_lock<std::mutex> lk_;
    cudaStream_t stream_ = nullptr;
  };

  // forget(p, bytes): called before that buffer is freed
  explicit Workspaces(void (*forget)(void *, size_t)) : forget_(forget) {}

  // At least `bytes` bytes for work on `stream`, else at least `least` (if not
  // 0), else an empty lease: there is no memory, or the stream is being
  // captured and has no buffer of that size yet.  The caller then runs kernels
  // that need less or none.
  Lease take(int dev, cudaStream_t stream, size_t bytes, size_t least, bool capturing) {
    Lease l;
    l.stream_ = stream;
    if (const std::shared_ptr<Entry> e = entry(dev, stream, !capturing)) {
      l.lk_ = std::unique_lock<std::mutex>(e->mu);
      if (e->bytes < bytes && !capturing) {
        // in stream order: all work that uses the buffer is on this stream
        if (e->p) {
          forget_(e->p, e->bytes);
          cudaFreeAsync(e->p, stream);
        }
        e->bytes = alloc(dev, stream, bytes, least, &e->p);
      }
      if (e->bytes >= bytes || (least && e->bytes >= least)) {
        l.p = e->p;
        l.bytes = e->bytes;
        l.entry_ = e;
      } else {
        l.lk_.unlock();
      }
    } else if (!capturing) {
      l.bytes = alloc(dev, stream, bytes, least, &l.p);  // more streams than entries: a buffer for this call
    }
    return l;
  }

 private:
  static constexpr size_t kMaxEntries = 16;
  // Entries are never evicted: another stream's work may be using the buffer.
  std::shared_ptr<Entry> entry(int dev, cudaStream_t stream, bool create) {
    std::lock_guard<std::mutex> lk(mu_);
    for (auto &e : entries_)
      if (e->dev == dev && e->stream == stream) return e;
    if (!create || entries_.size() >= kMaxEntries) return nullptr;
    auto e = std::make_shared<Entry>();
    e->dev = dev;
    e->stream = stream;
    entries_.push_back(e);
    return e;
  }
  // `bytes` or else `least` bytes in *p; the size, 0 (*p = nullptr) without memory
  size_t alloc(int dev, cudaStream_t stream, size_t bytes, size_t least, void **p) {
    for (const size_t want : {bytes, least})
      if (want && (*p = pool_.alloc(dev, want, stream))) return want;
    *p = nullptr;
    return 0;
  }
  void (*forget_)(void *, size_t);
  std::mutex mu_;
  std::vector<std::shared_ptr<Entry>> entries_;
  StreamPool pool_{64ull << 20};
};

}  // namespace apsp
