// Scratch memory that the library owns.  Host code only.
//
// Work on one stream is ordered, so a stream's solves share one buffer per
// (device, stream).  A solve in a caller's stream capture can not: its graph
// may be launched on any stream, at any time, long after the stream's buffer
// was outgrown.  Each capture has buffers of its own, which its graph (and
// whatever is instantiated, cloned or updated from it) holds as a CUDA user
// object; once the last of them is gone the memory goes back to the pool.
#pragma once

#include <algorithm>
#include <atomic>
#include <cstddef>
#include <memory>
#include <mutex>
#include <utility>
#include <vector>

#include "apsp_internal.h"

namespace apsp {

constexpr int kMaxDev = 64;

// While it lives, this thread may allocate and wait although some thread's
// stream capture forbids it: nothing here belongs to a capture.
class OutsideCapture {
 public:
  OutsideCapture() { cudaThreadExchangeStreamCaptureMode(&mode_); }
  ~OutsideCapture() { cudaThreadExchangeStreamCaptureMode(&mode_); }
  OutsideCapture(const OutsideCapture &) = delete;

 private:
  cudaStreamCaptureMode mode_ = cudaStreamCaptureModeRelaxed;
};

// Whether a stream is being captured, and into which graph (nullptr: the
// capture is invalid).
struct Capture {
  bool active = false;
  unsigned long long id = 0;
  cudaGraph_t graph = nullptr;
};
inline bool capture_of(cudaStream_t stream, Capture *c) {
  cudaStreamCaptureStatus status = cudaStreamCaptureStatusNone;
  if (cudaStreamGetCaptureInfo(stream, &status, &c->id, &c->graph, nullptr, nullptr, nullptr) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  c->active = status != cudaStreamCaptureStatusNone;
  if (status != cudaStreamCaptureStatusActive) c->graph = nullptr;
  return true;
}

// Device memory in stream order, from one pool per device.  Memory above
// `keep` bytes goes back to the device when nothing uses it.  What one stream
// freed is another's only once that work is done: a pool that made the second
// stream wait would put the two in a row.
class StreamPool {
 public:
  explicit StreamPool(uint64_t keep) : keep_(keep) {}
  void *alloc(int dev, size_t bytes, cudaStream_t stream) {
    const OutsideCapture guard;
    const cudaMemPool_t pool = of(dev);
    void *p = nullptr;
    return pool && got_memory(cudaMallocFromPoolAsync(&p, bytes, pool, stream)) ? p : nullptr;
  }

 private:
  cudaMemPool_t of(int dev) {
    std::lock_guard<std::mutex> lk(mu_);
    if (!pool_[dev]) {
      cudaMemPoolProps props{};
      props.allocType = cudaMemAllocationTypePinned;
      props.location.type = cudaMemLocationTypeDevice;
      props.location.id = dev;
      cudaMemPool_t pool = nullptr;
      int waits = 0;
      if (!got_memory(cudaMemPoolCreate(&pool, &props)) ||
          !got_memory(cudaMemPoolSetAttribute(pool, cudaMemPoolAttrReleaseThreshold, &keep_)) ||
          !got_memory(cudaMemPoolSetAttribute(pool, cudaMemPoolReuseAllowInternalDependencies, &waits)))
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
    unsigned long long id = 0;  // the stream's
    bool small = false;         // one of those for small buffers only
    std::mutex mu;              // held from take() until the work that uses the buffer is enqueued
    void *p = nullptr;
    size_t bytes = 0;
    // buffers of captures: the stream's handle, the capture whose graph holds the buffer
    cudaStream_t stream = nullptr;
    unsigned long long capture = 0;
    std::atomic<bool> unused{false};  // that graph and its offspring are gone
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
    // For this lease only: the next call may get another.
    bool passing() const { return p && !entry_; }
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

  // At least `bytes` bytes for work on `stream` (capture_of it), else at least `least` (if not
  // 0), else an empty lease: there is no memory.  The caller then runs kernels
  // that need less or none.
  // Nothing is allocated or freed in the order of cudaStreamPerThread, which
  // ends with its thread: a thread that ended with such frees pending left a
  // later device synchronize waiting.
  Lease take(int dev, cudaStream_t stream, const Capture &cap, size_t bytes, size_t least) {
    Lease l;
    l.stream_ = stream;
    give_back(dev);
    if (const std::shared_ptr<Entry> e =
            cap.active ? captured(dev, stream, cap, bytes, least) : entry(dev, stream, bytes)) {
      l.lk_ = std::unique_lock<std::mutex>(e->mu);
      if (e->bytes < bytes && !cap.active) {
        if (e->p) forget_(e->p, e->bytes);
        if (stream == cudaStreamPerThread) {
          replace_outside(e.get(), bytes, least);
        } else {  // in stream order: all work that uses the buffer is on this stream
          if (e->p) cudaFreeAsync(e->p, stream);
          e->bytes = alloc(pool_, dev, stream, bytes, least, &e->p);
        }
      }
      if (e->p && e->bytes >= (least ? std::min(bytes, least) : bytes)) {
        l.p = e->p;
        l.bytes = e->bytes;
        l.entry_ = e;
      } else {
        l.lk_.unlock();
      }
    } else if (!cap.active && stream != cudaStreamPerThread) {
      l.bytes = alloc(pool_, dev, stream, bytes, least, &l.p);  // more streams than entries: for this call
    }
    return l;
  }

 private:
  // Streams with a buffer of their own: 16, and 48 more for small buffers, the
  // ones of solves so short that an allocation and a graph captured anew show
  // (int32 n = 256 on 12 streams 7.6 us a solve; 39 where the last of them were
  // beyond the entries).
  static constexpr size_t kMaxEntries = 16, kMaxWithSmall = 64, kSmallBytes = 8u << 20;
  // By the stream's id, not its handle: every thread's cudaStreamPerThread is
  // another stream, and a destroyed stream's handle can come back while its
  // work still runs.  Entries are never evicted: another stream's work may be
  // using the buffer.
  std::shared_ptr<Entry> entry(int dev, cudaStream_t stream, size_t bytes) {
    unsigned long long id = 0;
    if (cudaStreamGetId(stream, &id) != cudaSuccess) {
      cudaGetLastError();
      return nullptr;
    }
    std::lock_guard<std::mutex> lk(mu_);
    for (auto &e : entries_)
      if (e->dev == dev && e->id == id) return e->small && bytes > kSmallBytes ? nullptr : e;
    const bool small = entries_.size() >= kMaxEntries;
    if (entries_.size() >= kMaxWithSmall || (small && bytes > kSmallBytes)) return nullptr;
    auto e = std::make_shared<Entry>();
    e->dev = dev;
    e->id = id;
    e->small = small;
    entries_.push_back(e);
    return e;
  }
  // The buffer of the solves that are captured on `stream` into `graph`, one
  // after the other; nullptr without memory.
  std::shared_ptr<Entry> captured(int dev, cudaStream_t stream, const Capture &cap, size_t bytes, size_t least) {
    if (!cap.graph) return nullptr;
    std::lock_guard<std::mutex> lk(mu_);
    for (auto &e : captured_)
      if (e->capture == cap.id && e->stream == stream && e->dev == dev && e->bytes >= bytes) return e;
    const OutsideCapture guard;
    const cudaStream_t home = home_stream(dev);
    if (!home) return nullptr;
    auto e = std::make_shared<Entry>();
    e->dev = dev;
    e->stream = stream;
    e->capture = cap.id;
    if (!(e->bytes = alloc(outside_, dev, home, bytes, least, &e->p))) return nullptr;
    auto *held = new std::shared_ptr<Entry>(e);
    cudaUserObject_t object = nullptr;
    const bool made =
        cudaUserObjectCreate(&object, held, &graph_gone, 1, cudaUserObjectNoDestructorSync) == cudaSuccess;
    if (!made) delete held;
    // the memory is there before any launch of the graph
    if (!made || cudaStreamSynchronize(home) != cudaSuccess ||
        cudaGraphRetainUserObject(cap.graph, object, 1, cudaGraphUserObjectMove) != cudaSuccess) {
      cudaGetLastError();
      if (made) cudaUserObjectRelease(object, 1);
      cudaFreeAsync(e->p, home);
      return nullptr;
    }
    captured_.push_back(e);
    return e;
  }
  // A larger buffer for a calling thread's own stream; it waits for that
  // stream's work with the old one.
  void replace_outside(Entry *e, size_t bytes, size_t least) {
    const OutsideCapture guard;
    if (e->p && cudaStreamSynchronize(cudaStreamPerThread) != cudaSuccess) return;
    std::lock_guard<std::mutex> lk(mu_);
    const cudaStream_t home = home_stream(e->dev);
    if (!home) return;
    if (e->p) cudaFreeAsync(e->p, home);
    e->bytes = alloc(outside_, e->dev, home, bytes, least, &e->p);
    cudaStreamSynchronize(home);
  }
  // Runs on a thread of the CUDA runtime when nothing refers to a capture's
  // graph any more: no CUDA calls in here.
  static void CUDART_CB graph_gone(void *held) {
    auto *e = static_cast<std::shared_ptr<Entry> *>(held);
    (*e)->unused = true;
    unused_ = true;
    delete e;
  }
  // Returns the buffers of captures that are gone to their pool.
  void give_back(int dev) {
    if (!unused_ || !unused_.exchange(false)) return;
    const OutsideCapture guard;
    std::lock_guard<std::mutex> lk(mu_);
    for (size_t i = 0; i < captured_.size();) {
      if (captured_[i]->unused && captured_[i]->dev == dev) {
        cudaFreeAsync(captured_[i]->p, home_[dev]);
        captured_.erase(captured_.begin() + i);
      } else {
        if (captured_[i]->unused) unused_ = true;  // for a call on its device
        ++i;
      }
    }
  }
  // The stream of the allocations outside_: nothing else runs on it.
  cudaStream_t home_stream(int dev) {
    if (!home_[dev] && !got_memory(cudaStreamCreateWithFlags(&home_[dev], cudaStreamNonBlocking)))
      home_[dev] = nullptr;
    return home_[dev];
  }
  // `bytes` or else `least` bytes in *p; the size, 0 (*p = nullptr) without memory
  static size_t alloc(StreamPool &pool, int dev, cudaStream_t stream, size_t bytes, size_t least, void **p) {
    for (const size_t want : {bytes, least})
      if (want && (*p = pool.alloc(dev, want, stream))) return want;
    *p = nullptr;
    return 0;
  }
  void (*forget_)(void *, size_t);
  std::mutex mu_;
  std::vector<std::shared_ptr<Entry>> entries_;
  StreamPool pool_{64ull << 20};
  std::vector<std::shared_ptr<Entry>> captured_;
  static inline std::atomic<bool> unused_{false};  // some entry of captured_ may be unused
  StreamPool outside_{64ull << 20};  // buffers that no stream's order covers
  cudaStream_t home_[kMaxDev] = {};
};

}  // namespace apsp
