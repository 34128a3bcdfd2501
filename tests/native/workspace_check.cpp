// Host check of the library's workspaces (csrc/workspace.h) on a stand-in for
// the CUDA runtime: this file defines the runtime functions that the header
// calls.  Exit status 0 when every check holds; each failure is printed.
#include <atomic>
#include <cstdio>
#include <map>
#include <mutex>
#include <set>
#include <thread>
#include <utility>
#include <vector>

#include "../../paper_1001_4108_gb300/csrc/workspace.h"

using apsp::Workspaces;

// ---- the stand-in: memory with a limit, the last error, counts of the calls
namespace {
std::mutex mu;
std::map<void *, size_t> live;
size_t limit = 1u << 30, used = 0;
cudaError_t last_error = cudaSuccess;
std::atomic<int> syncs{0};
int freed_leased = 0;
std::set<void *> forgotten, leased;
std::map<cudaStream_t, unsigned long long> capturing;            // stream -> capture, also its graph
std::map<unsigned long long, std::vector<cudaUserObject_t>> held;  // graph -> its objects
bool refuse_objects = false;
std::atomic<int> thread_count{0}, per_thread_order{0};
std::map<cudaStream_t, int> recreated;  // how often a handle was destroyed and handed out again

cudaError_t take(void **p, size_t bytes) {
  std::lock_guard<std::mutex> lk(mu);
  if (used + bytes > limit) return last_error = cudaErrorMemoryAllocation;
  *p = ::operator new(bytes);
  live[*p] = bytes;
  used += bytes;
  return cudaSuccess;
}
cudaError_t give(void *p) {
  std::lock_guard<std::mutex> lk(mu);
  auto it = live.find(p);
  if (it == live.end()) return last_error = cudaErrorInvalidValue;
  if (leased.count(p)) ++freed_leased;
  used -= it->second;
  live.erase(it);
  ::operator delete(p);
  return cudaSuccess;
}
void forget(void *p, size_t) {
  std::lock_guard<std::mutex> lk(mu);
  forgotten.insert(p);
}
cudaStream_t stream(int i) { return reinterpret_cast<cudaStream_t>((uintptr_t)0x1000 + 16 * i); }

int fails = 0;
void check(bool ok, const char *what) {
  if (ok) return;
  std::printf("%s\n", what);
  ++fails;
}
}  // namespace

extern "C" {
cudaError_t cudaMalloc(void **p, size_t bytes) { return take(p, bytes); }
cudaError_t cudaFree(void *p) {
  ++syncs;  // waits for all work of the device
  return give(p);
}
cudaError_t cudaDeviceSynchronize() {
  ++syncs;
  return cudaSuccess;
}
cudaError_t cudaMemPoolCreate(cudaMemPool_t *pool, const cudaMemPoolProps *) {
  *pool = reinterpret_cast<cudaMemPool_t>((uintptr_t)0x10);
  return cudaSuccess;
}
cudaError_t cudaMemPoolSetAttribute(cudaMemPool_t, cudaMemPoolAttr, void *) { return cudaSuccess; }
cudaError_t cudaMallocFromPoolAsync(void **p, size_t bytes, cudaMemPool_t, cudaStream_t s) {
  if (s == cudaStreamPerThread) ++per_thread_order;
  return take(p, bytes);
}
cudaError_t cudaFreeAsync(void *p, cudaStream_t s) {
  if (s == cudaStreamPerThread) ++per_thread_order;
  return give(p);
}
cudaError_t cudaThreadExchangeStreamCaptureMode(cudaStreamCaptureMode *mode) {
  thread_local cudaStreamCaptureMode current = cudaStreamCaptureModeGlobal;
  std::swap(*mode, current);
  return cudaSuccess;
}
cudaError_t cudaStreamCreateWithFlags(cudaStream_t *s, unsigned) {
  *s = stream(99);
  return cudaSuccess;
}
cudaError_t cudaStreamSynchronize(cudaStream_t s) {
  if (s != stream(99) && s != cudaStreamPerThread) ++syncs;
  return cudaSuccess;
}
cudaError_t cudaStreamGetCaptureInfo(cudaStream_t s, cudaStreamCaptureStatus *status, unsigned long long *id,
                                     cudaGraph_t *graph, const cudaGraphNode_t **, const cudaGraphEdgeData **,
                                     size_t *) {
  std::lock_guard<std::mutex> lk(mu);
  auto it = capturing.find(s);
  *status = it == capturing.end() ? cudaStreamCaptureStatusNone : cudaStreamCaptureStatusActive;
  if (it != capturing.end()) {
    *id = it->second;
    *graph = reinterpret_cast<cudaGraph_t>((uintptr_t)it->second);
  }
  return cudaSuccess;
}
cudaError_t cudaStreamGetId(cudaStream_t s, unsigned long long *id) {
  thread_local const unsigned long long mine = 1000 + thread_count++;
  *id = s == cudaStreamPerThread ? mine : reinterpret_cast<uintptr_t>(s) + recreated[s];
  return cudaSuccess;
}
cudaError_t cudaUserObjectCreate(cudaUserObject_t *o, void *p, cudaHostFn_t destroy, unsigned, unsigned) {
  *o = reinterpret_cast<cudaUserObject_t>(new std::pair<cudaHostFn_t, void *>(destroy, p));
  return cudaSuccess;
}
cudaError_t cudaUserObjectRelease(cudaUserObject_t o, unsigned) {
  auto *x = reinterpret_cast<std::pair<cudaHostFn_t, void *> *>(o);
  x->first(x->second);
  delete x;
  return cudaSuccess;
}
cudaError_t cudaGraphRetainUserObject(cudaGraph_t g, cudaUserObject_t o, unsigned, unsigned) {
  if (refuse_objects) return last_error = cudaErrorInvalidValue;
  held[(unsigned long long)reinterpret_cast<uintptr_t>(g)].push_back(o);
  return cudaSuccess;
}
cudaError_t cudaGetLastError() {
  const cudaError_t e = last_error;
  last_error = cudaSuccess;
  return e;
}
}

static Workspaces::Lease take(Workspaces &w, int dev, cudaStream_t s, size_t bytes, size_t least) {
  apsp::Capture c;
  check(apsp::capture_of(s, &c), "a stream's capture state");
  return w.take(dev, s, c, bytes, least);
}

static void reuse_and_growth() {
  Workspaces w(forget);
  void *a = nullptr;
  {
    Workspaces::Lease l = take(w, 0, stream(1), 1000, 0);
    check(l && l.bytes == 1000, "a first buffer");
    a = l.p;
  }
  check(take(w, 0, stream(1), 500, 0).p == a, "a smaller request reuses it");
  check(take(w, 0, stream(2), 500, 0).p != a, "another stream has its own");
  check(take(w, 1, stream(1), 500, 0).p != a, "so has another device");
  check(take(w, 0, stream(1), 2000, 0).bytes == 2000, "a larger request");
  check(forgotten.count(a) == 1, "graphs that use the old buffer are dropped");
  for (int i = 3; i < 40; ++i) take(w, 0, stream(i), 1000 * i, 0);
  check(syncs == 0, "growing buffers and many streams synchronize the device");
}

// No memory: less or none, and no error stays behind.
static void out_of_memory() {
  Workspaces w(forget);
  const size_t before = limit;
  check((bool)take(w, 0, stream(1), 100, 0), "a small buffer");
  limit = used + 400;
  check(take(w, 0, stream(1), 1000, 300).bytes == 300, "no memory for a larger one: the smaller size");
  check(last_error == cudaSuccess, "a failed allocation leaves an error for the launch checks");
  check(!take(w, 0, stream(1), 2000, 1000), "no memory");
  limit = used;
  check(!take(w, 0, stream(2), 1, 0) && last_error == cudaSuccess, "no memory on a new stream");
  limit = before;
  check(take(w, 0, stream(2), 1, 0).bytes == 1, "a later call finds memory");
}

// One handle, several streams: each has its own buffer.
static void stream_identity() {
  Workspaces w(forget);
  Workspaces::Lease mine = take(w, 0, cudaStreamPerThread, 1000, 0);
  void *other = nullptr;
  std::thread([&] { other = take(w, 0, cudaStreamPerThread, 1000, 0).p; }).join();
  check(mine && other && other != mine.p, "two threads' cudaStreamPerThread share a buffer");
  mine.release();
  check(take(w, 0, cudaStreamPerThread, 5000, 0).bytes == 5000, "and can grow");
  for (int i = 0; i < 20; ++i) std::thread([&] { take(w, 0, cudaStreamPerThread, 1000, 0); }).join();
  check(per_thread_order == 0, "memory in the order of a thread's own stream");
  Workspaces v(forget);
  void *a = take(v, 0, stream(1), 1000, 0).p;
  ++recreated[stream(1)];
  check(take(v, 0, stream(1), 1000, 0).p != a, "a new stream has the buffer of a destroyed one of that handle");
}

// Threads: while one holds a lease, its buffer is neither freed nor handed to
// another, whatever the others ask for; more streams than entries.
static void threads() {
  Workspaces w(forget);
  std::atomic<int> freed{0}, shared{0}, none{0};
  auto client = [&](int t, int s) {
    for (int i = 0; i < 200; ++i) {
      Workspaces::Lease l = take(w, 0, stream(s), 100 + 37 * ((i + t) % 5) * (1 + i / 20), 0);
      if (!l) {
        ++none;
        continue;
      }
      {
        std::lock_guard<std::mutex> lk(mu);
        if (!live.count(l.p)) ++freed;
        if (!leased.insert(l.p).second) ++shared;
      }
      std::this_thread::yield();
      std::lock_guard<std::mutex> lk(mu);
      if (!live.count(l.p)) ++freed;
      leased.erase(l.p);
    }
  };
  std::vector<std::thread> th;
  for (int t = 0; t < 40; ++t) th.emplace_back(client, t, t % 20);  // 20 streams, two threads each
  for (auto &x : th) x.join();
  check(freed == 0 && freed_leased == 0, "a buffer was freed while a thread held it");
  check(shared == 0, "two threads held one buffer");
  check(none == 0, "a stream found no memory");
}

// The graph of a capture and everything made from it are destroyed.
static void destroy_graph(unsigned long long id) {
  for (auto o : held[id]) cudaUserObjectRelease(o, 1);
  held.erase(id);
}

// Streams beyond the first ones keep small buffers, and get large ones for the
// call.
static void many_streams() {
  Workspaces w(forget);
  std::vector<void *> first;
  for (int i = 0; i < 40; ++i) first.push_back(take(w, 0, stream(i), 1000, 0).p);
  for (int i = 0; i < 40; ++i) {
    Workspaces::Lease l = take(w, 0, stream(i), 1000, 0);
    check(l.p == first[i] && !l.passing(), "a stream's small buffer stays");
  }
  const size_t before = used;
  for (int i = 30; i < 50; ++i) {
    Workspaces::Lease l = take(w, 0, stream(i), 9 << 20, 0);
    check(l && l.passing(), "a large buffer beyond the first streams is for the call");
  }
  check(used == before, "and given back after it");
  check(take(w, 0, stream(30), 1000, 0).p == first[30], "beside the stream's small one");
}

// Stream captures: buffers of their own, that live as long as the graph.
static void captures() {
  Workspaces w(forget);
  forgotten.clear();
  void *own = take(w, 0, stream(1), 1000, 0).p;
  capturing[stream(1)] = 1;
  void *a = take(w, 0, stream(1), 1000, 0).p;
  check(a && a != own, "a capture does not get the stream's buffer");
  check(take(w, 0, stream(1), 800, 0).p == a, "the next solve of that capture shares its buffer");
  void *b = take(w, 0, stream(1), 3000, 0).p;
  check(b && b != a && live.count(a), "a larger one gets another, and the first stays");
  capturing[stream(2)] = 1;  // forked in the same capture: runs beside it
  void *c = take(w, 0, stream(2), 1000, 0).p;
  check(c && c != a && c != b, "two streams of one capture have their own");
  capturing.clear();
  capturing[stream(1)] = 2;
  void *d = take(w, 0, stream(1), 1000, 0).p;
  check(d && d != a && d != own, "two captures on one stream have their own");
  capturing.clear();
  check(take(w, 0, stream(1), 1000, 0).p == own, "outside the captures, the stream's own");
  for (int i = 1; i < 30; ++i) take(w, 0, stream(i), 100000, 0);
  check(!live.count(own) && live.count(a) && live.count(b) && live.count(c) && live.count(d),
        "larger solves and other streams leave the captures' buffers alone");
  check(forgotten.count(a) + forgotten.count(b) + forgotten.count(c) + forgotten.count(d) == 0,
        "the library's graphs have no part in them");
  destroy_graph(1);
  take(w, 0, stream(1), 1, 0);
  check(!live.count(a) && !live.count(b) && !live.count(c) && live.count(d), "gone with their graph");
  destroy_graph(2);
  take(w, 0, stream(1), 1, 0);
  check(!live.count(d), "and the last");
  // no memory, or a graph that takes no objects: no buffer, none left behind
  const size_t before = limit, was = used;
  capturing[stream(3)] = 3;
  limit = used;
  check(!take(w, 0, stream(3), 1000, 100), "no memory in a capture");
  limit = before;
  refuse_objects = true;
  check(!take(w, 0, stream(3), 1000, 100), "an object that the graph refuses");
  refuse_objects = false;
  check(used == was && last_error == cudaSuccess, "nothing is left of either");
  capturing.clear();
  check(syncs == 0, "captures synchronize");
}

// A server's workspaces: a request's schedule does not depend on max_n.
static void request_sizes() {
  bool enough = true;
  for (const int64_t max_n : {1, 64, 65, 512, 1984, 2048, 2496, 3328, 3329, 4096, 6000, 16384})
    for (int64_t n = 1; n <= max_n; n += n < 200 ? 1 : 61)
      for (const int dtype : {APSP_I32, APSP_F32, APSP_I16})
        for (const int S : {64, 128}) {
          const size_t have = apsp::request_workspace_bytes(max_n);
          enough = enough && have >= apsp::workspace_bytes_for(n, dtype, S) &&
                   have >= apsp::fast_workspace_bytes(n, dtype, S, false, APSP_FLAG_NO_GRAPH, false);
        }
  check(enough, "a request has less memory than its schedule needs");
}

int main() {
  request_sizes();
  reuse_and_growth();
  out_of_memory();
  captures();
  many_streams();
  stream_identity();
  threads();
  std::printf(fails ? "%d failed checks\n" : "ok\n", fails);
  return fails ? 1 : 0;
}
