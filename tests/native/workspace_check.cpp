// Host check of the library's workspaces (csrc/workspace.h) on a stand-in for
// the CUDA runtime: this file defines the runtime functions that the header
// calls.  Exit status 0 when every check holds; each failure is printed.
#include <cstdio>
#include <map>
#include <mutex>
#include <set>

#include "../../paper_1001_4108_gb300/csrc/workspace.h"

using apsp::Workspaces;

// ---- the stand-in: memory with a limit, the last error, counts of the calls
namespace {
std::mutex mu;
std::map<void *, size_t> live;
size_t limit = 1u << 30, used = 0;
cudaError_t last_error = cudaSuccess;
int syncs = 0;
std::set<void *> forgotten;

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
  used -= it->second;
  live.erase(it);
  ::operator delete(p);
  return cudaSuccess;
}
void forget(void *p) { forgotten.insert(p); }
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
cudaError_t cudaFree(void *p) { return give(p); }
cudaError_t cudaDeviceSynchronize() {
  ++syncs;
  return cudaSuccess;
}
cudaError_t cudaGetLastError() {
  const cudaError_t e = last_error;
  last_error = cudaSuccess;
  return e;
}
}

static void reuse_and_growth() {
  Workspaces w(forget);
  size_t got = 0;
  void *a = w.get(0, stream(1), 1000, false, &got);
  check(a && got == 1000, "a first buffer");
  check(w.get(0, stream(1), 500, false, &got) == a && got == 1000, "a smaller request reuses it");
  check(w.get(0, stream(2), 500, false, &got) != a, "another stream has its own");
  void *b = w.get(0, stream(1), 2000, false, &got);
  check(b && got == 2000, "a larger request");
  check(forgotten.count(a) == 1, "graphs that use the old buffer are dropped");
}

// No memory: nullptr, the caller may ask for less, and no error stays behind.
static void out_of_memory() {
  Workspaces w(forget);
  size_t got = 0;
  const size_t before = limit;
  check(w.get(0, stream(1), 100, false, &got) != nullptr, "a small buffer");
  limit = used + 400;
  check(w.get(0, stream(1), 1000, false, &got) == nullptr, "no memory for a larger one");
  check(last_error == cudaSuccess, "a failed allocation leaves an error for the launch checks");
  check(w.get(0, stream(1), 300, false, &got) != nullptr && got == 300, "a smaller one is to be had");
  limit = used;
  check(w.get(0, stream(2), 1, false, &got) == nullptr && last_error == cudaSuccess, "no memory on a new stream");
  limit = before;
  check(w.get(0, stream(2), 1, false, &got) != nullptr && got == 1, "a later call finds memory");
}

int main() {
  reuse_and_growth();
  out_of_memory();
  std::printf(fails ? "%d failed checks\n" : "ok\n", fails);
  return fails ? 1 : 0;
}
