// Host check of the graph cache's key: two solves that differ in one thing the
// captured launches depend on never share a graph.  Exit status 0 when every
// check holds; each failure is printed.
#include <cstdio>

#include "../../paper_1001_4108_gb300/csrc/graph_key.h"

using apsp::graph_key;
using apsp::RunArgs;

static int fails = 0;

template <typename F>
static void differs(const char *what, F &&change) {
  char mem[64];
  RunArgs a{};
  a.d = mem;
  a.n = 1024;
  a.ld = 1024;
  a.S = 64;
  a.ws = mem + 16;
  a.ws_bytes = 66u << 14;  // 4 R + 2 tiles of 16 KiB
  a.first_src = mem + 32;
  a.first_src_ld = 1024;
  a.last_dst = mem + 32;
  a.last_dst_ld = 1024;
  RunArgs b = a;
  if (!(graph_key(a, APSP_I32, 0) == graph_key(b, APSP_I32, 0))) {
    std::printf("%s: equal solves have different keys\n", what);
    ++fails;
  }
  change(b);
  if (graph_key(a, APSP_I32, 0) == graph_key(b, APSP_I32, 0)) {
    std::printf("%s is not in the key\n", what);
    ++fails;
  }
}

int main() {
  differs("the workspace's size", [](RunArgs &b) { b.ws_bytes = 0; });
  differs("the host matrix's leading dimension (in)", [](RunArgs &b) { b.first_src_ld += 64; });
  differs("the host matrix's leading dimension (out)", [](RunArgs &b) { b.last_dst_ld += 64; });
  std::printf(fails ? "%d failed checks\n" : "ok\n", fails);
  return fails ? 1 : 0;
}
