// What a captured solve was captured with: launch_with_graph (api.cu) replays a
// graph only for a call that would capture the same one.
#pragma once

#include "apsp_internal.h"

namespace apsp {

// The matrix and everything the stage loops bake into their launches: which
// kernels run depends on the flags, the tile side and the size of the
// workspace as much as on the matrix.  Not compared: events (a traced call is
// never captured), the side stream (it changes the order of the launches
// only) and err (one address per device).
struct GraphKey {
  void *d;
  int64_t n, ld;
  int dtype, S, flags, dev;
  cudaStream_t stream;
  void *ws;
  size_t ws_bytes;
  void *via;
  int64_t via_ld;
  const void *first_src;
  int64_t first_src_ld;
  void *last_dst;
  int64_t last_dst_ld;
  bool operator==(const GraphKey &o) const {
    return d == o.d && n == o.n && ld == o.ld && dtype == o.dtype && S == o.S && flags == o.flags &&
           dev == o.dev && stream == o.stream && ws == o.ws && ws_bytes == o.ws_bytes && via == o.via &&
           via_ld == o.via_ld && first_src == o.first_src && first_src_ld == o.first_src_ld &&
           last_dst == o.last_dst && last_dst_ld == o.last_dst_ld;
  }
};

inline GraphKey graph_key(const RunArgs &a, int dtype, int dev) {
  return {a.d,   a.n,      a.ld,        dtype,          a.S,        a.flags,      dev, a.stream, a.ws, a.ws_bytes,
          a.via, a.via_ld, a.first_src, a.first_src_ld, a.last_dst, a.last_dst_ld};
}

}  // namespace apsp
