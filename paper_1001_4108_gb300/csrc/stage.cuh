// Two launches per stage at s = 64 (Fig. 2 of Lund & Smith), any alignment
// and leading dimension.
//
// For stage b, with c = b + 1:
//   head(b)  phase 3 of stage b on row and column c, then phases 1 and 2 of
//            stage c: everything the next stage reads;
//   rest(b)  phase 3 of stage b on every tile outside rows and columns b, c,
//            and the closed diagonal tile of stage b, moved to the matrix.
// head(-1) (phases 1 and 2 of stage 0) comes first and rest(R - 1) last.
// rest(b) needs nothing of head(b): it is launched as its programmatic
// dependent, starts as soon as head(b) runs and waits for it only before it
// ends, so that the two run side by side and the end of rest(b) is the end of
// both.  head(b + 1) waits for that.
//
// Why.  Below a few thousand vertices a stage's arithmetic is microseconds and
// the solve is bound by a chain of dependent steps: phase 3 of the next
// diagonal tile, its closure, the panels.  As separate launches on two
// streams the chain cost 17 us per stage at n = 1024, most of it launch and
// join latency.  Here no step of the chain crosses launches and none but the
// first crosses CTAs: the four CTAs of a cluster share the product that
// brings the diagonal tile up to date, then each closes the tile by itself
// (the same values in each) and updates its own strips of the panels.  The
// redundant closures run on SMs that a short stage would leave idle.
//
// What keeps the CTAs of a stage independent: phase 3 of stage b reads the
// panels of stage b from the workspace (two buffers, by stage parity), never
// from the matrix, and the closed diagonal tile goes to the workspace and
// reaches the matrix with the next rest.  So within a stage a matrix element
// is read and written by one CTA only, except tile (c, c), which the heads
// only read.
//
// Values: every element sees the same rounded sums as in the other schedules
// and min is exact, so results are bit-identical to theirs.
#pragma once

#include "../../include/apsp.h"
#include "apsp_internal.h"
#include "fw_kernels.cuh"
#include "launch.cuh"

#include <algorithm>

namespace apsp {

// Panel tiles in the workspace: element (k, x) of a 64 x 64 tile, x = its
// column (row panel) or row (column panel), at [k / 2][x][k % 2]: one 128-bit
// load yields k, k + 1 of two adjacent x.  Both operands of a tile product
// have this form, so the column panel is the row panel's product with the
// roles exchanged.
constexpr int kStS = 64;                 // tile side
constexpr int kStTile = kStS * kStS;     // words of a panel tile
constexpr int kStThreads = 256;
constexpr int kStCluster = 4;            // head CTAs that share phase 3 of the diagonal tile

template <typename T>
struct StageArgs {
  using C = typename Arith<T>::C;
  T *d;              // the matrix
  const T *src;      // where phase 3 of stage b reads its tiles (d, or the host matrix in stage 0)
  T *dst;            // where it writes them (d, or the host matrix in the last stage)
  int64_t n, ld, src_ld, dst_ld;
  int R, b;
  int half;          // head CTAs per panel: h < half row panel, h < 2 half column panel, the others help with the
                     // diagonal tile only
  int heads;         // head CTAs (a multiple of the cluster); in one launch with rest, its CTAs follow
  int rest;          // rest CTAs that update a tile
  int wait_first;    // rest: no head runs beside it
  int one;           // 1 (relax2)
  C *ws;
  int16_t *via;
  int64_t via_ld;
  int *err;
  // workspace: two buffers of row and column panel, two of the closed diagonal tile
  __device__ __forceinline__ C *row_panel(int stage) const { return ws + (size_t)(stage & 1) * 2 * R * kStTile; }
  __device__ __forceinline__ C *col_panel(int stage) const { return row_panel(stage) + (size_t)R * kStTile; }
  __device__ __forceinline__ C *diag(int stage) const { return ws + ((size_t)4 * R + (stage & 1)) * kStTile; }
  // int16: the panels once more, as rest reads them: two columns per word, and
  // rows with each entry in both halves of a word
  __device__ __forceinline__ uint32_t *packed_row(int stage) const {
    return reinterpret_cast<uint32_t *>(ws + ((size_t)4 * R + 2) * kStTile) + (size_t)(stage & 1) * 3 * R * (kStTile / 2);
  }
  __device__ __forceinline__ uint32_t *packed_col(int stage) const {
    return packed_row(stage) + (size_t)R * (kStTile / 2);
  }
};

__device__ __forceinline__ void bulk_load(void *dst, const void *src, uint32_t bytes, uint64_t *bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                   smem_u32(dst)),
               "l"(reinterpret_cast<uint64_t>(src)), "r"(bytes), "r"(smem_u32(bar))
               : "memory");
}
__device__ __forceinline__ void launch_dependents() {
#if APSP_PDL
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
#endif
}
__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ void cluster_arrive() {
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
}
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
// Four words to the same shared-memory place of CTA `rank` of the cluster.
template <typename C>
__device__ __forceinline__ void cluster_store4(C *p, uint32_t rank, C v0, C v1, C v2, C v3) {
  uint32_t a;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(smem_u32(p)), "r"(rank));
  asm volatile("st.shared::cluster.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(a), "r"(__builtin_bit_cast(uint32_t, v0)),
               "r"(__builtin_bit_cast(uint32_t, v1)), "r"(__builtin_bit_cast(uint32_t, v2)),
               "r"(__builtin_bit_cast(uint32_t, v3))
               : "memory");
}

// Rows (columns) of a thread: 2 t + e and 2 t + e + 32.
__device__ __forceinline__ int st_idx(int t, int a) { return 2 * t + 32 * (a >> 1) + (a & 1); }

// y[r][x] <- min(y[r][x], min_k A(k, row r) + B(k, column x)) over the k pairs
// kp0 .. kp0 + KP - 1.  A: rows of k pairs of AS words, the thread's row pairs
// at a + 64 m (m < M); B: rows of BS words, its column pairs at b + BSTEP q
// (q < Q).
// C = uint32_t: two int16 columns per word (packed).
template <> struct Vec4<uint32_t> { using V = uint4; };
template <bool FMA>
__device__ __forceinline__ uint32_t relax2(uint32_t acc, uint32_t a0, uint32_t a1, uint32_t b0, uint32_t b1, int) {
  return __viaddmin_s16x2(a1, b1, __viaddmin_s16x2(a0, b0, acc));
}
template <typename C, int KP, int M, int Q, int AS, int BS, int BSTEP, int UN>
__device__ __forceinline__ void st_product(C (&y)[2 * M][2 * Q], const C *a, const C *b, int one, int kp0 = 0) {
  using V = typename Vec4<C>::V;
#pragma unroll UN
  for (int i = 0; i < KP; ++i) {
    const int kp = kp0 + i;
    V av[M], bv[Q];
#pragma unroll
    for (int m = 0; m < M; ++m) av[m] = *reinterpret_cast<const V *>(a + kp * AS + 64 * m);
#pragma unroll
    for (int q = 0; q < Q; ++q) bv[q] = *reinterpret_cast<const V *>(b + kp * BS + BSTEP * q);
#pragma unroll
    for (int m = 0; m < M; ++m)
#pragma unroll
      for (int q = 0; q < Q; ++q) {
        y[2 * m][2 * q] = relax2<true>(y[2 * m][2 * q], av[m].x, av[m].y, bv[q].x, bv[q].y, one);
        y[2 * m][2 * q + 1] = relax2<false>(y[2 * m][2 * q + 1], av[m].x, av[m].y, bv[q].z, bv[q].w, one);
        y[2 * m + 1][2 * q] = relax2<false>(y[2 * m + 1][2 * q], av[m].z, av[m].w, bv[q].x, bv[q].y, one);
        y[2 * m + 1][2 * q + 1] = relax2<true>(y[2 * m + 1][2 * q + 1], av[m].z, av[m].w, bv[q].z, bv[q].w, one);
      }
  }
}

// Phase 1 (Sec. 3.2): closes the tile held as 4 x 4 registers per thread, 64
// sequential k steps, eight at a time.  The eight pivot rows (and columns) go
// to shared memory; one warp brings the rows up to date step by step (row
// k + p takes part in step p as it stands after steps 0 .. p - 1; the pivot
// columns' values it needs are in its own lanes), another does the columns;
// then all threads apply the eight steps to their elements, in any order:
// each candidate is the sum the step-by-step loop forms.  Seven short
// dependent steps inside a warp take the place of eight trips through shared
// memory and a CTA barrier: 156 cycles per k step, against 230 for fw_phase1
// (512 of the 1250 cycles of a group are the arithmetic of its eight steps on
// one SM, 650 the dependent steps with their round trip).  While those run,
// warps 4 to 7 do other work: beside(g), g = 0 .. 7.
// pivots: 2 x 1024 words (alternating between groups).
template <typename T, typename F>
__device__ __forceinline__ void st_close(typename Arith<T>::C (&x)[4][4], typename Arith<T>::C *pivots, int ty,
                                         int tx, int one, F &&beside) {
  using C = typename Arith<T>::C;
  using V = typename Vec4<C>::V;
  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
#pragma unroll
  for (int m = 0; m < 2; ++m) {  // pivots 32 m .. 32 m + 31
#pragma unroll 1
    for (int g = 0; g < 4; ++g) {
      const int t0 = 4 * g;  // thread rows (columns) t0 .. t0 + 3 own the pivots
      C *rr = pivots + (g & 1) * 1024, *cc = rr + 512;
      if ((ty & ~3) == t0) {
#pragma unroll
        for (int q = 0; q < 2; ++q)
          *reinterpret_cast<V *>(rr + (ty - t0) * 128 + 4 * tx + 64 * q) =
              V{x[2 * m][2 * q], x[2 * m + 1][2 * q], x[2 * m][2 * q + 1], x[2 * m + 1][2 * q + 1]};
      }
      if ((tx & ~3) == t0) {
#pragma unroll
        for (int q = 0; q < 2; ++q)
          *reinterpret_cast<V *>(cc + (tx - t0) * 128 + 4 * ty + 64 * q) =
              V{x[2 * q][2 * m], x[2 * q][2 * m + 1], x[2 * q + 1][2 * m], x[2 * q + 1][2 * m + 1]};
      }
      __syncthreads();
      if (warp < 2) {
        C *buf = warp == 0 ? rr : cc;
        C v[2][8];  // pivot q of this warp's panel at index lane + 32 h
#pragma unroll
        for (int h = 0; h < 2; ++h)
#pragma unroll
          for (int q = 0; q < 8; q += 2) {
            const C *p = buf + (q / 2) * 128 + 2 * (lane + 32 * h);
            v[h][q] = p[0];
            v[h][q + 1] = p[1];
          }
#pragma unroll
        for (int p = 0; p < 7; ++p) {
          C w[8];
#pragma unroll
          for (int q = p + 1; q < 8; ++q) w[q] = __shfl_sync(0xffffffffu, v[m][q], 8 * g + p);
#pragma unroll
          for (int q = p + 1; q < 8; ++q)
#pragma unroll
            for (int h = 0; h < 2; ++h) v[h][q] = Arith<T>::relax(v[h][q], w[q], v[h][p]);
        }
#pragma unroll
        for (int h = 0; h < 2; ++h)
#pragma unroll
          for (int q = 0; q < 8; q += 2) {
            C *p = buf + (q / 2) * 128 + 2 * (lane + 32 * h);
            p[0] = v[h][q];
            p[1] = v[h][q + 1];
          }
      } else if (warp >= 4) {
        beside(4 * m + g);
      }
      __syncthreads();
      st_product<C, 4, 2, 2, 128, 128, 64, 4>(x, cc + 4 * ty, rr + 4 * tx, one);
    }
  }
}

// Two adjacent elements, read through L2 only.
__device__ __forceinline__ void ld2cg(const float *p, float &x, float &y) {
  const float2 v = __ldcg(reinterpret_cast<const float2 *>(p));
  x = v.x;
  y = v.y;
}
__device__ __forceinline__ void ld2cg(const int32_t *p, int32_t &x, int32_t &y) {
  const int2 v = __ldcg(reinterpret_cast<const int2 *>(p));
  x = v.x;
  y = v.y;
}
__device__ __forceinline__ void ld2cg(const int16_t *p, int32_t &x, int32_t &y) {
  const short2 v = __ldcg(reinterpret_cast<const short2 *>(p));
  x = v.x;
  y = v.y;
}
template <bool VIA>
__device__ __forceinline__ void stage_rest_packed(const StageArgs<int16_t> &g, int t, uint32_t *As, uint32_t *Bs,
                                                  uint64_t *bar);

// rest(b): phase 3 of stage b on the tiles outside rows and columns b, c: CTA t
// of g.rest updates one 64 x 64 tile, 4 x 4 elements per thread; one more CTA
// (t = g.rest) moves the closed diagonal tile of stage b to the matrix.  As, Bs:
// a tile each.
// Beside a head, rest(b) waits for nothing before it reads (fw_rest).  That it
// sees what head(b - 1) and rest(b - 1) wrote: it starts only once every CTA of
// head(b) has issued launch_dependents, each after its wait_prior_grid; that
// wait returns when rest(b - 1) has completed and its writes are performed; and
// rest(b - 1) completes after head(b - 1), for which its last CTA waits.  So
// all these writes are in L2 before rest(b) starts, and panels and matrix are
// read from L2 only (bulk copies, ld.cg): an SM's L1 may hold older lines, as
// launch_dependents by itself orders no memory.
template <typename T, bool VIA>
__device__ __forceinline__ void stage_rest(const StageArgs<T> &g, int t, typename Arith<T>::C *As,
                                           typename Arith<T>::C *Bs, uint64_t *bar) {
  using C = typename Arith<T>::C;
  constexpr int S = kStS;
  const int tid = threadIdx.x, warp = tid / 32, lane = tid % 32;
  const int b = g.b, R = g.R, c = b + 1;
  const bool last = b == R - 1;
  if (t == g.rest) {
    const C *dg = g.diag(b);
    const int64_t c0 = (int64_t)b * S;
    C v[kStTile / kStThreads];
#pragma unroll
    for (int u = 0; u < kStTile / kStThreads; ++u) v[u] = __ldcg(dg + tid + kStThreads * u);
#pragma unroll
    for (int u = 0; u < kStTile / kStThreads; ++u) {
      const int e = tid + kStThreads * u;
      const int64_t i = c0 + e / S, j = c0 + e % S;
      if (i < g.n && j < g.n) g.d[i * g.ld + j] = last ? Arith<T>::finish(v[u]) : (T)v[u];
    }
  } else if constexpr (std::is_same<T, int16_t>::value) {
    stage_rest_packed<VIA>(g, t, reinterpret_cast<uint32_t *>(As), reinterpret_cast<uint32_t *>(Bs), bar);
  } else {
    // the tile rows (columns) of the launch are all but b and c, in order
    const int skip = c < R ? 2 : 1, nr = R - skip;
    const int tr = t / nr, tc = t - tr * nr;
    const int I = tr < b ? tr : tr + skip, J = tc < b ? tc : tc + skip;
    if (tid == 0) {
      mbar_arrive_expect_tx(bar, 2 * kStTile * sizeof(C));
      bulk_load(As, g.col_panel(b) + (size_t)I * kStTile, kStTile * sizeof(C), bar);
      bulk_load(Bs, g.row_panel(b) + (size_t)J * kStTile, kStTile * sizeof(C), bar);
    }
    const int ty = 4 * (warp / 2) + lane / 8, tx = 8 * (warp % 2) + lane % 8;
    const int64_t i0 = (int64_t)I * S + 2 * ty, j0 = (int64_t)J * S + 2 * tx;
    const bool whole = (int64_t)(I + 1) * S <= g.n && (int64_t)(J + 1) * S <= g.n;
    // whole tiles and rows that allow two elements per access
    const bool pair_in = whole && reinterpret_cast<uintptr_t>(g.src) % (2 * sizeof(T)) == 0 && g.src_ld % 2 == 0;
    const bool pair_out = whole && reinterpret_cast<uintptr_t>(g.dst) % (2 * sizeof(T)) == 0 && g.dst_ld % 2 == 0;
    C x[4][4];
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
      for (int e = 0; e < 4; e += 2) {
        const int64_t i = i0 + st_idx(0, a), j = j0 + st_idx(0, e);
        const T *p = g.src + i * g.src_ld + j;
        if (pair_in) {
          ld2cg(p, x[a][e], x[a][e + 1]);
        } else {
          x[a][e] = i < g.n && j < g.n ? Arith<T>::load(__ldcg(p)) : Arith<T>::inf();
          x[a][e + 1] = i < g.n && j + 1 < g.n ? Arith<T>::load(__ldcg(p + 1)) : Arith<T>::inf();
        }
      }
    C x0[4][4];  // path bookkeeping: the values to be replaced
    if (VIA) {
#pragma unroll
      for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int e = 0; e < 4; ++e) x0[a][e] = x[a][e];
    }
    const bool late = !mbar_wait_bounded(bar, 0);
    if (!late) st_product<C, 32, 2, 2, 128, 128, 64, 2>(x, As + 4 * ty, Bs + 4 * tx, g.one);
    if (__any_sync(0xffffffffu, late)) {  // give up: wait (bounded) for the copies in flight, store nothing
      if (lane == 0) {
        atomicCAS(g.err, 0, (int)kDevTimeoutTma);
        mbar_wait_bounded(bar, 0);
      }
    } else {
#pragma unroll
      for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int e = 0; e < 4; e += 2) {
          const int64_t i = i0 + st_idx(0, a), j = j0 + st_idx(0, e);
          if (VIA && g.via && i < g.n) {
            if (j < g.n) note_via(g.via, g.via_ld, i, j, x[a][e], x0[a][e], b);
            if (j + 1 < g.n) note_via(g.via, g.via_ld, i, j + 1, x[a][e + 1], x0[a][e + 1], b);
          }
          const T v0 = last ? Arith<T>::finish(x[a][e]) : (T)x[a][e];
          const T v1 = last ? Arith<T>::finish(x[a][e + 1]) : (T)x[a][e + 1];
          T *p = g.dst + i * g.dst_ld + j;
          if (pair_out) {
            st2(p, v0, v1);
          } else if (i < g.n) {
            if (j < g.n) p[0] = v0;
            if (j + 1 < g.n) p[1] = v1;
          }
        }
    }
  }
}

// rest(b) for int16, two columns per 32-bit word (DPX viaddmin.s16x2): sums fit
// in 16 bits, signed.  Thread rows st_idx(ty, .), words 2 tx, 2 tx
// + 1 (columns 4 tx .. 4 tx + 3).
template <bool VIA>
__device__ __forceinline__ void stage_rest_packed(const StageArgs<int16_t> &g, int t, uint32_t *As, uint32_t *Bs,
                                                  uint64_t *bar) {
  constexpr int S = kStS;
  const int tid = threadIdx.x, warp = tid / 32, lane = tid % 32;
  const int b = g.b, R = g.R, c = b + 1;
  const int skip = c < R ? 2 : 1, nr = R - skip;
  const int tr = t / nr, tc = t - tr * nr;
  const int I = tr < b ? tr : tr + skip, J = tc < b ? tc : tc + skip;
  if (tid == 0) {
    mbar_arrive_expect_tx(bar, (kStTile + kStTile / 2) * 4);
    bulk_load(As, g.packed_col(b) + (size_t)I * kStTile, kStTile * 4, bar);
    bulk_load(Bs, g.packed_row(b) + (size_t)J * (kStTile / 2), kStTile / 2 * 4, bar);
  }
  const int ty = 4 * (warp / 2) + lane / 8, tx = 8 * (warp % 2) + lane % 8;
  const int64_t i0 = (int64_t)I * S + 2 * ty, j0 = (int64_t)J * S + 4 * tx;
  const bool whole = (int64_t)(I + 1) * S <= g.n && (int64_t)(J + 1) * S <= g.n;
  // whole tiles and rows that allow four columns per access
  const bool quad = whole && reinterpret_cast<uintptr_t>(g.d) % 8 == 0 && g.ld % 4 == 0;
  uint32_t x[4][2], x0[4][2];
#pragma unroll
  for (int a = 0; a < 4; ++a) {
    const int64_t i = i0 + st_idx(0, a);
    const int16_t *p = g.d + i * g.ld + j0;
    if (quad) {
      const uint2 v = __ldcg(reinterpret_cast<const uint2 *>(p));
      x[a][0] = v.x;
      x[a][1] = v.y;
    } else {
#pragma unroll
      for (int w = 0; w < 2; ++w) {
        const uint32_t lo = i < g.n && j0 + 2 * w < g.n ? (uint16_t)__ldcg(p + 2 * w) : 16383u;
        const uint32_t hi = i < g.n && j0 + 2 * w + 1 < g.n ? (uint16_t)__ldcg(p + 2 * w + 1) : 16383u;
        x[a][w] = lo | (hi << 16);
      }
    }
  }
  if (VIA) {
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
      for (int w = 0; w < 2; ++w) x0[a][w] = x[a][w];
  }
  const bool late = !mbar_wait_bounded(bar, 0);
  if (!late) st_product<uint32_t, 32, 2, 1, 128, 64, 0, 4>(x, As + 4 * ty, Bs + 4 * tx, g.one);
  if (__any_sync(0xffffffffu, late)) {  // give up: wait (bounded) for the copies in flight, store nothing
    if (lane == 0) {
      atomicCAS(g.err, 0, (int)kDevTimeoutTma);
      mbar_wait_bounded(bar, 0);
    }
    return;
  }
#pragma unroll
  for (int a = 0; a < 4; ++a) {
    const int64_t i = i0 + st_idx(0, a);
    int16_t *p = g.d + i * g.ld + j0;
    if (quad) *reinterpret_cast<uint2 *>(p) = make_uint2(x[a][0], x[a][1]);
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const int16_t v = (int16_t)(x[a][e / 2] >> (16 * (e % 2)) & 0xffffu);
      if (i < g.n && j0 + e < g.n) {
        if (VIA && g.via)
          note_via(g.via, g.via_ld, i, j0 + e, (int)v, (int)(int16_t)(x0[a][e / 2] >> (16 * (e % 2)) & 0xffffu), b);
        if (!quad) p[e] = v;
      }
    }
  }
}

// Shared memory of a head CTA whose strips are W columns (rows) wide.
template <typename C, int W>
struct HeadSmem {
  C a[kStTile];             // column panel tile (c, b)
  C b[kStTile];             // row panel tile (b, c)
  C form[kStTile];          // the closed diagonal tile as an operand
  C tile[kStTile];          // the diagonal tile after stage b, [row / 2][column][row % 2]
  C op[kStS * W];           // stage b's panel strip, [k / 2][W][2]
  C strip[kStS * W];        // the strip after stage b
  C pivots[2048];           // closure
};

template <typename T, int W, bool VIA>
__global__ void __launch_bounds__(kStThreads) __cluster_dims__(kStCluster, 1, 1) fw_head(const StageArgs<T> g) {
  using C = typename Arith<T>::C;
  using V = typename Vec4<C>::V;
  constexpr int S = kStS, Q = W / 16, kUnits = S / W;
  extern __shared__ unsigned char smem_raw[];
  HeadSmem<C, W> &sm = *reinterpret_cast<HeadSmem<C, W> *>(
      reinterpret_cast<unsigned char *>((reinterpret_cast<uintptr_t>(smem_raw) + 127) & ~uintptr_t(127)));
  __shared__ __align__(8) uint64_t bar;
  const int tid = threadIdx.x, warp = tid / 32, lane = tid % 32;
  if (tid == 0) {
    mbar_init(&bar, 1);
    fence_mbar_init();
  }
  __syncthreads();
  wait_prior_grid();
  launch_dependents();

  const int b = g.b, c = b + 1, R = g.R, h = blockIdx.x;
  if (h >= g.heads) {  // rest(b) in the same launch
    if (h - g.heads <= g.rest) stage_rest<T, VIA>(g, h - g.heads, sm.a, sm.b, &bar);
    return;
  }
  const bool cross = b >= 0;
  if (cross) cluster_arrive();
  const bool lead = h == 0;           // writes the closed tile to the workspace
  const bool cols = h >= g.half;      // this CTA's strips: of the column panel, else of the row panel
  const int u = cols ? h - g.half : h;
  const bool has = h < 2 * g.half && u < kUnits * (R - 1);  // else only helps with the diagonal tile
  const int J = skip_pivot(u / kUnits, c);                  // the strip's tile and first column (row)
  const int64_t c0 = (int64_t)c * S, x0 = (int64_t)J * S + W * (u % kUnits);
  const bool upd = has && cross && J != b;  // tile b of panel c was a panel tile of stage b: no phase 3
  if (cross && tid == 0) {
    mbar_arrive_expect_tx(&bar, 2 * kStTile * sizeof(C));
    bulk_load(sm.a, g.col_panel(b) + (size_t)c * kStTile, kStTile * sizeof(C), &bar);
    bulk_load(sm.b, g.row_panel(b) + (size_t)c * kStTile, kStTile * sizeof(C), &bar);
  }

  // ---- the strip: element (k, x), k = the index within the k-block, x = the
  // column (row panel) or row (column panel).  Phase 3 of stage b on it: warps
  // 4 to 7, rows st_idx(sy, .), columns 2 sx + 16 q + f.
  const bool helps = warp >= 4;
  const int sy = 4 * (warp & 3) + lane / 8, sx = lane % 8;
  C y[4][2 * Q];
  if (has && helps) {
    const T *p = upd ? g.src : g.d;
    const int64_t pld = upd ? g.src_ld : g.ld;
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
      for (int f = 0; f < 2 * Q; ++f) {
        const int64_t k = c0 + st_idx(sy, a), x = x0 + 2 * sx + 16 * (f >> 1) + (f & 1);
        y[a][f] = k < g.n && x < g.n ? Arith<T>::load(cols ? p[x * pld + k] : p[k * pld + x]) : Arith<T>::inf();
      }
  }
  if (upd) {  // stage b's panel strip
    const C *p = (cols ? g.col_panel(b) : g.row_panel(b)) + (size_t)J * kStTile + 2 * W * (u % kUnits);
#pragma unroll
    for (int i = 0; i < Q; ++i) {
      const int e = tid + kStThreads * i, kp = e / (W / 2), at = 4 * (e % (W / 2));
      *reinterpret_cast<V *>(sm.op + kp * 2 * W + at) = *reinterpret_cast<const V *>(p + kp * 128 + at);
    }
  }

  // ---- phase 3 of stage b on the diagonal tile: 16 rows per CTA of the
  // cluster, sent to all four
  const T *tsrc = cross ? g.src : g.d;  // stage 0's panels are in the matrix
  const int64_t tld = cross ? g.src_ld : g.ld;
  const int ty = 4 * (warp / 2) + lane / 8, tx = 8 * (warp % 2) + lane % 8;
  C x[4][4];
  bool late = false;
  if (cross) {
    const int r0 = 16 * (int)cluster_rank() + 2 * warp;  // rows r0, r0 + 1; columns 2 lane, 2 lane + 1
    C t[2][2];
#pragma unroll
    for (int e = 0; e < 2; ++e)
#pragma unroll
      for (int f = 0; f < 2; ++f) {
        const int64_t i = c0 + r0 + e, j = c0 + 2 * lane + f;
        t[e][f] = i < g.n && j < g.n ? Arith<T>::load(tsrc[i * tld + j]) : Arith<T>::inf();
      }
    late = !mbar_wait_bounded(&bar, 0);
    if (!late) st_product<C, 32, 1, 1, 128, 128, 64, 8>(t, sm.a + 2 * r0, sm.b + 4 * lane, g.one);
    cluster_wait();  // the other CTAs have started: their shared memory can be written
#pragma unroll
    for (int r = 0; r < kStCluster; ++r)
      cluster_store4<C>(sm.tile + r0 * S + 4 * lane, r, t[0][0], t[1][0], t[0][1], t[1][1]);
    cluster_arrive();
    cluster_wait();
#pragma unroll
    for (int m = 0; m < 2; ++m)
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        const V v = *reinterpret_cast<const V *>(sm.tile + (ty + 16 * m) * 128 + 4 * tx + 64 * q);
        x[2 * m][2 * q] = v.x;
        x[2 * m + 1][2 * q] = v.y;
        x[2 * m][2 * q + 1] = v.z;
        x[2 * m + 1][2 * q + 1] = v.w;
      }
  } else {
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const int64_t i = c0 + st_idx(ty, a), j = c0 + st_idx(tx, e);
        x[a][e] = i < g.n && j < g.n ? Arith<T>::load(tsrc[i * tld + j]) : Arith<T>::inf();
      }
  }
  if (__syncthreads_or(late)) {
    if (tid == 0) {
      atomicCAS(g.err, 0, (int)kDevTimeoutTma);
      mbar_wait_bounded(&bar, 0);
    }
    return;
  }
  if (!lead && !has) return;
  // path bookkeeping of the diagonal tile
  C before[4][4];
  if (VIA && g.via && lead) {
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const int64_t i = c0 + st_idx(ty, a), j = c0 + st_idx(tx, e);
        before[a][e] = x[a][e];
        if (cross && i < g.n && j < g.n)
          note_via(g.via, g.via_ld, i, j, x[a][e], Arith<T>::load(tsrc[i * tld + j]), b);
      }
  }

  // ---- phase 1 of stage c, with phase 3 of stage b on the strip beside it
  const C *ca = cols ? sm.b : sm.a;
  st_close<T>(x, sm.pivots, ty, tx, g.one, [&](int k) {
    if (upd) st_product<C, 4, 2, Q, 128, 2 * W, 32, 2>(y, ca + 4 * sy, sm.op + 4 * sx, g.one, 4 * k);
  });
  if (lead) {
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const int64_t i = c0 + st_idx(ty, a), j = c0 + st_idx(tx, e);
        if (VIA && g.via && i < g.n && j < g.n) note_via(g.via, g.via_ld, i, j, x[a][e], before[a][e], c);
      }
  }
  // the closed tile as an operand: D(i, k) for row panel strips, D(k, j) for column panel strips
#pragma unroll
  for (int m = 0; m < 2; ++m)
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      if (cols)
        *reinterpret_cast<V *>(sm.form + (ty + 16 * m) * 128 + 4 * tx + 64 * q) =
            V{x[2 * m][2 * q], x[2 * m + 1][2 * q], x[2 * m][2 * q + 1], x[2 * m + 1][2 * q + 1]};
      else
        *reinterpret_cast<V *>(sm.form + (tx + 16 * q) * 128 + 4 * ty + 64 * m) =
            V{x[2 * m][2 * q], x[2 * m][2 * q + 1], x[2 * m + 1][2 * q], x[2 * m + 1][2 * q + 1]};
    }

  if (lead) {  // here and in pairs: 4 % of an int32 n = 1024 solve against word stores before the operand's
    C *dg = g.diag(c);
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
      for (int e = 0; e < 4; e += 2) st2(dg + st_idx(ty, a) * S + st_idx(tx, e), x[a][e], x[a][e + 1]);
  }
  if (!has) return;
  if (helps) {  // the strip after stage b
    if (VIA && g.via && upd) {
#pragma unroll
      for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int f = 0; f < 2 * Q; ++f) {
          const int64_t k = c0 + st_idx(sy, a), x = x0 + 2 * sx + 16 * (f >> 1) + (f & 1);
          if (k < g.n && x < g.n)
            note_via(g.via, g.via_ld, cols ? x : k, cols ? k : x, y[a][f],
                     Arith<T>::load(cols ? g.src[x * g.src_ld + k] : g.src[k * g.src_ld + x]), b);
        }
    }
#pragma unroll
    for (int m = 0; m < 2; ++m)
#pragma unroll
      for (int q = 0; q < Q; ++q)
        *reinterpret_cast<V *>(sm.strip + (sy + 16 * m) * 2 * W + 4 * sx + 32 * q) =
            V{y[2 * m][2 * q], y[2 * m + 1][2 * q], y[2 * m][2 * q + 1], y[2 * m + 1][2 * q + 1]};
  }
  __syncthreads();

  // ---- phase 2 of stage c on the strip: rows 2 ry + e, columns 2 sx + 16 q + f
  const int ry = 4 * warp + lane / 8;
  C *out = (cols ? g.col_panel(c) : g.row_panel(c)) + (size_t)J * kStTile + 2 * W * (u % kUnits);
  const bool last = c == R - 1;
  C z[2][2 * Q], o[2][2 * Q];
#pragma unroll
  for (int q = 0; q < Q; ++q) {
    const V v = *reinterpret_cast<const V *>(sm.strip + ry * 2 * W + 4 * sx + 32 * q);
    z[0][2 * q] = v.x;
    z[1][2 * q] = v.y;
    z[0][2 * q + 1] = v.z;
    z[1][2 * q + 1] = v.w;
#pragma unroll
    for (int e = 0; e < 4; ++e) o[e & 1][2 * q + (e >> 1)] = z[e & 1][2 * q + (e >> 1)];
  }
  st_product<C, 32, 1, Q, 128, 2 * W, 32, Q == 1 ? 8 : 4>(z, sm.form + 4 * ry, sm.strip + 4 * sx, g.one);
#pragma unroll
  for (int q = 0; q < Q; ++q)
    *reinterpret_cast<V *>(out + ry * 128 + 4 * sx + 32 * q) =
        V{z[0][2 * q], z[1][2 * q], z[0][2 * q + 1], z[1][2 * q + 1]};
  if constexpr (std::is_same<T, int16_t>::value) {
    const int xs = W * (u % kUnits);
#pragma unroll
    for (int q = 0; q < Q; ++q) {
      uint32_t v[4];  // (e, f) = (0, 0), (1, 0), (0, 1), (1, 1)
#pragma unroll
      for (int i = 0; i < 4; ++i) v[i] = (uint32_t)z[i & 1][2 * q + (i >> 1)] & 0xffffu;
      if (cols)
        *reinterpret_cast<uint4 *>(g.packed_col(c) + (size_t)J * kStTile + ry * 128 + 2 * xs + 4 * sx + 32 * q) =
            make_uint4(v[0] * 0x10001u, v[1] * 0x10001u, v[2] * 0x10001u, v[3] * 0x10001u);
      else
        *reinterpret_cast<uint2 *>(g.packed_row(c) + (size_t)J * (kStTile / 2) + ry * 64 + xs + 2 * sx + 16 * q) =
            make_uint2(v[0] | v[2] << 16, v[1] | v[3] << 16);
    }
  }
#pragma unroll
  for (int e = 0; e < 2; ++e)
#pragma unroll
    for (int f = 0; f < 2 * Q; ++f) {
      const int64_t k = c0 + 2 * ry + e, xx = x0 + 2 * sx + 16 * (f >> 1) + (f & 1);
      if (k < g.n && xx < g.n) {
        if (VIA && g.via) note_via(g.via, g.via_ld, cols ? xx : k, cols ? k : xx, z[e][f], o[e][f], c);
        const T t = last ? Arith<T>::finish(z[e][f]) : (T)z[e][f];
        if (cols) g.d[xx * g.ld + k] = t;
        else g.d[k * g.ld + xx] = t;
      }
    }
}

// rest(b) on its own: four CTAs per SM, so that the loads and stores of some
// run beside the arithmetic of the others; beside a head CTA two, by shared
// memory it asks for and does not use (kRestPad): the heads' chain bounds the
// stage, and with more rest CTAs on its SM a head gets too little of the ALU
// (n = 1792 int32 590 us with the pad, 667 without).
constexpr size_t kRestPad = 20 * 1024;
template <typename T, bool VIA>
__global__ void __launch_bounds__(kStThreads, VIA ? 3 : 4) fw_rest(const StageArgs<T> g) {
  using C = typename Arith<T>::C;
  __shared__ __align__(128) C As[kStTile];
  __shared__ __align__(128) C Bs[kStTile];
  __shared__ __align__(8) uint64_t bar;
  if (threadIdx.x == 0) {
    mbar_init(&bar, 1);
    fence_mbar_init();
  }
  __syncthreads();
  if (g.wait_first) wait_prior_grid();
  launch_dependents();
  stage_rest<T, VIA>(g, blockIdx.x, As, Bs, &bar);
  // one CTA waits for head(b), so that this launch ends after it
  if (!g.wait_first && blockIdx.x == gridDim.x - 1) wait_prior_grid();
}

// How a stage's head is cut, by the number of stages R: narrow strips while
// each head CTA can have an SM to itself, and one launch per stage while rest
// has a handful of tiles (with more, the next stage's heads are placed two to
// an SM).  Measured, us per solve: n = 768 int32 164 with W = 32, 173 with 16;
// n = 512 fp32 104 with 16, 111 with 32; n = 1920 int32 676 with 32, 727 with
// 64; n = 2048 int32 779 with 64, 821 with 32, fp32 with unaligned rows 885 and
// 1071, int16 676 and 594; n = 2304 int16 799 and 840.  In one launch: n = 256 53 (57
// with two), n = 512 118 (104), n = 1024 323 (227).
struct HeadCut {
  int W;        // strip width: 16, 32 or 64
  bool merged;  // rest(b) in the head's launch
};
inline HeadCut head_cut(int R, bool i16) {
  if (R <= 9) return {16, R <= 5};
  if (R <= (i16 ? 33 : 30)) return {32, false};
  return {64, false};
}

template <typename T, int W, bool VIA>
static cudaError_t launch_head(const StageArgs<T> &g, int grid, cudaStream_t st) {
  // more than half of an SM's shared memory: the next stage's heads, launched
  // while these run, must not end up two to an SM (n = 1792 int16 494 us, 586
  // without, int32 574 and 587)
  constexpr size_t smem = std::max<size_t>(sizeof(HeadSmem<typename Arith<T>::C, W>) + 128, 116 * 1024);
  static thread_local uint64_t done = 0;  // bit per device
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
  if (!(done & (1ull << dev))) {
    // one shared-memory split for both kernels, so that an SM can run them together
    const auto carve = cudaFuncAttributePreferredSharedMemoryCarveout;
    cudaError_t e =
        cudaFuncSetAttribute(fw_head<T, W, VIA>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(fw_head<T, W, VIA>, carve, cudaSharedmemCarveoutMaxShared);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(fw_rest<T, VIA>, carve, cudaSharedmemCarveoutMaxShared);
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(fw_rest<T, VIA>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kRestPad);
    if (e != cudaSuccess) return e;
    done |= 1ull << dev;
  }
  return launch(fw_head<T, W, VIA>, dim3(grid), kStThreads, smem, st, 0, g);
}

// All stages of one matrix with s = 64 and two stages or more.  ws: stage_ws_bytes bytes, 16-byte
// aligned.
template <typename T, bool VIA>
static int run_stages(const RunArgs &a) {
  constexpr int S = kStS;
  const int R = (int)((a.n + S - 1) / S);
  StageArgs<T> g{};
  g.d = static_cast<T *>(a.d);
  g.n = a.n;
  g.ld = a.ld;
  g.R = R;
  g.ws = static_cast<typename Arith<T>::C *>(a.ws);
  g.via = a.via;
  g.via_ld = a.via_ld;
  g.err = a.err;
  g.one = 1;
  const HeadCut cut = head_cut(R, std::is_same<T, int16_t>::value);
  g.half = S / cut.W * (R - 1);
  g.heads = (2 * g.half + kStCluster - 1) / kStCluster * kStCluster;
  for (int b = -1; b < R; ++b) {
    g.b = b;
    g.src = b == 0 && a.first_src ? static_cast<const T *>(a.first_src) : g.d;
    g.src_ld = b == 0 && a.first_src ? a.first_src_ld : a.ld;
    g.dst = b == R - 1 && a.last_dst ? static_cast<T *>(a.last_dst) : g.d;
    g.dst_ld = b == R - 1 && a.last_dst ? a.last_dst_ld : a.ld;
    const bool head = b + 1 < R, merged = head && b >= 0 && cut.merged;
    const int nr = R - (head ? 2 : 1);
    g.rest = nr * nr;
    g.wait_first = head ? 0 : 1;
    if (head) {
      const int grid = g.heads + (merged ? (g.rest + kStCluster) / kStCluster * kStCluster : 0);
      const cudaError_t e = cut.W == 16   ? launch_head<T, 16, VIA>(g, grid, a.stream)
                            : cut.W == 32 ? launch_head<T, 32, VIA>(g, grid, a.stream)
                                          : launch_head<T, 64, VIA>(g, grid, a.stream);
      if (e != cudaSuccess) return APSP_ECUDA;
    }
    if (b >= 0 && !merged &&
        launch(fw_rest<T, VIA>, dim3(g.rest + 1), kStThreads, kRestPad, a.stream, 0, g) != cudaSuccess)
      return APSP_ECUDA;
  }
  return cudaPeekAtLastError() == cudaSuccess ? APSP_OK : APSP_ECUDA;
}

}  // namespace apsp
