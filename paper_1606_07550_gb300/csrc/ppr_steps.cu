// Batched personalised PageRank, step by step over the whole GPU (section 4
// Table "snap_methods" and section 4.3, "Fast Random Walk Algorithms").
//
// The other schedule of ppr_batch (ppr.cu, ppr_kernel) gives a job to one
// thread-block cluster for all of its steps: up to eight SMs, however large
// the graph and however few the jobs.  Here a job's rows are cut into items
// of one 256-thread block each, and a step of every job of a wave is one
// launch over all their items (two where a graph has long rows), so a single
// query on a large graph uses every SM.
//
// Width.  A job of k columns is stored W wide, the smallest of 1, 4, 16 and 64
// that holds k: a node's columns are W consecutive floats, and a warp reads
// 32 (W <= 16: 8 to 32 per row) edges at once instead of spending a 256-byte
// row slot on each.  Lanes hold four columns each (one when W = 1), so a
// 64-column gather is one 16-byte load per lane and two edges per load.
//
// Waves.  The jobs of a width run in waves of up to kWaveBytes of workspace, every
// job of a wave at the same step.  A launch takes its items job by job, so
// the blocks on the GPU at one time gather from few jobs, whose previous
// contributions L2 (129 MB) and, being written by an earlier launch, the L1s
// can hold.
//
// What bounds it.  64 columns, FP32, 256 batch graphs (n in [1e3, 2e5], mean
// degree 4 to 32): 268 ms for 50 steps, 8 TB/s of gathered bytes; latency-bound at
// 24 warps an SM (80 registers; 64 spill and measured 302 ms, 128 at 16 warps
// 272), DRAM 21%, L2 32-47% of peak.  On clusters (ppr.cu) the same call took
// 1,015 ms, 64 columns of one 2^20-node graph 1,420 ms (here 26 ms) and one
// column of a 100,000-node graph 90 ms (here 1.6 ms).
//
// Short rows.  Two thirds of an R-MAT graph's rows have up to eight edges and
// cost latency, not bytes: two at a time, half a warp each, took the batch
// from 300 to 270 ms.
//
// Long rows.  A warp takes a row of up to kLongDeg edges; a longer one is cut
// into chunks that a launch of its own sums first, a warp per chunk, since one
// warp would hold up the step (16 edges per 0.6 us or so: a row of 1,024 edges
// is 40 us).
//
// Order of additions.  A column's bits depend on its graph alone, not on the
// width, the other columns or the other jobs.  A row's sum, over its edges in
// order, is taken in blocks of 64 edges: edge t of a block belongs to slot
// t mod 8; a slot adds its eight edges in order; the even slots are added as
// (S0 + S2) + (S4 + S6) and the odd ones alike, to the row's running even and
// odd sums, whose sum is the row's.  A long row is the sum of its chunks, each
// taken this way, added in order by eights (the sum of eight, then one addition:
// one after another, the 157 equal chunk sums of a hub of 20,000 in-edges round
// alike, 2e-6 of the whole).  The dangling mass and the residual are FP32 sums
// over the rows of a piece (about kPieceWork units of work), 32 rows at a time,
// the short rows (up to kShortDeg edges) before the others, each in row order;
// then exact integer sums of those in units of 2^-60, in any order (a dangling
// mass can be below zero: what a row has sent as BF16 deltas passes its
// contribution by up to 2^-9 of the last delta, and where x falls to less than
// that in a step, a cycle's front passing with d above 0.998, the rows after it
// have x < 0 for one step).
//
// The server (serve.cu) runs its slots' steps on the same kernels, 64 columns
// wide.
//
// Storage of the contributions as in ppr.cu: FP32; FP16 times 2^10; BF16 as
// error-feedback deltas (X then holds the running sums y, S the sent ones).
#include <algorithm>
#include <climits>
#include <type_traits>
#include <vector>

#include <cuda_fp16.h>

#include "gpr_internal.cuh"
#include "ppr_internal.cuh"

namespace gpr {

constexpr int kStThreads = 32 * kStWarps;
constexpr int32_t kLongDeg = 128;    // a batch's longer rows are summed by chunks
constexpr int32_t kShortDeg = 8;     // rows that half a warp takes

// Edges per chunk of a row of deg edges, more than long_deg: long_deg, or about
// sqrt(2 deg), since the chunk sums of one row are added by one warp.
__host__ __device__ __forceinline__ int32_t chunk_edges(int32_t deg, int32_t long_deg) {
  int32_t c = long_deg;
  while (deg / c >= 2 * c) c *= 2;
  return c;
}

template <int W>
struct Geo {
  static constexpr int V = W >= 4 ? 4 : 1;             // columns per lane
  static constexpr int L = W / V;                      // lanes per edge
  static constexpr int G = 32 / L < 8 ? 32 / L : 8;    // edges of a row per load
  static constexpr int R = 32 / (L * G);               // rows side by side in a warp
};

constexpr float kScale16 = 1024.0f, kUnscale16 = 1.0f / 1024.0f;

// V consecutive contributions, through the read-only path (L1 and L2).
template <int V>
__device__ __forceinline__ void ld_c(const float* p, float (&v)[V]) {
  if constexpr (V == 4) {
    const float4 f = __ldg(reinterpret_cast<const float4*>(p));
    v[0] = f.x, v[1] = f.y, v[2] = f.z, v[3] = f.w;
  } else {
    v[0] = __ldg(p);
  }
}
template <int V>
__device__ __forceinline__ void ld_c(const __nv_bfloat16* p, float (&v)[V]) {
  if constexpr (V == 4) {
    const uint2 u = __ldg(reinterpret_cast<const uint2*>(p));
    v[0] = __uint_as_float(u.x << 16), v[1] = __uint_as_float(u.x & 0xFFFF0000u);
    v[2] = __uint_as_float(u.y << 16), v[3] = __uint_as_float(u.y & 0xFFFF0000u);
  } else {
    v[0] = __bfloat162float(__ldg(p));
  }
}
template <int V>
__device__ __forceinline__ void ld_c(const __half* p, float (&v)[V]) {
  if constexpr (V == 4) {
    const uint2 u = __ldg(reinterpret_cast<const uint2*>(p));
    const float2 a = __half22float2(*reinterpret_cast<const __half2*>(&u.x));
    const float2 b = __half22float2(*reinterpret_cast<const __half2*>(&u.y));
    v[0] = a.x * kUnscale16, v[1] = a.y * kUnscale16, v[2] = b.x * kUnscale16, v[3] = b.y * kUnscale16;
  } else {
    v[0] = __half2float(__ldg(p)) * kUnscale16;
  }
}
// V floats of per-row state: read once and written once per step, streaming.
template <int V>
__device__ __forceinline__ void ld_f(const float* p, float (&v)[V]) {
  if constexpr (V == 4) {
    const float4 f = __ldcs(reinterpret_cast<const float4*>(p));
    v[0] = f.x, v[1] = f.y, v[2] = f.z, v[3] = f.w;
  } else {
    v[0] = __ldcs(p);
  }
}
template <int V>
__device__ __forceinline__ void st_f(float* p, const float (&v)[V]) {
  if constexpr (V == 4)
    __stcs(reinterpret_cast<float4*>(p), make_float4(v[0], v[1], v[2], v[3]));
  else
    __stcs(p, v[0]);
}
template <int V>
__device__ __forceinline__ void st_c(float* p, const float (&v)[V]) {
  if constexpr (V == 4)
    *reinterpret_cast<float4*>(p) = make_float4(v[0], v[1], v[2], v[3]);
  else
    *p = v[0];
}
__device__ __forceinline__ uint32_t pack_bf16(float a, float b) {
  const __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
  return *reinterpret_cast<const uint32_t*>(&h);
}
__device__ __forceinline__ uint32_t pack_half(float a, float b) {
  const __half2 h = __floats2half2_rn(a * kScale16, b * kScale16);
  return *reinterpret_cast<const uint32_t*>(&h);
}
template <int V>
__device__ __forceinline__ void st_c(__nv_bfloat16* p, const float (&v)[V]) {
  if constexpr (V == 4)
    *reinterpret_cast<uint2*>(p) = make_uint2(pack_bf16(v[0], v[1]), pack_bf16(v[2], v[3]));
  else
    *p = __float2bfloat16_rn(v[0]);
}
template <int V>
__device__ __forceinline__ void st_c(__half* p, const float (&v)[V]) {
  if constexpr (V == 4)
    *reinterpret_cast<uint2*>(p) = make_uint2(pack_half(v[0], v[1]), pack_half(v[2], v[3]));
  else
    *p = __float2half_rn(v[0] * kScale16);
}

// Two FP32 additions in one instruction.
__device__ __forceinline__ float2 add2(float2 a, float2 b) {
  unsigned long long x, y, z;
  asm("mov.b64 %0, {%1, %2};" : "=l"(x) : "f"(a.x), "f"(a.y));
  asm("mov.b64 %0, {%1, %2};" : "=l"(y) : "f"(b.x), "f"(b.y));
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(z) : "l"(x), "l"(y));
  float2 r;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(z));
  return r;
}

// The sum of the contributions of edges [e0, e1), the whole warp on one row
// (W = 16, 64), in the order described above: every lane returns its columns'
// sums.  idx: this lane's source of edge e0 + lane (loaded ahead by the
// caller), or n, the zero row, past the end: groups of edges are read whole.
// base: the lane's columns in row 0; a lane whose columns are not running has
// stride 0 and its columns in the zero row there.
template <typename T, int W>
__device__ __forceinline__ void gather_warp_row(const int32_t* __restrict__ row_idx, const T* __restrict__ base,
                                                int32_t stride, int32_t n, int32_t e0, int32_t e1, int32_t idx,
                                                int lane, float (&y)[Geo<W>::V]) {
  constexpr int V = Geo<W>::V, L = Geo<W>::L, G = Geo<W>::G;
  constexpr int P = 8 / G;  // slots of this lane's edges: G * i + g, i < P
  static_assert(Geo<W>::R == 1 && V == 4, "one row per warp, four columns per lane");
  const int g = lane / L;
  float2 tot[2] = {{0.f, 0.f}, {0.f, 0.f}};
  for (int32_t b = e0; b < e1; b += 64) {
    float2 s[P][2];
#pragma unroll
    for (int i = 0; i < P; ++i) s[i][0] = s[i][1] = make_float2(0.f, 0.f);
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int32_t e = b + 32 * h;
      if (e >= e1) break;
      if (e > e0) idx = e + lane < e1 ? __ldcs(row_idx + e + lane) : n;
      const int cnt = min(32, e1 - e);
      auto group = [&](auto loads, int j) {
        constexpr int U = decltype(loads)::value;
        float c[U][V];
#pragma unroll
        for (int i = 0; i < U; ++i) {
          const int32_t u = __shfl_sync(0xffffffffu, idx, j + G * i + g);
          ld_c<V>(base + (int64_t)u * stride, c[i]);
        }
#pragma unroll
        for (int i = 0; i < U; ++i) {
          s[i % P][0] = add2(s[i % P][0], make_float2(c[i][0], c[i][1]));
          s[i % P][1] = add2(s[i % P][1], make_float2(c[i][2], c[i][3]));
        }
      };
      if constexpr (G == 2) {
        // 16 edges in flight where no sums are held beside them yet, then 8 (16
        // throughout spills 60 registers a lane, whose traffic was more than
        // the gathers': 256 batch graphs, FP32, 274 ms against 268; 64 in BF16
        // 94.3 against 85.2; one 2^20-node graph 28.6 against 26.0)
        int j = 0;
        if (h == 0 && cnt > 8) {
          float c[8][V];
#pragma unroll
          for (int i = 0; i < 8; ++i) ld_c<V>(base + (int64_t)__shfl_sync(0xffffffffu, idx, 2 * i + g) * stride, c[i]);
#pragma unroll
          for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int v = 0; v < 2; ++v)
              s[i][v] = add2(add2(make_float2(0.f, 0.f), make_float2(c[i][2 * v], c[i][2 * v + 1])),
                             make_float2(c[i + 4][2 * v], c[i + 4][2 * v + 1]));
          j = 16;
        }
        for (; j < cnt; j += 8) group(std::integral_constant<int, 4>{}, j);
      } else {
        if (cnt > 8)
          group(std::integral_constant<int, 4>{}, 0);
        else
          group(std::integral_constant<int, 1>{}, 0);
      }
    }
    // even and odd slots: (S0 + S2) + (S4 + S6), (S1 + S3) + (S5 + S7)
#pragma unroll
    for (int v = 0; v < 2; ++v) {
      float2 t;
      if constexpr (P == 4) {
        t = add2(add2(s[0][v], s[1][v]), add2(s[2][v], s[3][v]));
      } else {
        static_assert(P == 1, "two or eight edges per load");
        t = s[0][v];
#pragma unroll
        for (int o = 2 * L; o <= 4 * L; o *= 2)
          t = add2(t, make_float2(__shfl_xor_sync(0xffffffffu, t.x, o), __shfl_xor_sync(0xffffffffu, t.y, o)));
      }
      tot[v] = add2(tot[v], t);
    }
  }
#pragma unroll
  for (int v = 0; v < 2; ++v) {
    y[2 * v] = tot[v].x + __shfl_xor_sync(0xffffffffu, tot[v].x, L);
    y[2 * v + 1] = tot[v].y + __shfl_xor_sync(0xffffffffu, tot[v].y, L);
  }
}

// The same for two rows of at most kShortDeg = 8 edges at once, half a warp each
// (W = 64), an edge per slot.  idx: lane l holds source l mod 16 of its half's
// row, or n.
template <typename T>
__device__ __forceinline__ void gather_pair(const T* __restrict__ base, int32_t stride, int32_t idx, int lane,
                                            float (&y)[4]) {
  static_assert(kShortDeg == 8, "an edge per slot");
  float c[8][4];
#pragma unroll
  for (int i = 0; i < 8; ++i)
    ld_c<4>(base + (int64_t)__shfl_sync(0xffffffffu, idx, (lane & 16) + i) * stride, c[i]);
#pragma unroll
  for (int v = 0; v < 4; v += 2) {
    auto p = [&](int i) { return make_float2(c[i][v], c[i][v + 1]); };
    const float2 t = add2(add2(add2(p(0), p(2)), add2(p(4), p(6))), add2(add2(p(1), p(3)), add2(p(5), p(7))));
    y[v] = t.x;
    y[v + 1] = t.y;
  }
}

// The same for W = 1 and 4: eight lanes per block of 64 edges, so a warp takes
// four blocks of one long row at a time (edges [e0, e1), the same for all
// lanes).
template <typename T, int W>
__device__ __forceinline__ void gather_narrow_long(const int32_t* __restrict__ row_idx, const T* __restrict__ C,
                                                   int32_t e0, int32_t e1, int lane, float (&y)[Geo<W>::V]) {
  constexpr int V = Geo<W>::V;
  static_assert(Geo<W>::R == 4, "eight lanes per block of edges");
  const int g = lane & 7, q = lane >> 3;
  float tot[V];
#pragma unroll
  for (int v = 0; v < V; ++v) tot[v] = 0.f;
  for (int32_t b = e0; b < e1; b += 256) {
    float s[V];
#pragma unroll
    for (int v = 0; v < V; ++v) s[v] = 0.f;
    int32_t u[8];
    float c[8][V];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const int32_t e = b + 64 * q + 8 * i + g;
      u[i] = e < e1 ? __ldcs(row_idx + e) : -1;
    }
#pragma unroll
    for (int i = 0; i < 8; ++i) {
#pragma unroll
      for (int v = 0; v < V; ++v) c[i][v] = 0.f;
      if (u[i] >= 0) ld_c<V>(C + (int64_t)u[i] * W, c[i]);
    }
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
      for (int v = 0; v < V; ++v) s[v] += c[i][v];
#pragma unroll
    for (int v = 0; v < V; ++v) {
      s[v] += __shfl_xor_sync(0xffffffffu, s[v], 2);
      s[v] += __shfl_xor_sync(0xffffffffu, s[v], 4);
      // the four blocks in order (lanes of even g: even slots, of odd g: odd)
#pragma unroll
      for (int k = 0; k < 4; ++k) tot[v] += __shfl_sync(0xffffffffu, s[v], 8 * k + (lane & 1));
    }
  }
#pragma unroll
  for (int v = 0; v < V; ++v) y[v] = tot[v] + __shfl_xor_sync(0xffffffffu, tot[v], 1);
}

// The same for four rows of at most 64 edges at once, eight lanes per row
// (edges [e0, e1) of this lane's row; u: its first four sources, or -1).
template <typename T, int W>
__device__ __forceinline__ void gather_narrow_short(const int32_t* __restrict__ row_idx, const T* __restrict__ C,
                                                    int32_t e0, int32_t e1, const int32_t (&u0)[4], int lane,
                                                    float (&y)[Geo<W>::V]) {
  constexpr int V = Geo<W>::V;
  const int g = lane & 7;
  float s[V];
#pragma unroll
  for (int v = 0; v < V; ++v) s[v] = 0.f;
  auto add4 = [&](const int32_t (&u)[4]) {
    float c[4][V];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
#pragma unroll
      for (int v = 0; v < V; ++v) c[i][v] = 0.f;
      if (u[i] >= 0) ld_c<V>(C + (int64_t)u[i] * W, c[i]);
    }
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int v = 0; v < V; ++v) s[v] += c[i][v];
  };
  add4(u0);
  const int32_t e = e0 + 32 + g;
  if (__any_sync(0xffffffffu, e < e1)) {
    int32_t u[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) u[i] = e + 8 * i < e1 ? __ldcs(row_idx + e + 8 * i) : -1;
    add4(u);
  }
#pragma unroll
  for (int v = 0; v < V; ++v) {
    s[v] += __shfl_xor_sync(0xffffffffu, s[v], 2);
    s[v] += __shfl_xor_sync(0xffffffffu, s[v], 4);
    y[v] = s[v] + __shfl_xor_sync(0xffffffffu, s[v], 1);
  }
}

// What a block needs of its job's column state.
template <int W>
struct ColShared {
  float d[W], b[W], bp[W];
  int32_t seed[W];  // relabelled seed row of a running column, else -1
  uint8_t live[W];
  uint32_t seeded[32];  // bit (p mod 1024): some running column's seed row is p modulo 1024
};

// The V columns from c0 on, which this lane holds.
template <int V>
struct LaneCols {
  int c0;
  bool on;       // some of them are running
  uint32_t live; // bit v: column c0 + v is running
};

// A row's state in this lane's columns, loaded before the row's gathers.
template <int V>
struct RowState {
  float inv, x[V], sent[V];
};
template <typename T, int W>
__device__ __forceinline__ RowState<Geo<W>::V> row_state(const float* inv_deg, const float* X, const float* S, int32_t p,
                                                         const LaneCols<Geo<W>::V>& lc) {
  constexpr int V = Geo<W>::V;
  RowState<V> r;
  r.inv = __ldg(inv_deg + p);
  if (lc.on) {
    ld_f<V>(X + (int64_t)p * W + lc.c0, r.x);
    if constexpr (std::is_same<T, __nv_bfloat16>::value) ld_f<V>(S + (int64_t)p * W + lc.c0, r.sent);
  }
  return r;
}

// Finishes row p for this lane's columns, from their sums y: stores the state
// (if wx) and the contributions (if wc), and returns in dn[] and rs[] the
// row's part of the dangling mass and the residual.
template <typename T, int W>
__device__ __forceinline__ void finish_cols(int32_t p, const float (&y)[Geo<W>::V], const RowState<Geo<W>::V>& rst,
                                            const LaneCols<Geo<W>::V>& lc, const ColShared<W>& cs,
                                            float* __restrict__ X, float* __restrict__ S, T* __restrict__ Cout,
                                            bool wx, bool wc, float (&dn)[Geo<W>::V], float (&rs)[Geo<W>::V]) {
  constexpr int V = Geo<W>::V;
  constexpr bool kDelta = std::is_same<T, __nv_bfloat16>::value;
  const int64_t o = (int64_t)p * W + lc.c0;
  const float inv = rst.inv;
  float xo[V], nx[V], add[V];
  bool seed[V];
#pragma unroll
  for (int v = 0; v < V; ++v) {
    xo[v] = rst.x[v];
    seed[v] = cs.seed[lc.c0 + v] == p;
    add[v] = seed[v] ? cs.b[lc.c0 + v] : 0.f;
  }
  if constexpr (kDelta) {
    float sent[V], q[V];
#pragma unroll
    for (int v = 0; v < V; ++v) {
      const bool live = (lc.live >> v) & 1u;
      sent[v] = rst.sent[v];
      const float yn = xo[v] + y[v];
      const float old = fmaf(cs.d[lc.c0 + v], xo[v], seed[v] ? cs.bp[lc.c0 + v] : 0.f);
      nx[v] = fmaf(cs.d[lc.c0 + v], yn, add[v]);
      rs[v] = fabsf(nx[v] - old);
      q[v] = live ? __bfloat162float(__float2bfloat16_rn(nx[v] * inv - sent[v])) : 0.f;
      sent[v] += q[v];
      if (live) xo[v] = yn;
      dn[v] = inv == 0.f ? nx[v] : 0.f;
    }
    if (wx) {
      st_f<V>(X + o, xo);
      st_f<V>(S + o, sent);
    }
    if (wc) st_c<V>(Cout + o, q);
  } else {
    float c[V];
#pragma unroll
    for (int v = 0; v < V; ++v) {
      nx[v] = (lc.live >> v) & 1u ? fmaf(cs.d[lc.c0 + v], y[v], add[v]) : xo[v];
      rs[v] = fabsf(nx[v] - xo[v]);
      c[v] = nx[v] * inv;
      dn[v] = inv == 0.f ? nx[v] : 0.f;
    }
    if (wx) st_f<V>(X + o, nx);
    if (wc) st_c<V>(Cout + o, c);
  }
}

// The sum of a long row's chunk sums, in order.
template <int W>
__device__ __forceinline__ void sum_chunks(const float* __restrict__ chunk_sum, int32_t first, int32_t deg,
                                           int32_t long_deg, int c0, float (&y)[Geo<W>::V]) {
  constexpr int V = Geo<W>::V;
  const int32_t c = chunk_edges(deg, long_deg), cnt = (deg + c - 1) / c;
  const float* base = chunk_sum + (int64_t)first * W + c0;
#pragma unroll
  for (int v = 0; v < V; ++v) y[v] = 0.f;
  int32_t k = 0;
  for (; k + 8 <= cnt; k += 8) {
    float z[8][V], t[V];
#pragma unroll
    for (int i = 0; i < 8; ++i) ld_c<V>(base + (int64_t)(k + i) * W, z[i]);
#pragma unroll
    for (int v = 0; v < V; ++v) t[v] = z[0][v];
#pragma unroll
    for (int i = 1; i < 8; ++i)
#pragma unroll
      for (int v = 0; v < V; ++v) t[v] += z[i][v];
#pragma unroll
    for (int v = 0; v < V; ++v) y[v] += t[v];
  }
  float t[V];
#pragma unroll
  for (int v = 0; v < V; ++v) t[v] = 0.f;
  for (; k < cnt; ++k) {
    float z[V];
    ld_c<V>(base + (int64_t)k * W, z);
#pragma unroll
    for (int v = 0; v < V; ++v) t[v] += z[v];
  }
#pragma unroll
  for (int v = 0; v < V; ++v) y[v] += t[v];
}

// The same of a slot's long row p, from the plan's chunks.
template <int W>
__device__ __forceinline__ void sum_plan_chunks(const StepJob* J, int32_t p, int c0, float (&y)[Geo<W>::V]) {
  constexpr int V = Geo<W>::V;
  int32_t lo = 0, hi = J->n_heavy;  // p's place among the long rows
  while (hi - lo > 1) {
    const int32_t mid = lo + (hi - lo) / 2;
    if (J->heavy_rows[mid] <= p)
      lo = mid;
    else
      hi = mid;
  }
  const int32_t sp = J->split0 + lo;
#pragma unroll
  for (int v = 0; v < V; ++v) y[v] = 0.f;
  for (int pass = 0; pass < 2; ++pass) {
    const int32_t k0 = pass == 0 ? J->split_hbeg[sp] : J->split_cbeg[sp];
    const int32_t k1 = pass == 0 ? J->split_hend[sp] : J->split_cend[sp];
    for (int32_t k = k0; k < k1; k += 8) {
      float t[V];
#pragma unroll
      for (int v = 0; v < V; ++v) t[v] = 0.f;
#pragma unroll 4
      for (int32_t q = k; q < min(k + 8, k1); ++q) {
        float z[V];
        ld_c<V>((const float*)J->chunk_sum + (int64_t)q * W + c0, z);
#pragma unroll
        for (int v = 0; v < V; ++v) t[v] += z[v];
      }
#pragma unroll
      for (int v = 0; v < V; ++v) y[v] += t[v];
    }
  }
}

// One step of every item: item (job, q) takes the pieces
// [q * per, (q + 1) * per) * kStWarps of its job, its warps one after another.
// kSlot: a slot of the server (its long rows' chunks are the plan's).
template <typename T, int W, bool kSlot>
__global__ void __launch_bounds__(kStThreads, 3) ppr_rows_kernel(const StepJob* __restrict__ jobs,
                                                             const StepItem* __restrict__ items, int step,
                                                             uint32_t* __restrict__ live_jobs) {
  constexpr int V = Geo<W>::V, L = Geo<W>::L, R = Geo<W>::R;
  __shared__ ColShared<W> cs;
  __shared__ unsigned long long s_acc[kStWarps][2][W];
  __shared__ int s_last, s_next;
  const StepItem item = items[blockIdx.x];
  const StepJob* J = jobs + item.slot;
  StepState* st = J->st;
  if (__ldcg(&st->live) == 0) return;  // the same for every block of the job: changed only after all have arrived
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  if (tid < 32) cs.seeded[tid] = 0;
  __syncthreads();
  if (tid < W) {
    const bool live = st->status[tid] == kColRunning;
    if (live) atomicOr(&cs.seeded[(st->seed[tid] >> 5) & 31], 1u << (st->seed[tid] & 31));
    cs.d[tid] = st->d[tid];
    cs.b[tid] = st->b[tid];
    cs.bp[tid] = st->bprev[tid];
    cs.seed[tid] = live ? st->seed[tid] : -1;
    cs.live[tid] = live;
  }
  const int32_t* __restrict__ col_ptr = J->col_ptr;
  const int32_t* __restrict__ row_idx = J->row_idx;
  const int32_t* __restrict__ prows = J->prows;
  const int parity = (J->parity + step) & 1;
  const T* __restrict__ Cin = (const T*)J->C[parity];
  T* __restrict__ Cout = (T*)J->C[parity ^ 1];
  const float* __restrict__ chunk_sum = J->chunk_sum;
  int32_t long_deg = kLongDeg;
  if constexpr (kSlot) long_deg = J->long_deg;
  const int32_t per = J->per, piece0 = item.part * kStWarps * per, pieces = min(kStWarps * per, J->npieces - piece0);
  if (tid == 0) s_next = kStWarps;
  __syncthreads();
  const int c0 = (lane % L) * V;
  // a lane whose columns are all finished reads the zero row and writes nothing
  bool on = false;
#pragma unroll
  for (int v = 0; v < V; ++v) on = on || cs.live[c0 + v] != 0;
  const int32_t n = J->n, stride = on ? W : 0;
  const T* __restrict__ cbase = Cin + c0 + (on ? 0 : (int64_t)n * W);
  const int g = (lane / L) & 7;  // the lane's edge group
  const float* __restrict__ inv_deg = J->inv_deg;
  float* __restrict__ X = J->X;
  float* __restrict__ S = J->S;
  LaneCols<V> lc;
  lc.c0 = c0;
  lc.on = on;
  lc.live = 0;
#pragma unroll
  for (int v = 0; v < V; ++v) lc.live |= (uint32_t)(cs.live[c0 + v] != 0) << v;
  for (int i = lane; i < 2 * W; i += 32) (&s_acc[warp][0][0])[i] = 0ull;
  __syncwarp();

  for (int32_t piece = warp; piece < pieces;) {
    const int32_t r0 = prows[piece0 + piece], r1 = prows[piece0 + piece + 1];
    if (lane == 0) piece = atomicAdd(&s_next, 1);  // the warp's next piece
    piece = __shfl_sync(0xffffffffu, piece, 0);
    float dsum[V], rsum[V];
#pragma unroll
    for (int v = 0; v < V; ++v) dsum[v] = rsum[v] = 0.f;
    for (int32_t base = r0; base < r1; base += 32) {
      // 32 rows: their offsets, and which have anything to do (a row without
      // in-edges keeps x = 0 unless it is a running column's seed)
      const int32_t p = base + lane;
      int32_t e0 = 0, e1 = 0;
      bool act = false;
      if (p < r1) {
        e0 = col_ptr[p];
        e1 = col_ptr[p + 1];
        act = e1 > e0 || ((cs.seeded[(p >> 5) & 31] >> (p & 31)) & 1u);
      }
      uint32_t shorts = __ballot_sync(0xffffffffu, act && e1 - e0 <= kShortDeg);
      uint32_t others = __ballot_sync(0xffffffffu, act && e1 - e0 > kShortDeg);
      if constexpr (R == 1) {
        uint32_t mask = shorts;
        int32_t nrow, ne0, ne1, nidx;
        if constexpr (W == 64) {
          // two short rows at a time, half a warp each; the next two rows'
          // sources are loaded ahead
          auto ahead = [&]() {
            int b = __ffs(mask) - 1;
            mask &= mask - 1;
            if (lane >= 16) b = __ffs(mask) - 1;
            mask &= mask - 1;  // (0 stays 0)
            nrow = b >= 0 ? base + b : -1;
            ne0 = __shfl_sync(0xffffffffu, e0, b & 31);
            ne1 = __shfl_sync(0xffffffffu, e1, b & 31);
            if (b < 0) ne0 = ne1 = 0;
            nidx = ne0 + (lane & 15) < ne1 ? __ldcs(row_idx + ne0 + (lane & 15)) : n;
          };
          bool more = mask != 0;
          if (more) ahead();
          while (more) {
            const int32_t row = nrow, idx = nidx;
            RowState<V> rst;
            rst.inv = 1.f;
            if (row >= 0) rst = row_state<T, W>(inv_deg, X, S, row, lc);
            more = mask != 0;
            if (more) ahead();
            float y[V], dn[V], rs[V];
            gather_pair<T>(cbase, stride, idx, lane, y);
#pragma unroll
            for (int v = 0; v < V; ++v) dn[v] = rs[v] = 0.f;
            if (row >= 0 && on) finish_cols<T, W>(row, y, rst, lc, cs, X, S, Cout, true, true, dn, rs);
            // both halves add the first row's part, then the second's
            const bool dang = __any_sync(0xffffffffu, rst.inv == 0.f);
#pragma unroll
            for (int v = 0; v < V; ++v) {
              const float o = __shfl_xor_sync(0xffffffffu, rs[v], 16);
              rsum[v] = lane < 16 ? (rsum[v] + rs[v]) + o : (rsum[v] + o) + rs[v];
              if (dang) {
                const float od = __shfl_xor_sync(0xffffffffu, dn[v], 16);
                dsum[v] = lane < 16 ? (dsum[v] + dn[v]) + od : (dsum[v] + od) + dn[v];
              }
            }
          }
          mask = others;
        }
        // a row at a time, loading ahead alike
        auto ahead = [&]() {
          const bool s = W != 64 && shorts != 0;  // (W = 16 takes the short rows here, first)
          uint32_t& m = s ? shorts : others;
          const int b = __ffs(m) - 1;
          m &= m - 1;
          nrow = base + b;
          ne0 = __shfl_sync(0xffffffffu, e0, b);
          ne1 = __shfl_sync(0xffffffffu, e1, b);
          nidx = ne0 + lane < ne1 && ne1 - ne0 <= long_deg ? __ldcs(row_idx + ne0 + lane) : n;
        };
        if (W == 64) shorts = 0;
        bool more = (shorts | others) != 0;
        if (more) ahead();
        while (more) {
          const int32_t row = nrow, a0 = ne0, a1 = ne1, idx = nidx;
          const RowState<V> rst = row_state<T, W>(inv_deg, X, S, row, lc);
          more = (shorts | others) != 0;
          if (more) ahead();
          float y[V];
          if (a1 - a0 > long_deg) {
            if constexpr (kSlot)
              sum_plan_chunks<W>(J, row, c0, y);
            else
              sum_chunks<W>(chunk_sum, J->long_base[row], a1 - a0, long_deg, c0, y);
          } else
            gather_warp_row<T, W>(row_idx, cbase, stride, n, a0, a1, idx, lane, y);
          if (on) {
            float dn[V], rs[V];
            finish_cols<T, W>(row, y, rst, lc, cs, X, S, Cout, g == 0, g == 1, dn, rs);
#pragma unroll
            for (int v = 0; v < V; ++v) {
              dsum[v] += dn[v];
              rsum[v] += rs[v];
            }
          }
        }
      } else {
        // four active rows side by side, eight lanes each; the next four rows'
        // sources are loaded ahead
        const int q = lane >> 3;
        int32_t nrow, ne0, ne1, nu[4];
        auto ahead = [&]() {
          int mine = -1;
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            uint32_t& m = shorts ? shorts : others;
            if (q == k && m) mine = __ffs(m) - 1;
            m &= m - 1;  // (0 stays 0)
          }
          ne0 = __shfl_sync(0xffffffffu, e0, mine & 31);
          ne1 = __shfl_sync(0xffffffffu, e1, mine & 31);
          nrow = mine >= 0 ? base + mine : -1;
          if (mine < 0) ne0 = ne1 = 0;
#pragma unroll
          for (int i = 0; i < 4; ++i)
            nu[i] = ne0 + g + 8 * i < ne1 && ne1 - ne0 <= 64 ? __ldcs(row_idx + ne0 + g + 8 * i) : -1;
        };
        bool more = (shorts | others) != 0;
        if (more) ahead();
        while (more) {
          const int32_t row = nrow, a0 = ne0, a1 = ne1;
          const int32_t u[4] = {nu[0], nu[1], nu[2], nu[3]};
          RowState<V> rst;
          if (row >= 0) rst = row_state<T, W>(inv_deg, X, S, row, lc);
          more = (shorts | others) != 0;
          if (more) ahead();
          float y[V];
          const int32_t deg = a1 - a0;
          gather_narrow_short<T, W>(row_idx, Cin, a0, deg <= 64 ? a1 : a0, u, lane, y);
          if (deg > long_deg) sum_chunks<W>(chunk_sum, J->long_base[row], deg, long_deg, c0, y);
          uint32_t lm = __ballot_sync(0xffffffffu, deg > 64 && deg <= long_deg) & 0x01010101u;  // a lane of each
          while (lm) {
            const int src = __ffs(lm) - 1;
            lm &= lm - 1;
            float z[V];
            gather_narrow_long<T, W>(row_idx, Cin, __shfl_sync(0xffffffffu, a0, src),
                                     __shfl_sync(0xffffffffu, a1, src), lane, z);
            if (q == src >> 3) {
#pragma unroll
              for (int v = 0; v < V; ++v) y[v] = z[v];
            }
          }
          float dn[V], rs[V];
#pragma unroll
          for (int v = 0; v < V; ++v) dn[v] = rs[v] = 0.f;
          if (row >= 0 && g == 0) finish_cols<T, W>(row, y, rst, lc, cs, X, S, Cout, true, true, dn, rs);
#pragma unroll
          for (int k = 0; k < 4; ++k)
#pragma unroll
            for (int v = 0; v < V; ++v) {
              dsum[v] += __shfl_sync(0xffffffffu, dn[v], 8 * k);
              rsum[v] += __shfl_sync(0xffffffffu, rs[v], 8 * k);
            }
        }
      }
    }
    if (lane < L) {
#pragma unroll
      for (int v = 0; v < V; ++v) {
        s_acc[warp][0][c0 + v] += std::is_same<T, __nv_bfloat16>::value ? fix60_signed(dsum[v]) : fix60(dsum[v]);
        s_acc[warp][1][c0 + v] += fix60(rsum[v]);
      }
    }
  }
  __syncthreads();
  for (int i = tid; i < 2 * W; i += kStThreads) {
    const int v = i / W, k = i % W;
    unsigned long long t = 0ull;
#pragma unroll
    for (int w = 0; w < kStWarps; ++w) t += s_acc[w][v][k];
    if (t != 0ull && cs.live[k]) atomicAdd(&st->acc[v][k], t);
  }
  // the last item of the job decides which columns stop and sets the next
  // step's seed coefficients
  __threadfence();
  __syncthreads();
  if (tid == 0) s_last = atomicAdd(&st->arrived, 1u) == (unsigned)(J->nitems - 1);
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  int live = 0;
  if (tid < W && cs.live[tid]) {
    const double D = fix60_value(__ldcg(&st->acc[0][tid])), res = fix60_value(__ldcg(&st->acc[1][tid]));
    st->acc[0][tid] = st->acc[1][tid] = 0ull;
    const double d = cs.d[tid];
    const int32_t it = st->iters[tid] + 1;
    int32_t stall = st->stall[tid];
    if (res < st->best[tid]) {
      st->best[tid] = res;
      stall = 0;
    } else {
      ++stall;
    }
    const float tol = st->tol[tid];
    const bool stop = (tol > 0.f && ((d / (1.0 - d)) * res <= (double)tol || stall >= kStallSteps)) ||
                      it >= st->max_iters[tid];
    st->bprev[tid] = cs.b[tid];
    st->b[tid] = (float)((1.0 - d) + d * D);
    st->res[tid] = res;
    st->iters[tid] = it;
    st->stall[tid] = stall;
    if (stop) st->status[tid] = kColDone;
    live = !stop;
  }
  live = __syncthreads_count(live);
  if (tid == 0) {
    st->arrived = 0;
    st->live = live;
    if (live == 0) atomicSub(live_jobs, 1u);
  }
}

// The sum of one chunk of a long row, a warp's work.
template <typename T, int W>
__device__ __forceinline__ void long_chunk(const StepJob* J, int32_t e0, int32_t e1, int32_t ch, int step, int lane) {
  constexpr int V = Geo<W>::V, L = Geo<W>::L, R = Geo<W>::R;
  const StepState* st = J->st;
  if (st->live == 0) return;
  const int c0 = (lane % L) * V;
  bool on = false;
#pragma unroll
  for (int v = 0; v < V; ++v) on = on || st->status[c0 + v] == kColRunning;
  const T* __restrict__ Cin = (const T*)J->C[(J->parity + step) & 1];
  float y[V];
  if constexpr (R == 1) {
    const int32_t n = J->n;
    const int32_t idx = e0 + lane < e1 ? __ldcs(J->row_idx + e0 + lane) : n;
    gather_warp_row<T, W>(J->row_idx, Cin + c0 + (on ? 0 : (int64_t)n * W), on ? W : 0, n, e0, e1, idx, lane, y);
  } else {
    gather_narrow_long<T, W>(J->row_idx, Cin, e0, e1, lane, y);
  }
  if (on && lane < L) st_c<V>(J->chunk_sum + (int64_t)ch * W + c0, y);
}

// The chunk sums of the long rows of a batch's wave, a warp per chunk of its
// list.
template <typename T, int W>
__global__ void __launch_bounds__(kStThreads) ppr_long_kernel(const StepJob* __restrict__ jobs,
                                                             const LongChunk* __restrict__ chunks,
                                                             const int32_t* __restrict__ nchunks, int step) {
  const int32_t total = *nchunks;
  for (int32_t ch = blockIdx.x * kStWarps + (threadIdx.x >> 5); ch < total; ch += gridDim.x * kStWarps) {
    const LongChunk lc = chunks[ch];
    long_chunk<T, W>(jobs + lc.slot, lc.e0, lc.e1, ch, step, threadIdx.x & 31);
  }
}

// The same of the server's slots: item (slot, q) takes the slot's chunks
// [q * kStWarps, (q + 1) * kStWarps).
template <typename T>
__global__ void __launch_bounds__(kStThreads) ppr_slot_long_kernel(const StepJob* __restrict__ jobs,
                                                                  const StepItem* __restrict__ items, int step) {
  const StepItem item = items[blockIdx.x];
  const StepJob* J = jobs + item.slot;
  const int32_t ch = item.part * kStWarps + (threadIdx.x >> 5);
  if (ch >= J->nchunks) return;
  long_chunk<T, kPprCols>(J, J->chunk_begin[ch], J->chunk_end[ch], ch, step, threadIdx.x & 31);
}

// Row boundaries of a job's pieces: equal shares of edges + 3 * rows.
__device__ __forceinline__ void piece_bounds(const int32_t* __restrict__ col_ptr, int32_t n, int64_t m, int32_t cnt,
                                             int32_t* __restrict__ prows) {
  const int64_t work = m + 3 * (int64_t)n;
  for (int32_t i = blockIdx.x * blockDim.x + threadIdx.x; i <= cnt; i += gridDim.x * blockDim.x) {
    const int64_t key = (work * i + cnt - 1) / cnt;
    int32_t lo = 0, hi = n;
    if (i == cnt) lo = hi;
    while (lo < hi) {
      const int32_t mid = lo + (hi - lo) / 2;
      if ((int64_t)col_ptr[mid] + 3 * (int64_t)mid < key)
        lo = mid + 1;
      else
        hi = mid;
    }
    prows[i] = lo;
  }
}
__global__ void ppr_bounds_kernel(const StepJob* __restrict__ jobs) {
  const StepJob* J = jobs + blockIdx.y;
  piece_bounds(J->col_ptr, J->n, J->m, J->npieces, J->prows);
}

__global__ void ppr_graph_bounds_kernel(const int32_t* __restrict__ col_ptr, int32_t n, int64_t m, int32_t cnt,
                                        int32_t* __restrict__ prows) {
  piece_bounds(col_ptr, n, m, cnt, prows);
}

// Column k starts from its record; returns whether it has a step to run.
__device__ __forceinline__ int start_column(const StepJob* J, const PprCol& c, int k) {
  StepState* st = J->st;
  const int32_t seed = J->old2new[c.seed];
  const double d = c.damping, D = J->inv_deg[seed] == 0.f ? 1.0 : 0.0;
  const int live = c.max_iters > 0;
  st->d[k] = c.damping;
  st->b[k] = (float)((1.0 - d) + d * D);
  st->bprev[k] = 1.f;  // x_0 = e_seed
  st->tol[k] = c.tol;
  st->max_iters[k] = c.max_iters;
  st->seed[k] = seed;
  st->status[k] = live ? kColRunning : kColDone;
  st->iters[k] = 0;
  st->stall[k] = 0;
  st->res[k] = 0.0;
  st->best[k] = INFINITY;
  st->acc[0][k] = st->acc[1][k] = 0ull;
  return live;
}

// x_0 = e_seed: the state and contributions of a job's rows (item by item),
// the chunks of its long rows (wherever the wave's list has room: a row's
// chunks stay together and in order) and, in the job's first item, the state
// of its columns.
template <typename T, int W>
__global__ void __launch_bounds__(kStThreads) ppr_start_kernel(const StepJob* __restrict__ jobs,
                                                              const StepItem* __restrict__ items,
                                                              LongChunk* __restrict__ chunks,
                                                              int32_t* __restrict__ nchunks,
                                                              uint32_t* __restrict__ live_jobs) {
  constexpr bool kDelta = std::is_same<T, __nv_bfloat16>::value;
  __shared__ int32_t s_seed[W];
  const StepItem item = items[blockIdx.x];
  const StepJob* J = jobs + item.slot;
  const int tid = threadIdx.x;
  if (tid < W) {
    const PprCol c = J->cols[tid];
    s_seed[tid] = c.status == kColFresh ? J->old2new[c.seed] : -1;
  }
  if (item.part == 0) {
    StepState* st = J->st;
    int live = 0;
    if (tid < kPprCols) {
      const PprCol c = J->cols[tid];
      if (tid < W && c.status == kColFresh)
        live = start_column(J, c, tid);
      else
        st->status[tid] = kColEmpty;
    }
    live = __syncthreads_count(live);
    if (tid == 0) {
      st->arrived = 0;
      st->live = live;
      if (live > 0) atomicAdd(live_jobs, 1u);
    }
  }
  __syncthreads();
  const int32_t per = J->per, piece0 = min(item.part * kStWarps * per, J->npieces);
  const int32_t r0 = J->prows[piece0], r1 = J->prows[min(piece0 + kStWarps * per, J->npieces)];
  for (int32_t p = r0 + tid; p < r1; p += kStThreads) {
    const int32_t e0 = J->col_ptr[p], deg = J->col_ptr[p + 1] - e0;
    if (deg <= kLongDeg) continue;
    const int32_t c = chunk_edges(deg, kLongDeg), cnt = (deg + c - 1) / c, first = atomicAdd(nchunks, cnt);
    J->long_base[p] = first;
    for (int32_t k = 0; k < cnt; ++k)
      chunks[first + k] = LongChunk{item.slot, e0 + k * c, e0 + min(deg, (k + 1) * c), 0};
  }
  const int64_t i0 = (int64_t)r0 * W, i1 = (int64_t)r1 * W;
  T* Cc = (T*)J->C[0];
  T* Co = (T*)J->C[1];
  if (item.part == 0 && tid < W) {
    const float zero[1] = {0.f};
    st_c<1>(Cc + (int64_t)J->n * W + tid, zero);
    st_c<1>(Co + (int64_t)J->n * W + tid, zero);
  }
  for (int64_t i = i0 + tid; i < i1; i += kStThreads) {
    const int32_t p = (int32_t)(i / W), k = (int32_t)(i % W);
    float x = 0.f, c[1] = {0.f};
    if (s_seed[k] == p) {
      x = 1.f;
      c[0] = J->inv_deg[p];
    }
    if (kDelta) {  // nothing gathered yet; the first delta is the whole contribution
      J->X[i] = 0.f;
      J->S[i] = __bfloat162float(__float2bfloat16_rn(c[0]));
    } else {
      J->X[i] = x;
    }
    st_c<1>(Cc + i, c);
    c[0] = 0.f;
    st_c<1>(Co + i, c);
  }
}

// The same for the columns that have joined a server's slot (status kColFresh
// in its records) since its last steps; those that finished then leave, and so
// do those whose record says that they are gone: the records are the server's
// word, the state is this side's.
template <typename T>
__global__ void __launch_bounds__(kStThreads) ppr_join_kernel(const StepJob* __restrict__ jobs,
                                                             const StepItem* __restrict__ items) {
  constexpr bool kDelta = std::is_same<T, __nv_bfloat16>::value;
  constexpr int W = kPprCols;
  __shared__ int32_t s_seed[W];
  __shared__ uint8_t s_fresh[W];
  const StepItem item = items[blockIdx.x];
  const StepJob* J = jobs + item.slot;
  const int tid = threadIdx.x;
  int fresh = 0, going = 0;
  if (tid < W) {
    const PprCol c = J->cols[tid];
    fresh = c.status == kColFresh;
    going = c.status == kColRunning;
    s_fresh[tid] = (uint8_t)fresh;
    s_seed[tid] = fresh ? J->old2new[c.seed] : -1;
  }
  if (item.part == 0) {
    StepState* st = J->st;
    int live = 0;
    if (tid < W) {
      if (fresh)
        live = start_column(J, J->cols[tid], tid);
      else if (going && st->status[tid] == kColRunning)
        live = 1;
      else
        st->status[tid] = kColEmpty;
    }
    live = __syncthreads_count(live);
    if (tid == 0) {
      st->arrived = 0;
      st->live = live;
    }
  }
  if (!__syncthreads_or(fresh)) return;
  const int parity = J->parity & 1;
  T* Cc = (T*)J->C[parity];
  T* Co = (T*)J->C[parity ^ 1];
  const int32_t per = J->per, piece0 = min(item.part * kStWarps * per, J->npieces);
  const int64_t i0 = (int64_t)J->prows[piece0] * W;
  const int64_t i1 = (int64_t)J->prows[min(piece0 + kStWarps * per, J->npieces)] * W;
  for (int64_t i = i0 + tid; i < i1; i += kStThreads) {
    const int32_t p = (int32_t)(i / W), k = (int32_t)(i % W);
    if (!s_fresh[k]) continue;
    float x = 0.f, c[1] = {0.f};
    if (s_seed[k] == p) {
      x = 1.f;
      c[0] = J->inv_deg[p];
    }
    if (kDelta) {
      J->X[i] = 0.f;
      J->S[i] = __bfloat162float(__float2bfloat16_rn(c[0]));
    } else {
      J->X[i] = x;
    }
    st_c<1>(Cc + i, c);
    c[0] = 0.f;
    st_c<1>(Co + i, c);
  }
}

// The finished columns by node id, and the records of all.
template <typename T, int W>
__global__ void __launch_bounds__(kStThreads) ppr_out_kernel(const StepJob* __restrict__ jobs,
                                                            const StepItem* __restrict__ items) {
  constexpr bool kDelta = std::is_same<T, __nv_bfloat16>::value;
  __shared__ float s_d[W], s_b[W];
  __shared__ int32_t s_seed[W], s_ldo[W];
  __shared__ float* s_out[W];  // null: not finished
  const StepItem item = items[blockIdx.x];
  const StepJob* J = jobs + item.slot;
  const StepState* st = J->st;
  const int tid = threadIdx.x;
  int done = 0;
  if (tid < W) {
    const int32_t status = st->status[tid];
    done = status == kColDone;
    s_d[tid] = st->d[tid];
    s_b[tid] = st->bprev[tid];
    s_seed[tid] = st->seed[tid];
    PprCol* c = J->cols + tid;
    s_out[tid] = done ? c->out : nullptr;
    s_ldo[tid] = c->ldo;
    if (item.part == 0 && status != kColEmpty) {
      c->status = status;
      c->iters = st->iters[tid];
      c->residual = st->res[tid];
    }
  }
  if (!__syncthreads_or(done)) return;
  const int32_t per = J->per, piece0 = min(item.part * kStWarps * per, J->npieces);
  const int64_t i0 = (int64_t)J->prows[piece0] * W;
  const int64_t i1 = (int64_t)J->prows[min(piece0 + kStWarps * per, J->npieces)] * W;
  for (int64_t i = i0 + tid; i < i1; i += kStThreads) {
    const int32_t p = (int32_t)(i / W), k = (int32_t)(i % W);
    float* out = s_out[k];
    if (!out) continue;
    float x = __ldcs(J->X + i);
    if (kDelta) x = fmaf(s_d[k], x, p == s_seed[k] ? s_b[k] : 0.f);
    out[(int64_t)J->new2old[p] * s_ldo[k]] = x;
  }
}

// ---- host side ----------------------------------------------------------------

static int width_of(int k) { return k <= 1 ? 1 : k <= 4 ? 4 : k <= 16 ? 16 : 64; }

// Workspace of one wave, at most (a larger job is a wave of its own).  256 batch
// graphs x 64 columns, 50 steps: 368 ms with waves of 192 MB, 293 ms with 1.5 GB,
// 270 ms with one wave of 7.2 GB: a launch's start and end cost more than what
// waves small enough for L2 save, since a launch takes its items job by job.  Above
// that nothing is gained: 4,096 graphs in FP32 / BF16 3.99 / 4.17 s with 8 GB, 4.01 /
// 4.28 with 12, 4.04 / 4.38 with 16.
constexpr int64_t kWaveBytes = (int64_t)8 << 30;
constexpr int64_t kMinWaveBytes = (int64_t)64 << 20;  // tried down to here when memory is short
constexpr int64_t kMaxPer = 4;                        // pieces per warp of an item

// Steps between two looks at whether every column has reached its tolerance.
constexpr int kStCheck = 16;

// A group of jobs of one width that take their steps together.
struct Wave {
  int w;
  int32_t job0, jobs;    // consecutive jobs
  int32_t item0, items;  // their items
  int per;               // pieces per warp of an item
  int64_t work, edges;
  int64_t chunks;        // long-row chunks at most
};

struct WaveBuffers {
  const StepJob* jobs;
  const StepItem* items;
  LongChunk* chunks;
  int32_t* counters;  // [0] chunks of the wave, [1] jobs with running columns
};

template <typename T, int W>
static void run_wave(const Wave& wv, const WaveBuffers& B, int32_t max_iters, bool check, cudaStream_t s) {
  const StepItem* items = B.items + wv.item0;
  uint32_t* live_dev = (uint32_t*)B.counters + 1;
  GPR_CUDA(cudaMemsetAsync(B.counters, 0, 8, s));
  ppr_start_kernel<T, W><<<wv.items, kStThreads, 0, s>>>(B.jobs, items, B.chunks, B.counters, live_dev);
  GPR_CUDA(cudaGetLastError());
  int64_t launches = 2;
  const int long_grid = (int)std::min<int64_t>((wv.chunks + kStWarps - 1) / kStWarps, (int64_t)num_sms() * 8);
  for (int32_t it = 0; it < max_iters; ++it) {
    if (check && it > 0 && it % kStCheck == 0) {
      uint32_t live = 0;
      GPR_CUDA(cudaMemcpyAsync(&live, live_dev, 4, cudaMemcpyDeviceToHost, s));
      GPR_CUDA(cudaStreamSynchronize(s));
      if (live == 0) break;
    }
    if (long_grid > 0) {
      ppr_long_kernel<T, W><<<long_grid, kStThreads, 0, s>>>(B.jobs, B.chunks, B.counters, it);
      ++launches;
    }
    ppr_rows_kernel<T, W, false><<<wv.items, kStThreads, 0, s>>>(B.jobs, items, it, live_dev);
    ++launches;
  }
  ppr_out_kernel<T, W><<<wv.items, kStThreads, 0, s>>>(B.jobs, items);
  GPR_CUDA(cudaGetLastError());
  count_launches(launches);
}

template <typename T>
static void run_wave_w(const Wave& wv, const WaveBuffers& B, int32_t max_iters, bool check, cudaStream_t s) {
  switch (wv.w) {
    case 1: run_wave<T, 1>(wv, B, max_iters, check, s); break;
    case 4: run_wave<T, 4>(wv, B, max_iters, check, s); break;
    case 16: run_wave<T, 16>(wv, B, max_iters, check, s); break;
    default: run_wave<T, 64>(wv, B, max_iters, check, s); break;
  }
}

static void run_waves(const std::vector<StepRequest>& reqs, int32_t max_iters, bool tol, gpr_dtype dt,
                      int64_t wave_bytes, bool* launched, cudaStream_t s) {
  std::vector<void*> tmp;
  auto alloc = [&](size_t bytes) {
    void* p = dalloc(bytes, s);
    tmp.push_back(p);
    return (char*)p;
  };
  auto round_up = [](int64_t b) { return (b + 255) & ~(int64_t)255; };
  try {
    const int64_t tsz = dt == GPR_FP32 ? 4 : 2;
    // widest first, then the largest work first
    std::vector<int32_t> order(reqs.size());
    for (size_t i = 0; i < order.size(); ++i) order[i] = (int32_t)i;
    auto work = [&](int32_t i) { return reqs[i].graph->m + 3 * (int64_t)reqs[i].graph->n; };
    std::stable_sort(order.begin(), order.end(), [&](int32_t a, int32_t b) {
      const int wa = width_of(reqs[a].k), wb = width_of(reqs[b].k);
      return wa != wb ? wa > wb : work(a) > work(b);
    });
    std::vector<Wave> waves;
    std::vector<StepJob> jobs;
    int64_t ws_bytes = 0, bound_bytes = 0, used = 0, wave = 0;
    for (int32_t r : order) {
      const gpr_graph* g = reqs[r].graph;
      const int w = width_of(reqs[r].k);
      const int64_t cells = (int64_t)g->n * w;
      const int64_t chunks = g->m / (kLongDeg / 2);  // a long row's chunks are at least half full
      const int64_t bytes = cells * (4 + 2 * tsz + (dt == GPR_BF16 ? 4 : 0)) + (int64_t)g->n * 4 +
                            chunks * (w * 4 + (int64_t)sizeof(LongChunk));
      if (waves.empty() || waves.back().w != w || wave + bytes > wave_bytes) {
        Wave wv{};
        wv.w = w;
        wv.job0 = (int32_t)jobs.size();
        waves.push_back(wv);
        used = wave = 0;
      }
      Wave& wv = waves.back();
      wave += bytes;
      StepJob J{};
      J.col_ptr = g->col_ptr;
      J.row_idx = g->row_idx;
      J.inv_deg = g->plan.inv_deg;
      J.old2new = g->plan.old2new;
      J.new2old = g->plan.new2old;
      J.n = g->n;
      J.m = g->m;
      J.cols = reqs[r].cols;
      J.long_deg = kLongDeg;
      J.npieces = ppr_pieces(g);
      // the job's part of the wave's workspace, as offsets for now
      auto take = [&](int64_t bytes) {
        const int64_t at = used;
        used += round_up(bytes);
        return (void*)(uintptr_t)at;
      };
      J.X = (float*)take(cells * 4);
      J.C[0] = take((cells + w) * tsz);
      J.C[1] = take((cells + w) * tsz);
      J.S = dt == GPR_BF16 ? (float*)take(cells * 4) : nullptr;
      J.long_base = (int32_t*)take((int64_t)g->n * 4);
      J.st = (StepState*)take(sizeof(StepState));
      ws_bytes = std::max(ws_bytes, used);
      J.prows = (int32_t*)(uintptr_t)bound_bytes;
      bound_bytes += round_up(((int64_t)J.npieces + 1) * 4);
      jobs.push_back(J);
      ++wv.jobs;
      wv.work += work(r);
      wv.chunks += chunks;
    }
    // items: a block of kStWarps x per pieces, so that a step has several
    // blocks for every SM, and few pieces wait on a block's start and end
    std::vector<StepItem> items;
    int64_t chunk_cells = 0, chunk_cap = 0;
    for (Wave& wv : waves) {
      const int64_t blocks = (int64_t)num_sms() * 8;
      wv.per = (int)std::max<int64_t>(1, std::min<int64_t>(kMaxPer, wv.work / (blocks * kStWarps * kPieceWork)));
      wv.item0 = (int32_t)items.size();
      for (int32_t j = wv.job0; j < wv.job0 + wv.jobs; ++j) {
        jobs[j].per = wv.per;
        jobs[j].nitems = (jobs[j].npieces + kStWarps * wv.per - 1) / (kStWarps * wv.per);
        for (int32_t q = 0; q < jobs[j].nitems; ++q) items.push_back(StepItem{j, q});
      }
      wv.items = (int32_t)items.size() - wv.item0;
      chunk_cap = std::max(chunk_cap, wv.chunks);
      chunk_cells = std::max(chunk_cells, wv.chunks * wv.w);
    }
    char* ws = alloc((size_t)ws_bytes);
    char* bounds = alloc((size_t)bound_bytes);
    for (StepJob& J : jobs) {
      auto at = [&](void* off) { return (void*)(ws + (uintptr_t)off); };
      J.X = (float*)at(J.X);
      J.C[0] = at(J.C[0]);
      J.C[1] = at(J.C[1]);
      if (dt == GPR_BF16) J.S = (float*)at(J.S);
      J.long_base = (int32_t*)at(J.long_base);
      J.st = (StepState*)at(J.st);
      J.prows = (int32_t*)(bounds + (uintptr_t)J.prows);
    }
    StepJob* jobs_dev = (StepJob*)alloc(jobs.size() * sizeof(StepJob));
    StepItem* items_dev = (StepItem*)alloc(items.size() * sizeof(StepItem));
    WaveBuffers B{};
    B.jobs = jobs_dev;
    B.items = items_dev;
    B.chunks = (LongChunk*)alloc((size_t)std::max<int64_t>(chunk_cap, 1) * sizeof(LongChunk));
    float* chunk_sum = (float*)alloc((size_t)std::max<int64_t>(chunk_cells, 1) * 4);
    for (StepJob& J : jobs) J.chunk_sum = chunk_sum;  // a wave's list is shared by its jobs
    B.counters = (int32_t*)alloc(8);
    *launched = true;
    GPR_CUDA(cudaMemcpyAsync(jobs_dev, jobs.data(), jobs.size() * sizeof(StepJob), cudaMemcpyHostToDevice, s));
    GPR_CUDA(cudaMemcpyAsync(items_dev, items.data(), items.size() * sizeof(StepItem), cudaMemcpyHostToDevice, s));
    for (size_t j0 = 0; j0 < jobs.size(); j0 += 32768) {  // grid.y is at most 65535
      const unsigned nj = (unsigned)std::min<size_t>(32768, jobs.size() - j0);
      ppr_bounds_kernel<<<dim3(4, nj), 256, 0, s>>>(jobs_dev + j0);
      GPR_CUDA(cudaGetLastError());
      count_launches(1);
    }
    for (const Wave& wv : waves) {
      if (dt == GPR_BF16)
        run_wave_w<__nv_bfloat16>(wv, B, max_iters, tol, s);
      else if (dt == GPR_FP16)
        run_wave_w<__half>(wv, B, max_iters, tol, s);
      else
        run_wave_w<float>(wv, B, max_iters, tol, s);
    }
    for (void* p : tmp) dfree(p, s);
  } catch (...) {
    for (void* p : tmp) dfree(p, s);
    throw;
  }
}

void run_ppr_steps(const std::vector<StepRequest>& reqs, int32_t max_iters, bool tol, gpr_dtype dt, cudaStream_t s) {
  if (reqs.empty()) return;
  for (int64_t wave_bytes = kWaveBytes;; wave_bytes /= 8) {
    bool launched = false;
    try {
      run_waves(reqs, max_iters, tol, dt, wave_bytes, &launched, s);
      return;
    } catch (const StatusFail& f) {
      // not enough memory for a wave's workspace: smaller waves
      if (launched || f.st != GPR_ENOMEM || wave_bytes / 8 < kMinWaveBytes) throw;
    }
  }
}

// ---- the server's slots ---------------------------------------------------------

int32_t ppr_pieces(const gpr_graph* g) {
  const int64_t work = g->m + 3 * (int64_t)g->n;
  return (int32_t)std::max<int64_t>(1, std::min<int64_t>((work + kPieceWork - 1) / kPieceWork, g->n));
}

void ppr_piece_bounds(const gpr_graph* g, int32_t* prows, cudaStream_t s) {
  const int32_t cnt = ppr_pieces(g);
  ppr_graph_bounds_kernel<<<std::min(1024, cnt / 256 + 1), 256, 0, s>>>(g->col_ptr, g->n, g->m, cnt, prows);
  GPR_CUDA(cudaGetLastError());
  count_launches(1);
}

void heavy_of(const gpr_graph* g, const int32_t** rows, int32_t* n, int32_t* deg, int32_t* split0) {
  const Plan& P = g->plan;
  *rows = P.rows;
  *n = 0;
  *deg = INT_MAX;
  *split0 = 0;
  // the long rows are the last chunked (lanes 0) bucket; the plan's split
  // entries list the rows of every chunked bucket in bucket order
  int32_t before = 0;
  for (int b = 0; b < P.nbuckets; ++b)
    if (P.bucket[b].lanes == 0) {
      *split0 = before;
      *rows = P.rows + P.bucket[b].row_begin;
      *n = P.bucket[b].row_end - P.bucket[b].row_begin;
      *deg = b > 0 ? P.deg_threshold[b - 1] : -1;  // bucket 0 holds every degree from 0
      before += *n;
    }
}

template <typename T>
static void slot_steps(const StepJob* jobs, const StepItem* items, int nitems, const StepItem* citems, int ncitems,
                       int32_t steps, uint32_t* scratch, cudaStream_t s) {
  ppr_join_kernel<T><<<nitems, kStThreads, 0, s>>>(jobs, items);
  for (int32_t it = 0; it < steps; ++it) {
    if (ncitems > 0) ppr_slot_long_kernel<T><<<ncitems, kStThreads, 0, s>>>(jobs, citems, it);
    ppr_rows_kernel<T, kPprCols, true><<<nitems, kStThreads, 0, s>>>(jobs, items, it, scratch);
  }
  ppr_out_kernel<T, kPprCols><<<nitems, kStThreads, 0, s>>>(jobs, items);
  GPR_CUDA(cudaGetLastError());
  count_launches(2 + (int64_t)steps * (ncitems > 0 ? 2 : 1));
}

void ppr_slot_steps(const StepJob* jobs, const StepItem* items, int nitems, const StepItem* citems, int ncitems,
                    int32_t steps, gpr_dtype dt, uint32_t* scratch, cudaStream_t s) {
  if (nitems <= 0) return;
  if (dt == GPR_BF16)
    slot_steps<__nv_bfloat16>(jobs, items, nitems, citems, ncitems, steps, scratch, s);
  else if (dt == GPR_FP16)
    slot_steps<__half>(jobs, items, nitems, citems, ncitems, steps, scratch, s);
  else
    slot_steps<float>(jobs, items, nitems, citems, ncitems, steps, scratch, s);
}

}  // namespace gpr
