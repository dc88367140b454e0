// The whole PageRank iteration of a small graph in one launch (section 4 Table
// "snap_methods"): the step of pr_step.cuh for graphs whose steps are bound by
// launches and latency, not by bytes.
//
// One block of 768 threads per SM, or one thread-block cluster where the
// graph is small enough that its hardware barrier is worth more than the other
// SMs.  Each step, a block copies the contributions of the first H relabelled
// ids (the most-read ones; all of them where they fit) into shared memory,
// sums its rows, finishes them and meets the other blocks at a barrier.
//
// What bounds it.  10,000 nodes, 100,000 edges, 50 steps: 650 us as a CUDA graph of
// six kernels a step, 163 us here, 3.2 us a step: the barrier and the writes
// before it 1.7, the sums 0.9, coefficients and copy 0.6.  250,000 nodes,
// 4,000,000 edges (R-MAT, BF16): 1,910 us against 740, 15 us a step, bound by the
// shared-memory and L1 slots of the gathers, about 10 cycles for 32 edges: long
// rows' chunks 4.7, slices 3.6, then the long rows' ends 2 to 3 on the blocks that
// have most and the barrier.
//
// Layout (made once per graph).  The rows run by descending in-degree.  Rows of
// up to kPersShort edges are sliced by 32, a lane a row, their sources stored
// slice by slice, edge by edge (lane l of edge j at off + 32 j + l, -1 past a
// row's end; SELL-C-sigma of Kreutzer et al. 2014 with C = 32 and all rows
// sorted): every index load of a warp is one 128-byte line and a row needs no
// reduction.  (Lanes sharing a row, four edges ahead, spent 400 issue and
// load slots a task: 10 us a step for 10,000 nodes and 100,000 edges on 16
// SMs.)  Longer rows, the longest first, and then the slices go to the block with
// the least estimated work so far; blocks cut long rows into chunks for their
// warps and add a row's chunk sums after a block barrier.
//
// Mass, dangling mass and residual: FP32 per thread and over the warp as in the
// pull kernels, then exact integer sums of multiples of 2^-60 over warps and
// blocks, so runs are bitwise identical.  A thread has more rows here, and where
// most rows hold the same rank all threads round alike, so its mass and dangling
// mass are sums of two floats (2^20 nodes and edges: L1 error 3.3e-8; with plain
// sums 6.4e-8, with the pull kernels 3.5e-8; 50 steps of 900,000 nodes and 4,100,000 edges 1,068 ->
// 1,090 us).
//
// The centralities take the same kernel a step at a time (kProduct):
// one launch a product instead of six.
//
// The barrier's wait is bounded: after kSpinLimit polls a block sets the error
// flag, writes NaN ranks and returns, and so do the others.
#pragma once

#include <cooperative_groups.h>

#include "pr_step.cuh"

namespace gpr {

constexpr int kPersThreads = 768;  // 80 registers a thread: a spill is reloaded from L2 after every barrier
constexpr int kPersWarps = kPersThreads / 32;
constexpr int32_t kPersShort = 64;      // rows up to here are sliced
constexpr int32_t kPersChunk = 256;     // edges of a long row's chunk, at least
constexpr int kPersRowChunks = 64;      // chunks of one long row, at most
constexpr int kPersLongRows = 512;      // long rows of one block, at most
constexpr int kPersChunks = 1280;       // chunks of one block, at most
constexpr int kPersIdx = 8;             // indices of a chunk that a lane holds
constexpr int kPersSlice = 8;           // and of a slice

struct PersistArgs {
  const int32_t* row_idx;
  const int32_t* row;       // n: the rows by descending in-degree
  const float* inv;         // n: their inverse out-degrees
  const int2* span;         // n_long: their edges
  const int32_t* off;       // nslices + 1: slices of rows [n_long, n)
  const int32_t* sell;
  const int32_t* deal;      // the blocks' shares: long rows of block b at deal[deal[b]] .. deal[deal[b + 1] - 1],
                            // slices at deal[deal[nblk + 1 + b]] .. (deal[2 nblk + 1] is the end)
  const float* inv_deg;     // by relabelled id
  const int32_t* old2new;
  int32_t n, n_long, nslices, H;
  float* xi;                // x of row[i]
  float* x;                 // x by relabelled id, written by the last step
  void* c[2];
  unsigned long long* sums; // (iters + 1) x 3, zero
  unsigned int* bar;        // [0] arrivals, zero; [1] error flag
  double* log_row;          // mass, dangling mass, residual of the last step
  float* out;
  // damping, (1 - d) / n and 1 / n, each the sum of two floats
  float d_hi, d_lo, t_hi, t_lo, in_hi, in_lo;
  int32_t iters;
};

// The stored contribution of source u: from the shared-memory copy of the first
// H, from L2 above, 0 for u < 0.  Predicated loads, no branch: a warp's loads
// overlap whichever way its lanes go.  The bits, to be taken by pers_value once
// all loads of a group are on their way.
__device__ __forceinline__ uint32_t pers_bits(uint32_t s_c, const float* c, int32_t u, int32_t H) {
  uint32_t v = 0;
  asm volatile(
      "{\n\t.reg .pred p, q;\n\tsetp.lt.u32 p, %1, %2;\n\tsetp.ge.s32 q, %1, %2;\n\t"
      "@p ld.shared.u32 %0, [%3];\n\t@q ld.global.cg.u32 %0, [%4];\n\t}"
      : "+r"(v)
      : "r"(u), "r"(H), "r"(s_c + 4u * (uint32_t)u), "l"(c + u));
  return v;
}
__device__ __forceinline__ uint32_t pers_bits(uint32_t s_c, const __nv_bfloat16* c, int32_t u, int32_t H) {
  uint32_t v = 0;
  asm volatile(
      "{\n\t.reg .pred p, q;\n\tsetp.lt.u32 p, %1, %2;\n\tsetp.ge.s32 q, %1, %2;\n\t"
      "@p ld.shared.u16 %0, [%3];\n\t@q ld.global.cg.u16 %0, [%4];\n\t}"
      : "+r"(v)
      : "r"(u), "r"(H), "r"(s_c + 2u * (uint32_t)u), "l"(c + u));
  return v;
}
__device__ __forceinline__ float pers_value(uint32_t v, const float*) { return __uint_as_float(v); }
__device__ __forceinline__ float pers_value(uint32_t v, const __nv_bfloat16*) { return __uint_as_float(v << 16); }

// Numbers as unevaluated sums of two floats (Dekker): a fixed-point sum of
// 2^-60 units; a product; the rounded sum of two non-negative ones.
__device__ __forceinline__ float2 pers_pair(unsigned long long s) {
  // 24 bits from the leading one on, and the rest
  const int z = __clzll((long long)(s | 1ull)), sh = 40 - z;
  const unsigned long long hi = sh > 0 ? (s >> sh) << sh : s;
  const float a = (float)(uint32_t)(sh > 0 ? s >> sh : s), unit = __uint_as_float((uint32_t)(127 - kFixBits) << 23);
  const float scale = sh > 0 ? __uint_as_float((uint32_t)(127 + sh) << 23) : 1.0f;
  const unsigned long long lo = s - hi;  // below 2^40
  const float b = fmaf((float)(uint32_t)(lo >> 16), 65536.0f, (float)(uint32_t)(lo & 0xFFFFu));
  return make_float2(a * scale * unit, b * unit);
}
__device__ __forceinline__ float2 pers_mul(float2 a, float2 b) {
  const float p = a.x * b.x;
  const float e = fmaf(a.x, b.x, -p) + fmaf(a.x, b.y, a.y * b.x);
  const float s = p + e;
  return make_float2(s, e - (s - p));
}
__device__ __forceinline__ float pers_add(float2 a, float2 b) {
  const float s = a.x + b.x, v = s - a.x;
  return s + (((a.x - (s - v)) + (b.x - v)) + (a.y + b.y));
}

// Edges per chunk of a long row.
__host__ __device__ __forceinline__ int32_t pers_chunk(int32_t deg) {
  const int32_t c = (deg + kPersRowChunks - 1) / kPersRowChunks;
  return c > kPersChunk ? c : kPersChunk;
}

// kProduct: one product of a power iteration, x = y / (largest entry of the vector
// before; 0 if that is 0), from contributions and a largest entry that the
// caller or the product before left (no start vector, so no barrier); x and
// contributions stored, no output.  sums rows hold the largest entry's bits: a
// product can scale the vector by anything, which fixed-point sums would not
// follow, and its largest entry is exact in any order.  (A kernel of its own, so
// that the iteration's loops hold nothing of it.)
template <typename T, bool kCluster, bool kProduct = false>
__global__ void __launch_bounds__(kPersThreads, 1) persist_kernel(const __grid_constant__ PersistArgs A) {
  extern __shared__ __align__(16) unsigned char pers_smem[];
  T* s_c = reinterpret_cast<T*>(pers_smem);
  const uint32_t s_addr = (uint32_t)__cvta_generic_to_shared(s_c);
  __shared__ int2 s_span[kPersLongRows];
  __shared__ int32_t s_first[kPersLongRows + 1];  // first chunk of each long row of the block
  __shared__ float s_chunk[kPersChunks];          // a chunk's sum
  __shared__ int2 s_edges[kPersChunks];           // its edges
  __shared__ unsigned long long s_sum[3][kPersWarps];
  __shared__ float s_coef[2];
  __shared__ int s_bad;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int32_t nblk = gridDim.x, n = A.n, H = A.H;
  const int32_t* my_long = A.deal + A.deal[blockIdx.x];
  const int32_t* my_slice = A.deal + A.deal[nblk + 1 + blockIdx.x];
  const int32_t nl = A.deal[blockIdx.x + 1] - A.deal[blockIdx.x];
  const int32_t nsl = A.deal[nblk + 2 + blockIdx.x] - A.deal[nblk + 1 + blockIdx.x];
  unsigned int phase = 0;
  bool failed = false;

  // every block's writes before it are seen by every block's reads after it
  auto barrier = [&]() {
    if constexpr (kCluster) {
      cooperative_groups::this_cluster().sync();
    } else {
      __syncthreads();
      if (tid == 0) {
        phase += (unsigned int)nblk;
        asm volatile("fence.acq_rel.gpu;" ::: "memory");
        asm volatile("red.relaxed.gpu.global.add.u32 [%0], 1;" ::"l"(A.bar) : "memory");
        uint32_t spins = 0;
        int bad = 0;
        for (;;) {
          unsigned int v;
          asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(A.bar) : "memory");
          if (v >= phase) break;
          if (++spins > kSpinLimit || ((spins & 1023) == 0 && *(volatile unsigned int*)(A.bar + 1))) {
            atomicOr(A.bar + 1, 1u);
            bad = 1;
            break;
          }
        }
        s_bad = bad;
      }
      __syncthreads();
      failed = s_bad != 0;
    }
  };
  // the block's sums into row `it`
  auto add_sums = [&](int32_t it) {
    __syncthreads();
    if (warp < 3) {
      unsigned long long t = lane < kPersWarps ? s_sum[warp][lane] : 0ull;
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
      if (lane == 0 && t) atomicAdd(A.sums + 3 * (int64_t)it + warp, t);
    }
  };
  auto add_max = [&](int32_t it, float mx) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    if (lane == 0 && mx > 0.f) atomicMax((unsigned int*)(A.sums + 3 * (int64_t)it), __float_as_uint(mx));
  };

  // the block's long rows and their chunks
  for (int32_t j = tid; j < nl; j += kPersThreads) s_span[j] = A.span[my_long[j]];
  __syncthreads();
  if (warp == 0) {
    int32_t run = 0;
    for (int32_t j0 = 0; j0 < nl; j0 += 32) {
      int32_t k = 0;
      if (j0 + lane < nl) {
        const int2 s = s_span[j0 + lane];
        const int32_t c = pers_chunk(s.y - s.x);
        k = (s.y - s.x + c - 1) / c;
      }
      int32_t v = k;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int32_t y = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o) v += y;
      }
      if (j0 + lane < nl) s_first[j0 + lane] = run + v - k;
      run += __shfl_sync(0xffffffffu, v, 31);
    }
    if (lane == 0) s_first[nl] = run;
  }
  __syncthreads();
  for (int32_t j = warp; j < nl; j += kPersWarps) {
    const int2 s = s_span[j];
    const int32_t c = pers_chunk(s.y - s.x), q0 = s_first[j], q1 = s_first[j + 1];
    for (int32_t q = q0 + lane; q < q1; q += 32) {
      const int32_t e0 = s.x + (q - q0) * c;
      s_edges[q] = make_int2(e0, min(s.y, e0 + c));
    }
  }

  // x_0 = 1/n and its contributions
  const float x0 = 1.0f / (float)n;
  if constexpr (!kProduct) {
    T* c0 = (T*)A.c[0];
    int32_t rows = 0, ends = 0;  // of the thread, without out-edges
    for (int32_t v = blockIdx.x * kPersThreads + tid; v < n; v += nblk * kPersThreads) {
      const float idg = A.inv_deg[v];
      store_rank(c0, v, x0 * idg);
      if (A.iters == 0) A.x[v] = x0;
      ++rows;
      if (idg == 0.f) ++ends;
    }
    rows = __reduce_add_sync(0xffffffffu, rows);
    ends = __reduce_add_sync(0xffffffffu, ends);
    if (lane == 0) {
      s_sum[0][warp] = fix60(x0) * (unsigned)rows;
      s_sum[1][warp] = fix60(x0) * (unsigned)ends;
      s_sum[2][warp] = 0ull;
    }
    add_sums(0);
  }
  if constexpr (kProduct) __syncthreads();  // (add_sums has one)
  const int32_t nchunks = s_first[nl];

  // a slice: this lane's row, its width and its first indices
  struct Slice {
    int32_t i, r, at, width;
    float inv;
    int32_t u[kPersSlice];
  };
  auto load_slice = [&](int32_t k) {  // the block's k-th
    Slice w;
    w.i = -1;
    w.r = w.at = w.width = 0;
    w.inv = 0.f;
    if (k < nsl) {
      const int32_t s = __ldg(my_slice + k);
      const int32_t i = A.n_long + 32 * s + lane, o0 = __ldg(A.off + s), o1 = __ldg(A.off + s + 1);
      w.at = o0 + lane;
      w.width = (o1 - o0) >> 5;
      if (i < n) {
        w.i = i;
        w.r = __ldg(A.row + i);
        w.inv = __ldg(A.inv + i);
      }
    }
#pragma unroll
    for (int j = 0; j < kPersSlice; ++j) w.u[j] = j < w.width ? __ldg(A.sell + w.at + 32 * j) : -1;
    return w;
  };
  const bool single = warp + kPersWarps >= nsl;  // the warp's one slice stays in its registers
  Slice cur = load_slice(warp);
  float cx = x0;
  if constexpr (!kProduct) barrier();

  for (int32_t it = 0; it < A.iters && !failed; ++it) {
    const T* cin = (const T*)A.c[it & 1];
    T* cout = (T*)A.c[(it & 1) ^ 1];
    const bool last = it + 1 == A.iters;
    // the step's coefficients (warp 0) beside the copy of the first H contributions
    if (warp == 0) {
      if (lane == 0 && kProduct) {
        const float m = __uint_as_float(__ldcg((const unsigned int*)(A.sums + 3 * (int64_t)it)));
        s_coef[0] = m > 0.f ? 1.0f / m : 0.f;
        s_coef[1] = 0.f;
      } else if (lane == 0) {
        // mass and dangling mass as sums of two floats (48 bits; the FP64 pipe
        // would take longer than the rest of the step), 1 / mass by a Newton
        // step on the FP32 reciprocal
        const float2 m = pers_pair(__ldcg(A.sums + 3 * (int64_t)it)), g = pers_pair(__ldcg(A.sums + 3 * (int64_t)it + 1));
        const float r0 = 1.0f / m.x;
        const float2 r = make_float2(r0, r0 * fmaf(-m.y, r0, fmaf(-m.x, r0, 1.0f)));
        const float2 a = pers_mul(make_float2(A.d_hi, A.d_lo), r);
        const float2 t = pers_mul(pers_mul(a, g), make_float2(A.in_hi, A.in_lo));
        s_coef[0] = a.x + a.y;
        s_coef[1] = pers_add(make_float2(A.t_hi, A.t_lo), t);
      }
    } else {
      const int4* src = reinterpret_cast<const int4*>(cin);
      int4* dst = reinterpret_cast<int4*>(s_c);
      constexpr int step = kPersThreads - 32;
      const int32_t nvec = H / (16 / (int)sizeof(T));  // H is a multiple of 8
      for (int32_t i0 = tid - 32; i0 < nvec; i0 += 4 * step) {
        int4 v[4];
#pragma unroll
        for (int k = 0; k < 4; ++k)
          if (i0 + k * step < nvec) v[k] = __ldcg(src + i0 + k * step);
#pragma unroll
        for (int k = 0; k < 4; ++k)
          if (i0 + k * step < nvec) dst[i0 + k * step] = v[k];
      }
    }
    __syncthreads();
    const float ca = s_coef[0], cb = s_coef[1];
    float mass = 0.f, dang = 0.f, res = 0.f, mass_c = 0.f, dang_c = 0.f;
    auto two = [](float& s, float& c, float v) {  // s + c += v
      const float t = s + v, b = t - s;
      c += (s - (t - b)) + (v - b);
      s = t;
    };
    auto finish = [&](int32_t i, int32_t r, float inv, float xo, float y) {
      const float xs = fmaf(ca, y, cb);
      A.xi[i] = xs;
      if (last) A.x[r] = xs;
      if (!last || kProduct) store_rank(cout, r, xs * inv);
      if constexpr (kProduct)
        mass = fmaxf(mass, xs);
      else
        two(mass, mass_c, xs);
      res += fabsf(xs - xo);
      if (inv == 0.0f) two(dang, dang_c, xs);
      return xs;
    };
    auto gather = [&](const auto& u) {
      constexpr int N = sizeof(u) / sizeof(int32_t);
      uint32_t b[N];
      float v[N];
#pragma unroll
      for (int k = 0; k < N; ++k) b[k] = pers_bits(s_addr, cin, u[k], H);
#pragma unroll
      for (int k = 0; k < N; ++k) v[k] = pers_value(b[k], cin);
#pragma unroll
      for (int o = 1; o < N; o *= 2)
#pragma unroll
        for (int k = 0; k < N; k += 2 * o) v[k] += v[k + o];
      return v[0];
    };
    // the chunks of the block's long rows, a warp each, the next indices loaded
    // while the current ones are gathered
    if (warp < nchunks) {
      int32_t u[kPersIdx], q = warp;
      int2 s = s_edges[q];
      auto load = [&](int32_t e) {
#pragma unroll
        for (int k = 0; k < kPersIdx; ++k) u[k] = e + 32 * k < s.y ? __ldg(A.row_idx + e + 32 * k) : -1;
      };
      int32_t e = s.x + lane;
      load(e);
      float y = 0.f;
      for (;;) {
        int32_t c[kPersIdx];
#pragma unroll
        for (int k = 0; k < kPersIdx; ++k) c[k] = u[k];
        e += 32 * kPersIdx;
        const int32_t done = q;
        const bool end = e - lane >= s.y;  // the chunk's last indices: on to the next chunk
        if (end) {
          q += kPersWarps;
          if (q < nchunks) {
            s = s_edges[q];
            e = s.x + lane;
          }
        }
        if (q < nchunks) load(e);
        y += gather(c);
        if (end) {
          y = warp_sum(y);
          if (lane == 0) s_chunk[done] = y;
          y = 0.f;
          if (q >= nchunks) break;
        }
      }
    }
    // the warp's slices, loading ahead alike
    for (int32_t s = warp; s < nsl; s += kPersWarps) {
      const int32_t i = cur.i, r = cur.r, at = cur.at, width = cur.width;
      const float inv = cur.inv, xo = single ? cx : it > 0 && i >= 0 ? A.xi[i] : x0;
      int32_t u[kPersSlice];
#pragma unroll
      for (int k = 0; k < kPersSlice; ++k) u[k] = cur.u[k];
      float y = 0.f;
      for (int32_t j = kPersSlice;; j += kPersSlice) {
        int32_t c[kPersSlice];
#pragma unroll
        for (int k = 0; k < kPersSlice; ++k) c[k] = u[k];
        const bool end = j >= width;
        if (!end) {
#pragma unroll
          for (int k = 0; k < kPersSlice; ++k) u[k] = j + k < width ? __ldg(A.sell + at + 32 * (j + k)) : -1;
        } else if (!single) {
          cur = load_slice(s + kPersWarps < nsl ? s + kPersWarps : warp);
        }
        y += gather(c);
        if (end) break;
      }
      if (i >= 0) cx = finish(i, r, inv, xo, y);
    }
    if (nl > 0) {
      __syncthreads();
      if (32 * warp < nl) {
        const bool mine = tid < nl;
        int32_t i = 0, r = 0, q = 0, q1 = 0;
        float inv = 0.f, xo = x0, y = 0.f;
        if (mine) {
          i = __ldg(my_long + tid);
          r = __ldg(A.row + i);
          inv = __ldg(A.inv + i);
          if (it > 0) xo = A.xi[i];
          q = s_first[tid];
          q1 = s_first[tid + 1];
        }
        // (by eights: one after another, a hub's 64 equal chunk sums round alike, 6e-7
        // of them at an in-degree of 20,000 where the pull kernels have 3e-8)
        for (; q < q1; q += 8) {
          float z[8];
#pragma unroll
          for (int k = 0; k < 8; ++k) z[k] = q + k < q1 ? s_chunk[q + k] : 0.f;
          y += ((z[0] + z[1]) + (z[2] + z[3])) + ((z[4] + z[5]) + (z[6] + z[7]));
        }
        // (rows have different numbers of chunks: without this the lanes of each
        // number may finish by themselves, one number after another, which took
        // 10 us of a step)
        __syncwarp();
        if (mine) finish(i, r, inv, xo, y);
      }
    }
    if constexpr (kProduct) {
      add_max(it + 1, mass);
      return;
    }
    mass = warp_sum(mass);
    dang = warp_sum(dang);
    res = warp_sum(res);
    if (lane == 0) {
      s_sum[0][warp] = fix60(mass);
      s_sum[1][warp] = fix60(dang);
      s_sum[2][warp] = fix60(res);
    }
    if (!single) {
      mass_c = warp_sum(mass_c);
      dang_c = warp_sum(dang_c);
      if (lane == 0) {
        s_sum[0][warp] += fix60_signed(mass_c);
        s_sum[1][warp] += fix60_signed(dang_c);
      }
    }
    add_sums(it + 1);
    barrier();
  }

  // ranks by caller id; x_0 of a call without steps was written above
  for (int32_t v = blockIdx.x * kPersThreads + tid; v < n; v += nblk * kPersThreads)
    A.out[v] = failed ? __int_as_float(0x7fffffff) : __ldcg(A.x + A.old2new[v]);
  if (blockIdx.x == 0 && tid < 3) A.log_row[tid] = fix60_value(__ldcg(A.sums + 3 * (int64_t)A.iters + tid));
}

// ---- the layout -------------------------------------------------------------

// Sort keys of the rows by descending in-degree, and how many rows have each
// in-degree up to kPersShort (count[kPersShort + 1]: more).
__global__ void persist_keys_kernel(const int32_t* __restrict__ col_ptr, int32_t n, int b, int32_t max_in,
                                    uint64_t* __restrict__ keys, int32_t* __restrict__ count) {
  __shared__ int32_t s_count[kPersShort + 2];
  for (int i = threadIdx.x; i < kPersShort + 2; i += blockDim.x) s_count[i] = 0;
  __syncthreads();
  for (int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p < n; p += (int64_t)gridDim.x * blockDim.x) {
    const int32_t deg = col_ptr[p + 1] - col_ptr[p];
    keys[p] = (uint64_t)(max_in - deg) << b | (uint64_t)p;
    atomicAdd(&s_count[min(deg, kPersShort + 1)], 1);
  }
  __syncthreads();
  for (int i = threadIdx.x; i < kPersShort + 2; i += blockDim.x)
    if (s_count[i]) atomicAdd(count + i, s_count[i]);
}

// The rows in order with their inverse degrees, the long rows' edges and the
// slices (a warp each).
__global__ void persist_layout_kernel(const uint64_t* __restrict__ sorted, int b, const int32_t* __restrict__ col_ptr,
                                      const int32_t* __restrict__ row_idx, const float* __restrict__ inv_deg,
                                      int32_t n, int32_t n_long, int32_t nslices, const int32_t* __restrict__ off,
                                      int32_t* __restrict__ row, float* __restrict__ inv, int2* __restrict__ span,
                                      int32_t* __restrict__ sell) {
  const int64_t t0 = blockIdx.x * (int64_t)blockDim.x + threadIdx.x, nt = (int64_t)gridDim.x * blockDim.x;
  const uint64_t mask = (1ull << b) - 1;
  for (int64_t i = t0; i < n; i += nt) {
    const int32_t r = (int32_t)(sorted[i] & mask);
    row[i] = r;
    inv[i] = inv_deg[r];
    if (i < n_long) span[i] = make_int2(col_ptr[r], col_ptr[r + 1]);
  }
  const int lane = threadIdx.x & 31;
  for (int64_t s = t0 >> 5; s < nslices; s += nt >> 5) {
    const int64_t i = n_long + 32 * s + lane;
    int32_t e0 = 0, deg = 0;
    if (i < n) {
      const int32_t r = (int32_t)(sorted[i] & mask);
      e0 = col_ptr[r];
      deg = col_ptr[r + 1] - e0;
    }
    const int32_t o0 = off[s], width = (off[s + 1] - o0) >> 5;
    for (int32_t j = 0; j < width; ++j) sell[o0 + 32 * j + lane] = j < deg ? row_idx[e0 + j] : -1;
  }
}

}  // namespace gpr
