// Chunked vector kernels over the [N][8] Krylov vectors: work split, 16-byte accesses,
// block dot products and Gram-Schmidt updates (kernels_vec.cu, krylov_dev.cu).
#pragma once

#include "device_common.cuh"
#include "pse_internal.cuh"

namespace pse {
namespace {

// The chunked vector kernels: block b covers `chunk` elements of the [N][8]
// vectors of one suspension (blocks of suspension s start at blk0[s]).
struct Chunk {
  int s;
  int64_t beg, end;
};
struct VecArgs {
  const SysDev *sys;
  const int *blk0, *active;
  int nsys, chunk;
};

__device__ __forceinline__ Chunk chunk_of(const VecArgs &va, int b) {
  Chunk ch;
  ch.s = find_sys(va.blk0, va.nsys, b);
  const SysDev &q = va.sys[ch.s];
  ch.beg = 8 * q.p0 + (int64_t)(b - q.blk0) * va.chunk;
  const int64_t lim = 8 * (q.p0 + q.N);
  ch.end = ch.beg + va.chunk < lim ? ch.beg + va.chunk : lim;
  return ch;
}

inline VecArgs vec_args(const pse_ctx *c) {
  VecArgs v;
  v.sys = c->d_sys;
  v.blk0 = c->d_blk0;
  v.active = c->d_active;
  v.nsys = c->nsys;
  v.chunk = c->vchunk;
  return v;
}

// 16-byte vectors of the chunked kernels (a chunk holds a multiple of 8 elements
// and starts 32-byte aligned): 4 floats or 2 doubles per access.
template <typename T> struct V16;
template <> struct V16<float> {
  using t = float4;
  static constexpr int n = 4;
  static __device__ __forceinline__ void get(const float4 &v, float a[4]) {
    a[0] = v.x;
    a[1] = v.y;
    a[2] = v.z;
    a[3] = v.w;
  }
  static __device__ __forceinline__ float4 put(const float a[4]) { return make_float4(a[0], a[1], a[2], a[3]); }
};
template <> struct V16<double> {
  using t = double2;
  static constexpr int n = 2;
  static __device__ __forceinline__ void get(const double2 &v, double a[2]) {
    a[0] = v.x;
    a[1] = v.y;
  }
  static __device__ __forceinline__ double2 put(const double a[2]) { return make_double2(a[0], a[1]); }
};

constexpr int DOT_NT = 256, DOT_ROWS = 8;

// acc[r] += rows[r0 + r] . w over the block's chunk, r < nr <= DOT_ROWS; each
// thread keeps VEC_UNROLL independent 16-byte loads per row in flight.  w may be written
// by the same kernel (each thread reads the elements it wrote).
constexpr int VEC_UNROLL = 4;
template <typename T>
__device__ __forceinline__ void chunk_dots(const Chunk &ch, const T *__restrict__ rows, int64_t stride, int r0, int nr,
                                           const T *w, T acc[DOT_ROWS]) {
  using V = V16<T>;
  using VT = typename V::t;
#pragma unroll
  for (int r = 0; r < DOT_ROWS; ++r) acc[r] = 0;
  const int64_t step = (int64_t)blockDim.x * V::n;
  for (int64_t e0 = ch.beg + (int64_t)threadIdx.x * V::n; e0 < ch.end; e0 += VEC_UNROLL * step) {
    T wv[VEC_UNROLL][V::n];
#pragma unroll
    for (int u = 0; u < VEC_UNROLL; ++u) {
      const int64_t e = e0 + u * step;
      if (e < ch.end) V::get(*(const VT *)(w + e), wv[u]);
      else
#pragma unroll
        for (int i = 0; i < V::n; ++i) wv[u][i] = 0;
    }
#pragma unroll
    for (int r = 0; r < DOT_ROWS; ++r)
      if (r < nr) {
        const T *row = rows + (r0 + r) * stride;
        T x[VEC_UNROLL][V::n];
#pragma unroll
        for (int u = 0; u < VEC_UNROLL; ++u) {
          const int64_t e = e0 + u * step;
          if (e < ch.end) V::get(*(const VT *)(row + e), x[u]);
          else
#pragma unroll
            for (int i = 0; i < V::n; ++i) x[u][i] = 0;
        }
#pragma unroll
        for (int u = 0; u < VEC_UNROLL; ++u)
#pragma unroll
          for (int i = 0; i < V::n; ++i) acc[r] += x[u][i] * wv[u][i];
      }
  }
}

// partial[(r0 + r) * nblk + b] = sum over block b of acc[r] (FP64 across threads), r < nr.
// The eight sums of a warp are taken together: each exchange halves the rows a lane
// keeps, so a warp spends 8 conversions and 9 FP64 additions on them and not 48 (the
// FP64 unit, one warp instruction in 16 cycles, set the time of these kernels on small
// vectors: 31.4 -> 21.4 us per launch at N = 64000, 11 rows, 500 blocks).
template <typename T>
__device__ __forceinline__ void block_sums(const T acc[DOT_ROWS], int nr, double *partial, int64_t nblk, int b, int r0,
                                           double red[DOT_ROWS][DOT_NT / 32]) {
  static_assert(DOT_ROWS == 8 && DOT_NT == 256, "lane mapping");
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const bool b4 = lane & 16, b3 = lane & 8, b2 = lane & 4;
  double k4[4], k2[2];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const T keep = b4 ? acc[i + 4] : acc[i], send = b4 ? acc[i] : acc[i + 4];
    k4[i] = (double)keep + (double)__shfl_xor_sync(0xffffffffu, send, 16);
  }
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    const double keep = b3 ? k4[i + 2] : k4[i], send = b3 ? k4[i] : k4[i + 2];
    k2[i] = keep + __shfl_xor_sync(0xffffffffu, send, 8);
  }
  double v = (b2 ? k2[1] : k2[0]) + __shfl_xor_sync(0xffffffffu, b2 ? k2[0] : k2[1], 4);
  v += __shfl_xor_sync(0xffffffffu, v, 2);
  v += __shfl_xor_sync(0xffffffffu, v, 1);
  if ((lane & 3) == 0) red[4 * b4 + 2 * b3 + b2][wid] = v;
  __syncthreads();
  if (threadIdx.x < 64) {  // row threadIdx.x / 8, warp threadIdx.x % 8
    double sum = red[threadIdx.x >> 3][threadIdx.x & 7];
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
    const int r = threadIdx.x >> 3;
    if ((threadIdx.x & 7) == 0 && r < nr) partial[(r0 + r) * nblk + b] = sum;
  }
  __syncthreads();
}

// w[e] -= sum_r cs[r] rows[r][e] over the block's chunk, r < nr; returns this thread's
// sum of the new w[e]^2.
template <typename T>
__device__ __forceinline__ T chunk_sub(const Chunk &ch, T *w, const T *__restrict__ rows, int64_t stride, int nr,
                                       const T *cs) {
  using V = V16<T>;
  using VT = typename V::t;
  const int64_t step = (int64_t)blockDim.x * V::n;
  T sq = 0;
  for (int64_t e0 = ch.beg + (int64_t)threadIdx.x * V::n; e0 < ch.end; e0 += VEC_UNROLL * step) {
    T sum[VEC_UNROLL][V::n];
#pragma unroll
    for (int u = 0; u < VEC_UNROLL; ++u)
#pragma unroll
      for (int i = 0; i < V::n; ++i) sum[u][i] = 0;
    for (int r = 0; r < nr; ++r) {
      const T *row = rows + r * stride;
      T x[VEC_UNROLL][V::n];
#pragma unroll
      for (int u = 0; u < VEC_UNROLL; ++u) {
        const int64_t e = e0 + u * step;
        if (e < ch.end) V::get(*(const VT *)(row + e), x[u]);
        else
#pragma unroll
          for (int i = 0; i < V::n; ++i) x[u][i] = 0;
      }
#pragma unroll
      for (int u = 0; u < VEC_UNROLL; ++u)
#pragma unroll
        for (int i = 0; i < V::n; ++i) sum[u][i] += cs[r] * x[u][i];
    }
#pragma unroll
    for (int u = 0; u < VEC_UNROLL; ++u) {
      const int64_t e = e0 + u * step;
      if (e >= ch.end) continue;
      T out[V::n];
      V::get(*(const VT *)(w + e), out);
#pragma unroll
      for (int i = 0; i < V::n; ++i) {
        out[i] -= sum[u][i];
        sq += out[i] * out[i];
      }
      *(VT *)(w + e) = V::put(out);
    }
  }
  return sq;
}

}  // namespace
}  // namespace pse
