// Vector kernels: user-order <-> sorted-order permutations, in-kernel noise for
// the Lanczos start vector, Krylov inner products and combinations, and the
// position updates of the mid-point scheme (Sec. 3.4).
//
// Inner products in the mixed form: each thread sums its FP32 products over a
// short stretch of the vector, the cross-thread and cross-block sums are FP64.
// Inner products and combinations are per suspension: every block covers one
// chunk of one suspension's vector, results and coefficients live at
// d_coef[s * COEF_STRIDE + ...], and suspensions marked inactive are skipped.
#include <algorithm>

#include "device_common.cuh"
#include "pse_internal.cuh"
#include "vec_common.cuh"

namespace pse {
namespace {

// Sorted rows from user-order F and S (NULL: zero); with vcell also into cell-list order as the
// pair sum reads them (pos: a particle's place in that list).
template <typename T>
__global__ void k_gather_in(int64_t N, const int *perm, const T *F, const T *S, T *out, T *vcell, const int *pos) {
  using T4 = typename V4<T>::t;
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= N) return;
  const int64_t u = perm[i];
  T v[8];
#pragma unroll
  for (int m = 0; m < 3; ++m) v[m] = F ? F[3 * u + m] : (T)0;
#pragma unroll
  for (int m = 0; m < 5; ++m) v[3 + m] = S ? S[5 * u + m] : (T)0;
  T4 lo, hi;
  lo.x = v[0], lo.y = v[1], lo.z = v[2], lo.w = v[3];
  hi.x = v[4], hi.y = v[5], hi.z = v[6], hi.w = v[7];
  store_row((T4 *)out, i, lo, hi);
  if (vcell) {
    cell_row(lo, hi);
    store_row((T4 *)vcell, pos[i], lo, hi);
  }
}

// out = [F (user order, NULL: 0), slots 3..7 of s8 (sorted)]
template <typename T>
__global__ void k_gather_join(int64_t N, const int *perm, const T *F, const T *s8, T *out) {
  const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= 8 * N) return;
  const int64_t i = e >> 3;
  const int m = (int)(e & 7);
  out[e] = m < 3 ? (F ? F[3 * (int64_t)perm[i] + m] : (T)0) : s8[e];
}

// out = [0, -(slots 3..7 of v) - (those of sub)]; rows of v through perm when it is given
template <typename T>
__global__ void k_rhs(int64_t N, const int *perm, const T *v, const T *sub, T *out) {
  const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= 8 * N) return;
  const int64_t i = e >> 3;
  const int m = (int)(e & 7);
  T x = 0;
  if (m >= 3) {
    x = -v[8 * (perm ? (int64_t)perm[i] : i) + m];
    if (sub) x -= sub[e];
  }
  out[e] = x;
}

// Status words (kernels_config.cu): non-finite positions, list overflow, non-finite inputs.
__device__ __forceinline__ bool status_set(const int *flag) { return flag && (flag[0] | flag[1] | flag[2]); }

__global__ void k_commit(int64_t n, const double *__restrict__ src, double *__restrict__ dst, const int *flag) {
  const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e < n && !status_set(flag)) dst[e] = src[e];
}

template <typename T>
__global__ void k_scatter_out(int64_t N, const int *perm, const T *in, T *U, T *E, T scale, const int *flag) {
  int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= N || status_set(flag)) return;
  int u = perm[i];
  const T *v = in + 8 * (size_t)i;
  if (U)
    for (int m = 0; m < 3; ++m) U[3 * (size_t)u + m] = scale * v[m];
  if (E)
    for (int m = 0; m < 5; ++m) E[5 * (size_t)u + m] = scale * v[3 + m];
}

// 12-slot sorted rows [F(3), L(3), S(5), 0] from user-order arrays (any may be NULL: zero).
template <typename T>
__global__ void k_gather12(int64_t N, const int *perm, const T *F, const T *L, const T *S, T *out) {
  int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= N) return;
  const int64_t u = perm[i];
  T *o = out + 12 * (size_t)i;
  for (int m = 0; m < 3; ++m) o[m] = F ? F[3 * u + m] : (T)0;
  for (int m = 0; m < 3; ++m) o[3 + m] = L ? L[3 * u + m] : (T)0;
  for (int m = 0; m < 5; ++m) o[6 + m] = S ? S[5 * u + m] : (T)0;
  o[11] = (T)0;
}

// user-order U, Omega, E (any may be NULL: not written) from 12-slot sorted rows.
template <typename T>
__global__ void k_scatter12(int64_t N, const int *perm, const T *in, T *U, T *Om, T *E) {
  int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= N) return;
  const int64_t u = perm[i];
  const T *v = in + 12 * (size_t)i;
  if (U)
    for (int m = 0; m < 3; ++m) U[3 * u + m] = v[m];
  if (Om)
    for (int m = 0; m < 3; ++m) Om[3 * u + m] = v[3 + m];
  if (E)
    for (int m = 0; m < 5; ++m) E[5 * u + m] = v[6 + m];
}

template <typename T>
__global__ void k_gather8(int64_t N, const int *perm, const T *in, T *out) {
  int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= 8 * N) return;
  int64_t i = e >> 3;
  int c = (int)(e & 7);
  out[e] = in[8 * (size_t)perm[i] + c];
}

template <typename T>
__global__ void k_scatter8(int64_t N, const int *perm, const T *in, T *out, T scale) {
  int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= 8 * N) return;
  int64_t i = e >> 3;
  int c = (int)(e & 7);
  out[8 * (size_t)perm[i] + c] = scale * in[e];
}

// (seed, counter) come from rng[0..2) when rng is given (a captured graph reads them at launch)
template <typename T>
__global__ void k_philox_w1(int64_t N, const int *perm, uint64_t seed, uint64_t counter, const uint64_t *rng, T *out) {
  int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= 8 * N) return;
  if (rng) {
    seed = rng[0];
    counter = rng[1];
  }
  int64_t i = e >> 3;
  int c = (int)(e & 7);
  T z0, z1;
  normal_pair<T>(seed, counter, 1u, 8ull * (uint64_t)perm[i] + (uint64_t)c, z0, z1);
  out[e] = z0;
}

// w[e] = (SET ? 0 : w[e]) + sgn * sum_r coef[s][r] rows[r][e], r < nrows (or nrows_s[s])
template <typename T, bool SET>
__global__ void k_combine(VecArgs va, T *w, const T *__restrict__ rows, int64_t stride, int nrows,
                          const int *__restrict__ nrows_s, const double *__restrict__ coef, T sgn) {
  using V = V16<T>;
  using VT = typename V::t;
  __shared__ T cs[MAX_ROWS];
  const Chunk ch = chunk_of(va, blockIdx.x);
  if (!va.active[ch.s]) return;
  int nr = nrows;
  if (nrows_s) nr = min(nr, nrows_s[ch.s]);
  const double *cf = coef + (size_t)ch.s * COEF_STRIDE;
  for (int r = threadIdx.x; r < nr; r += blockDim.x) cs[r] = (T)cf[r];
  __syncthreads();
  const int64_t step = (int64_t)blockDim.x * V::n;
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
      if (SET) {
#pragma unroll
        for (int i = 0; i < V::n; ++i) out[i] = sgn * sum[u][i];
      } else {
        V::get(*(const VT *)(w + e), out);
#pragma unroll
        for (int i = 0; i < V::n; ++i) out[i] += sgn * sum[u][i];
      }
      *(VT *)(w + e) = V::put(out);
    }
  }
}

__device__ __forceinline__ double wrapL(double x, double L) {
  if (x >= 0.0 && x < L) return x;  // already inside: fmod would return x itself
  x = fmod(x, L);
  if (x < 0) x += L;
  if (x >= L) x = 0.0;
  return x;
}

template <typename T>
__global__ void k_midpoint(VecArgs va, const int64_t *__restrict__ p0, int64_t N, const double *x0, const T *B,
                           double fac, double *xo) {
  int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= 3 * N) return;
  int64_t u = e / 3;
  int d = (int)(e % 3);
  const SysDev &sd = va.sys[find_sys(p0, va.nsys, u)];
  const double x = x0[e] + fac * (double)B[8 * (size_t)u + d];
  xo[e] = sd.def ? x : wrapL(x, sd.L);  // on a deformed lattice the set-up wraps lattice coordinates
}

template <typename T>
__global__ void k_final(VecArgs va, const int64_t *__restrict__ p0, int64_t N, const int *inv, const double *x0,
                        const T *B, const T *Us, double dt, double *xo) {
  int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= 3 * N) return;
  int64_t u = e / 3;
  int d = (int)(e % 3);
  const SysDev &sd = va.sys[find_sys(p0, va.nsys, u)];
  double U = (double)B[8 * (size_t)u + d] + (double)Us[8 * (size_t)inv[u] + d];
  const double x = x0[e] + dt * U;
  xo[e] = sd.def ? x : wrapL(x, sd.L);
}

// Positions of a deformed cell (Sec. 2.3.3) wrapped per particle: x = A (A^{-1} x mod L).
__global__ void k_wrap_lattice(VecArgs va, const int64_t *__restrict__ p0, int64_t N, double *x) {
  const int64_t u = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (u >= N) return;
  const SysDev &sd = va.sys[find_sys(p0, va.nsys, u)];
  if (!sd.def) return;
  double *xu = x + 3 * u;
  double z[3];
#pragma unroll
  for (int i = 0; i < 3; ++i) z[i] = wrapL(sd.Ai[3 * i] * xu[0] + sd.Ai[3 * i + 1] * xu[1] + sd.Ai[3 * i + 2] * xu[2], sd.L);
#pragma unroll
  for (int i = 0; i < 3; ++i) xu[i] = sd.A[3 * i] * z[0] + sd.A[3 * i + 1] * z[1] + sd.A[3 * i + 2] * z[2];
}

// The direction W of the random finite difference as user-order 8-slot rows
// (slots 0..2, the rest zero): from wt (N x 3) or in-kernel (Philox stream 3,
// index 3 u + d, first normal of the pair).
template <typename T>
__global__ void k_rfd_noise(int64_t N, const T *wt, uint64_t seed, uint64_t counter, T *W8) {
  int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= 8 * N) return;
  const int64_t u = e >> 3;
  const int d = (int)(e & 7);
  T v = (T)0;
  if (d < 3) {
    if (wt) {
      v = wt[3 * u + d];
    } else {
      T z1;
      normal_pair<T>(seed, counter, 3u, 3ull * (uint64_t)u + (uint64_t)d, v, z1);
    }
  }
  W8[e] = v;
}

// x_{k+1} = x_k + dt (U^B + U_0 + fac (R_+ - R_-)), wrapped (all rows user order, slots 0..2).
template <typename T>
__global__ void k_rfd_final(VecArgs va, const int64_t *__restrict__ p0, int64_t N, const double *x0, const T *B,
                            const T *U0, const T *Rp, const T *Rm, double dt, double fac, double *xo) {
  int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= 3 * N) return;
  const int64_t u = e / 3;
  const int d = (int)(e % 3);
  const SysDev &sd = va.sys[find_sys(p0, va.nsys, u)];
  const size_t r = 8 * (size_t)u + d;
  const double U = (double)B[r] + (double)U0[r] + fac * ((double)Rp[r] - (double)Rm[r]);
  const double x = x0[e] + dt * U;
  xo[e] = sd.def ? x : wrapL(x, sd.L);
}

template <typename T>
__global__ void k_finite(const T *p, int64_t n, int *bad) {
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < n; e += (int64_t)gridDim.x * blockDim.x)
    if (!isfinite((double)p[e])) {
      atomicOr(bad, 1);
      return;
    }
}

unsigned grid_for(int64_t n, int nt = 256) { return (unsigned)ceil_div(n, nt); }

}  // namespace

#define DISPATCH(c, EXPR_F, EXPR_D) \
  do {                              \
    if ((c)->prec == PSE_MIXED) {   \
      EXPR_F;                       \
    } else {                        \
      EXPR_D;                       \
    }                               \
  } while (0)

int *next_queue(pse_ctx *c) { return c->d_queue + (c->queue_slot++ & 63); }

pse_status gather_in(pse_ctx *c, const void *F, const void *S, void *vout, bool cells, cudaStream_t s) {
  StageTimer timer(c, PSE_STAGE_VECTOR, s);
  c->nlaunch += 1;
  int64_t N = c->p.N;
  void *vc = cells ? c->d_vcell : nullptr;
  DISPATCH(c, (k_gather_in<float><<<grid_for(N), 256, 0, s>>>(N, c->d_perm, (const float *)F, (const float *)S, (float *)vout, (float *)vc, c->d_cell_key)),
           (k_gather_in<double><<<grid_for(N), 256, 0, s>>>(N, c->d_perm, (const double *)F, (const double *)S, (double *)vout, (double *)vc, c->d_cell_key)));
  PSE_CUDA_TRY(c, cudaGetLastError());
  return PSE_OK;
}

pse_status gather_join(pse_ctx *c, const void *F, const void *s8, void *vout, cudaStream_t s) {
  StageTimer timer(c, PSE_STAGE_VECTOR, s);
  c->nlaunch += 1;
  int64_t N = c->p.N;
  DISPATCH(c, (k_gather_join<float><<<grid_for(8 * N), 256, 0, s>>>(N, c->d_perm, (const float *)F, (const float *)s8, (float *)vout)),
           (k_gather_join<double><<<grid_for(8 * N), 256, 0, s>>>(N, c->d_perm, (const double *)F, (const double *)s8, (double *)vout)));
  PSE_CUDA_TRY(c, cudaGetLastError());
  return PSE_OK;
}

pse_status krylov_rhs(pse_ctx *c, const void *v8, bool user, const void *sub8, void *vout, cudaStream_t s) {
  StageTimer timer(c, PSE_STAGE_VECTOR, s);
  c->nlaunch += 1;
  int64_t N = c->p.N;
  const int *perm = user ? c->d_perm : nullptr;
  DISPATCH(c, (k_rhs<float><<<grid_for(8 * N), 256, 0, s>>>(N, perm, (const float *)v8, (const float *)sub8, (float *)vout)),
           (k_rhs<double><<<grid_for(8 * N), 256, 0, s>>>(N, perm, (const double *)v8, (const double *)sub8, (double *)vout)));
  PSE_CUDA_TRY(c, cudaGetLastError());
  return PSE_OK;
}

pse_status commit_positions(pse_ctx *c, const double *src, double *dst, cudaStream_t s) {
  StageTimer timer(c, PSE_STAGE_VECTOR, s);
  c->nlaunch += 1;
  k_commit<<<grid_for(3 * c->p.N), 256, 0, s>>>(3 * c->p.N, src, dst, c->d_flag);
  PSE_CUDA_TRY(c, cudaGetLastError());
  return PSE_OK;
}

pse_status gather12(pse_ctx *c, const void *F, const void *L, const void *S, void *vout, cudaStream_t s) {
  StageTimer timer(c, PSE_STAGE_VECTOR, s);
  c->nlaunch += 1;
  int64_t N = c->p.N;
  DISPATCH(c, (k_gather12<float><<<grid_for(N), 256, 0, s>>>(N, c->d_perm, (const float *)F, (const float *)L, (const float *)S, (float *)vout)),
           (k_gather12<double><<<grid_for(N), 256, 0, s>>>(N, c->d_perm, (const double *)F, (const double *)L, (const double *)S, (double *)vout)));
  PSE_CUDA_TRY(c, cudaGetLastError());
  return PSE_OK;
}

pse_status scatter12(pse_ctx *c, const void *vin, void *U, void *Om, void *E, cudaStream_t s) {
  StageTimer timer(c, PSE_STAGE_VECTOR, s);
  c->nlaunch += 1;
  int64_t N = c->p.N;
  DISPATCH(c, (k_scatter12<float><<<grid_for(N), 256, 0, s>>>(N, c->d_perm, (const float *)vin, (float *)U, (float *)Om, (float *)E)),
           (k_scatter12<double><<<grid_for(N), 256, 0, s>>>(N, c->d_perm, (const double *)vin, (double *)U, (double *)Om, (double *)E)));
  PSE_CUDA_TRY(c, cudaGetLastError());
  return PSE_OK;
}

pse_status scatter_out(pse_ctx *c, const void *vin, void *U, void *E, double scale, cudaStream_t s, bool guard) {
  StageTimer timer(c, PSE_STAGE_VECTOR, s);
  c->nlaunch += 1;
  int64_t N = c->p.N;
  const int *flag = guard ? c->d_flag : nullptr;
  DISPATCH(c, (k_scatter_out<float><<<grid_for(N), 256, 0, s>>>(N, c->d_perm, (const float *)vin, (float *)U, (float *)E, (float)scale, flag)),
           (k_scatter_out<double><<<grid_for(N), 256, 0, s>>>(N, c->d_perm, (const double *)vin, (double *)U, (double *)E, scale, flag)));
  PSE_CUDA_TRY(c, cudaGetLastError());
  return PSE_OK;
}

pse_status gather_user8(pse_ctx *c, const void *user8, void *vout, cudaStream_t s) {
  StageTimer timer(c, PSE_STAGE_VECTOR, s);
  c->nlaunch += 1;
  int64_t N = c->p.N;
  DISPATCH(c, (k_gather8<float><<<grid_for(8 * N), 256, 0, s>>>(N, c->d_perm, (const float *)user8, (float *)vout)),
           (k_gather8<double><<<grid_for(8 * N), 256, 0, s>>>(N, c->d_perm, (const double *)user8, (double *)vout)));
  PSE_CUDA_TRY(c, cudaGetLastError());
  return PSE_OK;
}

pse_status scatter_user8(pse_ctx *c, const void *vin, void *user8, double scale, cudaStream_t s) {
  StageTimer timer(c, PSE_STAGE_VECTOR, s);
  c->nlaunch += 1;
  int64_t N = c->p.N;
  DISPATCH(c, (k_scatter8<float><<<grid_for(8 * N), 256, 0, s>>>(N, c->d_perm, (const float *)vin, (float *)user8, (float)scale)),
           (k_scatter8<double><<<grid_for(8 * N), 256, 0, s>>>(N, c->d_perm, (const double *)vin, (double *)user8, scale)));
  PSE_CUDA_TRY(c, cudaGetLastError());
  return PSE_OK;
}

pse_status philox_w1(pse_ctx *c, uint64_t seed, uint64_t counter, void *vout, cudaStream_t s) {
  StageTimer timer(c, PSE_STAGE_VECTOR, s);
  c->nlaunch += 1;
  int64_t N = c->p.N;
  const uint64_t *rng = c->capturing ? c->d_rng : nullptr;
  DISPATCH(c, (k_philox_w1<float><<<grid_for(8 * N), 256, 0, s>>>(N, c->d_perm, seed, counter, rng, (float *)vout)),
           (k_philox_w1<double><<<grid_for(8 * N), 256, 0, s>>>(N, c->d_perm, seed, counter, rng, (double *)vout)));
  PSE_CUDA_TRY(c, cudaGetLastError());
  return PSE_OK;
}

// w -= sum_r coef[s][off + r] rows[r]  (r < nrows)
pse_status combine_sub(pse_ctx *c, void *w, const void *rows, int nrows, int off, cudaStream_t s) {
  StageTimer timer(c, PSE_STAGE_VECTOR, s);
  const int64_t n = 8 * c->p.N;
  const unsigned nb = (unsigned)c->nvblk;
  VecArgs va = vec_args(c);
  for (int r0 = 0; r0 < nrows; r0 += 128) {
    int nr = std::min(128, nrows - r0);
    c->nlaunch += 1;
    DISPATCH(c, (k_combine<float, false><<<nb, 256, 0, s>>>(va, (float *)w, (const float *)rows + (size_t)r0 * n, n, nr, nullptr, c->d_coef + off + r0, -1.0f)),
             (k_combine<double, false><<<nb, 256, 0, s>>>(va, (double *)w, (const double *)rows + (size_t)r0 * n, n, nr, nullptr, c->d_coef + off + r0, -1.0)));
  }
  PSE_CUDA_TRY(c, cudaGetLastError());
  return PSE_OK;
}

// y = sum_r coef[s][off + r] rows[r]  (r < d_nrows[s] <= maxrows <= 128)
pse_status combine_set(pse_ctx *c, void *y, const void *rows, const int *d_nrows, int maxrows, int off,
                       cudaStream_t s) {
  StageTimer timer(c, PSE_STAGE_VECTOR, s);
  const int64_t n = 8 * c->p.N;
  const unsigned nb = (unsigned)c->nvblk;
  VecArgs va = vec_args(c);
  if (maxrows > MAX_ROWS) {
    c->err = "too many Krylov vectors";
    return PSE_ERR_INVALID_ARG;
  }
  c->nlaunch += 1;
  DISPATCH(c, (k_combine<float, true><<<nb, 256, 0, s>>>(va, (float *)y, (const float *)rows, n, maxrows, d_nrows, c->d_coef + off, 1.0f)),
           (k_combine<double, true><<<nb, 256, 0, s>>>(va, (double *)y, (const double *)rows, n, maxrows, d_nrows, c->d_coef + off, 1.0)));
  PSE_CUDA_TRY(c, cudaGetLastError());
  return PSE_OK;
}

pse_status midpoint(pse_ctx *c, const double *x0, const void *B_user, double fac, double *xout, cudaStream_t s) {
  StageTimer timer(c, PSE_STAGE_VECTOR, s);
  c->nlaunch += 1;
  int64_t N = c->p.N;
  VecArgs va = vec_args(c);
  DISPATCH(c, (k_midpoint<float><<<grid_for(3 * N), 256, 0, s>>>(va, c->d_p0, N, x0, (const float *)B_user, fac, xout)),
           (k_midpoint<double><<<grid_for(3 * N), 256, 0, s>>>(va, c->d_p0, N, x0, (const double *)B_user, fac, xout)));
  PSE_CUDA_TRY(c, cudaGetLastError());
  return PSE_OK;
}

pse_status final_update(pse_ctx *c, const double *x0, const void *B_user, const void *U_sorted, double dt,
                        double *xout, cudaStream_t s) {
  StageTimer timer(c, PSE_STAGE_VECTOR, s);
  c->nlaunch += 1;
  int64_t N = c->p.N;
  VecArgs va = vec_args(c);
  DISPATCH(c, (k_final<float><<<grid_for(3 * N), 256, 0, s>>>(va, c->d_p0, N, c->d_inv, x0, (const float *)B_user, (const float *)U_sorted, dt, xout)),
           (k_final<double><<<grid_for(3 * N), 256, 0, s>>>(va, c->d_p0, N, c->d_inv, x0, (const double *)B_user, (const double *)U_sorted, dt, xout)));
  if (c->lattice) {
    c->nlaunch += 1;
    k_wrap_lattice<<<grid_for(N), 256, 0, s>>>(va, c->d_p0, N, xout);
  }
  PSE_CUDA_TRY(c, cudaGetLastError());
  return PSE_OK;
}

pse_status rfd_noise(pse_ctx *c, const void *wt, uint64_t seed, uint64_t counter, void *W8, cudaStream_t s) {
  StageTimer timer(c, PSE_STAGE_VECTOR, s);
  c->nlaunch += 1;
  int64_t N = c->p.N;
  DISPATCH(c, (k_rfd_noise<float><<<grid_for(8 * N), 256, 0, s>>>(N, (const float *)wt, seed, counter, (float *)W8)),
           (k_rfd_noise<double><<<grid_for(8 * N), 256, 0, s>>>(N, (const double *)wt, seed, counter, (double *)W8)));
  PSE_CUDA_TRY(c, cudaGetLastError());
  return PSE_OK;
}

pse_status rfd_final(pse_ctx *c, const double *x0, const void *B, const void *U0, const void *Rp, const void *Rm,
                     double dt, double fac, double *xout, cudaStream_t s) {
  StageTimer timer(c, PSE_STAGE_VECTOR, s);
  c->nlaunch += 1;
  int64_t N = c->p.N;
  VecArgs va = vec_args(c);
  DISPATCH(c, (k_rfd_final<float><<<grid_for(3 * N), 256, 0, s>>>(va, c->d_p0, N, x0, (const float *)B, (const float *)U0, (const float *)Rp, (const float *)Rm, dt, fac, xout)),
           (k_rfd_final<double><<<grid_for(3 * N), 256, 0, s>>>(va, c->d_p0, N, x0, (const double *)B, (const double *)U0, (const double *)Rp, (const double *)Rm, dt, fac, xout)));
  if (c->lattice) {
    c->nlaunch += 1;
    k_wrap_lattice<<<grid_for(N), 256, 0, s>>>(va, c->d_p0, N, xout);
  }
  PSE_CUDA_TRY(c, cudaGetLastError());
  return PSE_OK;
}

pse_status check_finite(pse_ctx *c, const void *ptr, int64_t n, bool dbl, int *bad, cudaStream_t s) {
  StageTimer timer(c, PSE_STAGE_VECTOR, s);
  c->nlaunch += 1;
  unsigned nb = std::min<unsigned>(grid_for(n), 2048);
  if (dbl) k_finite<double><<<nb, 256, 0, s>>>((const double *)ptr, n, bad);
  else k_finite<float><<<nb, 256, 0, s>>>((const float *)ptr, n, bad);
  PSE_CUDA_TRY(c, cudaGetLastError());
  return PSE_OK;
}

}  // namespace pse
