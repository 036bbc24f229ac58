// Krylov vector kernels and the device-side control of the Lanczos square root
// (Sec. 3.2: tridiagonal T_m, c_m = T_m^{1/2} e1, stopping rule
// |c_m - [c_{m-1}; 0]| / |c_m| <= tol) and of unrestarted GMRES for the stresslet
// constraint (Hessenberg column, Givens rotations, |r|/|b| <= tol, back substitution).
//
// One iteration after the product w = A v_j is four launches:
//   k_kr_dot      h1 = V^T w
//   k_kr_sub_dot  w -= V h1, h2 = V^T w
//   k_kr_finish   w -= V h2, |w|^2 (and beside it the tridiagonal square root), the
//                 scalar step of every suspension, loop control
//   k_kr_next     v_{j+1} = w / |w|, also in cell-list order for the next pair sum
// A sum over the blocks of a suspension is taken by the last of them to arrive (a
// counter, no waiting), which in k_kr_finish also takes the scalar step, so neither the
// sums nor the control cost a launch of their own.  The blocks hold at most 16384
// elements and fewer for small vectors (pse_ctx::vchunk), and w's update and the next
// dot products run over one block's rows back to back, out of L1 and L2.
//
// Bound by launch and reduction latency below about 10^5 particles and by HBM above.
// Per GMRES iteration, all vector and control kernels, against eleven separate launches
// on 16384-element blocks: N = 3000 63 -> 25 us, N = 64000 (11 rows) 120 -> 56 us,
// N = 2^20 (4 rows) 205 -> 156 us.
//
// The dot products, scale factors and combination coefficients live in the
// per-suspension coefficient blocks; loop control sets a flag (and, inside a CUDA graph,
// the while-node condition) so an iteration needs no host round trip.
#include <cuda_runtime.h>

#include <vector>

#include "device_common.cuh"
#include "krylov_math.cuh"
#include "pse_internal.cuh"
#include "vec_common.cuh"

namespace pse {
namespace {

struct KrArgs {
  VecArgs va;
  KDev k;
  int64_t stride, nblk;  // elements of a basis row, blocks of the launch
  double *partial;       // [row][block]
  int *done;             // arrival counters: one per suspension, one for the launch
};

// True in every thread of the last of n blocks to arrive at *ctr (zero before and after).
// What a thread wrote before the call is visible to the last block after it.
__device__ __forceinline__ bool last_block(int *ctr, int n) {
  __shared__ int s_last;
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) {
    s_last = atomicAdd(ctr, 1) == n - 1;
    if (s_last) *ctr = 0;
  }
  __syncthreads();
  const bool last = s_last != 0;
  if (last) __threadfence();
  return last;
}

// out[r] = sum over blocks [b0, b1) of the partials of row r < nr (one warp per row).
__device__ __forceinline__ void sum_partials(const KrArgs &a, int b0, int b1, int nr, double *out) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
  for (int r = wid; r < nr; r += nw) {
    double sum = 0;
    for (int b = b0 + lane; b < b1; b += 32) sum += __ldcg(a.partial + r * a.nblk + b);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
    if (lane == 0) out[r] = sum;
  }
}

// Dot products of the block's chunk of w with rows 0 .. nr - 1 into the partials; the
// suspension's last block sums them into out.
template <typename T>
__device__ __forceinline__ void block_dots(const KrArgs &a, const Chunk &ch, const T *__restrict__ rows, int nr,
                                           const T *w, double *out, double red[DOT_ROWS][DOT_NT / 32]) {
  for (int r0 = 0; r0 < nr; r0 += DOT_ROWS) {
    const int n = min(DOT_ROWS, nr - r0);
    T acc[DOT_ROWS];
    chunk_dots(ch, rows, a.stride, r0, n, w, acc);
    block_sums(acc, n, a.partial, a.nblk, blockIdx.x, r0, red);
  }
  const int b0 = a.va.blk0[ch.s], b1 = a.va.blk0[ch.s + 1];
  if (last_block(a.done + ch.s, b1 - b0)) sum_partials(a, b0, b1, nr, out);
}

// c = T^{1/2} e1 of the tridiagonal T (order m <= LZ_ROWS) by one warp: every lane
// solves (T / hi + s_k) x = e1 for its own node of the rational square root
// (sqrt_nodes), the lanes' solutions are summed in shared memory and multiplied by T.
// hi is the Gershgorin bound; lane 31 has no node and eliminates T / hi - 1 / SQRT_WINDOW
// instead, whose pivots tell whether the spectrum lies in the window.  False if it
// does not (the caller then takes the eigensolver).
//
// Bound by the latency of one reciprocal and three FP64 operations per row (the lanes
// run side by side); the implicit QL sweeps it replaces are one serial chain of about
// m^2 Givens rotations with a hypot and two divisions each.
constexpr int LZ_ROWS = 64;
__device__ bool tridiag_sqrt_e1_warp(int m, const double *al, const double *be, const double *nodes, double *sm,
                                     double *cv, int lane) {
  double *sa = sm, *sb = sm + LZ_ROWS, *x = sm + 2 * LZ_ROWS;  // x: [row][33]
  for (int i = lane; i < m; i += 32) {
    sa[i] = al[i];
    sb[i] = i < m - 1 ? be[i] : 0.0;
  }
  __syncwarp();
  double hi = 0.0;
  for (int i = lane; i < m; i += 32) hi = fmax(hi, sa[i] + sb[i] + (i > 0 ? sb[i - 1] : 0.0));
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) hi = fmax(hi, __shfl_xor_sync(0xffffffffu, hi, o));
  const double ih = recip(hi);  // T / hi has order one
  for (int i = lane; i < m; i += 32) {
    sa[i] *= ih;
    sb[i] *= ih;
  }
  __syncwarp();
  const bool node = lane < SQRT_NODES;
  const bool spd = shifted_solve_e1(m, sa, sb, node ? nodes[lane] : -1.0 / SQRT_WINDOW, x + lane, 33);
  if (!__all_sync(0xffffffffu, spd)) return false;
  const double w = node ? nodes[SQRT_NODES + lane] : 0.0;
  for (int i = 0; i < m; ++i) x[i * 33 + lane] = node ? w * x[i * 33 + lane] : 0.0;
  __syncwarp();
  for (int i = lane; i < m; i += 32) {
    double s[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll
    for (int k = 0; k < 32; ++k) s[k & 3] += x[i * 33 + k];
    x[i * 33 + 32] = (s[0] + s[1]) + (s[2] + s[3]);
  }
  __syncwarp();
  const double f = root(hi);
  for (int i = lane; i < m; i += 32) {
    double t = sa[i] * x[i * 33 + 32];
    if (i > 0) t += sb[i - 1] * x[(i - 1) * 33 + 32];
    if (i < m - 1) t += sb[i] * x[(i + 1) * 33 + 32];
    cv[i] = f * t;
  }
  __syncwarp();
  return true;
}

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Lanczos iteration j of suspension q, the part that needs h1 + h2 only (one warp; sm: LZ_ROWS *
// 35 doubles): alpha_j, c_m = T_m^{1/2} e1 and the relative change of the iterate.  A block
// of its own takes it beside the blocks that update w, and not their last one after
// them; and loop control counts suspensions, not blocks: k_kr_finish at 50,000 particles
// and ten iterations 23 -> 20 us per launch, at 3000 16 -> 14.
__device__ void lz_solve(const KDev &k, int q, int j, int lane, double *sm) {
  const int m = j + 1, L = k.lmax;
  const double *cf = k.coef + (size_t)q * COEF_STRIDE, *be = k.l_beta + (size_t)q * L, *cp = k.l_cprev + (size_t)q * L;
  double *al = k.l_alpha + (size_t)q * L, *cv = k.l_c + (size_t)q * L;
  if (lane == 0) al[j] = cf[CO_H1 + j] + cf[CO_H2 + j];
  __syncwarp();
  bool ok = true;
  if (j == 0) {
    if (lane == 0) cv[0] = root(fmax(al[0], 0.0));
  } else if (m > LZ_ROWS || !tridiag_sqrt_e1_warp(m, al, be, k.l_nodes, sm, cv, lane)) {
    // long recurrences, and spectra outside the window (rounding can take the smallest
    // eigenvalue of T to zero): one thread, work arrays in global memory
    if (lane == 0) ok = tridiag_sqrt_e1(m, al, be, k.l_work + (size_t)q * (2 * L + L * L), cv);
    ok = __shfl_sync(0xffffffffu, (int)ok, 0) != 0;
  }
  __syncwarp();
  if (ok && j > 0) {
    double num = 0, den = 0;
    for (int i = lane; i < m; i += 32) {
      const double c = cv[i], dv = c - (i < m - 1 ? cp[i] : 0.0);
      num += dv * dv;
      den += c * c;
    }
    const double err = root(warp_sum(num) * recip(warp_sum(den)));
    if (lane == 0) k.l_err[q] = err;
  }
  if (lane == 0) k.l_capped[q] = !ok;
}

// Lanczos step j of suspension q after lz_solve and |w|^2 (one warp): stopping rule, beta_j.
__device__ void lz_step(const KDev &k, int q, int j, int lane) {
  const int m = j + 1, L = k.lmax;
  double *cf = k.coef + (size_t)q * COEF_STRIDE;
  double *cp = k.l_cprev + (size_t)q * L;
  const double *cv = k.l_c + (size_t)q * L;
  const double bj = root(fmax(cf[CO_NRM], 0.0)), err = __ldcg(k.l_err + q);
  const bool ok = __ldcg(k.l_capped + q) == 0;
  bool stop = !ok || (j > 0 && k.ltol > 0 && err <= k.ltol);
  if (!stop) {
    for (int i = lane; i < m; i += 32) cp[i] = __ldcg(cv + i);
    if (bj == 0.0 || j == L - 1) stop = true;
  }
  if (stop) {
    const double b0 = k.l_b0[q];
    for (int i = lane; i < m; i += 32) cf[CO_Y + i] = b0 * __ldcg(cv + i);
  }
  __syncwarp();
  if (lane != 0) return;
  k.l_it[q] = m;
  if (stop) {
    k.active[q] = 0;
    k.nrows[q] = m;
    k.l_capped[q] = !ok || (k.ltol > 0 && !(err <= k.ltol) && m == L);
  } else {
    k.l_beta[(size_t)q * L + j] = bj;
    cf[CO_FAC] = recip(bj);
  }
}

// Scalar step of GMRES iteration j for suspension q, by one warp; sm: at least 4 * 128
// doubles.  The Hessenberg matrix is stored by columns (gmax + 1 reals each).
__device__ void gm_step(const KDev &k, int q, int j, int lane, double *sm) {
  const int M = k.gmax;
  double *cf = k.coef + (size_t)q * COEF_STRIDE;
  double *H = k.g_H + (size_t)q * (M + 1) * M, *cs = k.g_cs + (size_t)q * M, *sn = k.g_sn + (size_t)q * M;
  double *g = k.g_g + (size_t)q * (M + 1);
  double *col = sm, *sc = sm + 128, *ss = sm + 256, *sg = sm + 384;
  for (int i = lane; i <= j; i += 32) {
    col[i] = cf[CO_H1 + i] + cf[CO_H2 + i];
    sc[i] = i < j ? cs[i] : 0.0;
    ss[i] = i < j ? sn[i] : 0.0;
    sg[i] = g[i];
  }
  __syncwarp();
  const double hn = root(fmax(cf[CO_NRM], 0.0));
  if (lane == 0) {
    double a = col[0];
    for (int i = 0; i < j; ++i) {  // previous rotations
      const double b = col[i + 1];
      col[i] = sc[i] * a + ss[i] * b;
      a = -ss[i] * a + sc[i] * b;
    }
    const double r = root(a * a + hn * hn), ir = recip(r);
    const double c = r == 0 ? 1.0 : a * ir, s = r == 0 ? 0.0 : hn * ir;
    col[j] = r;
    cs[j] = c;
    sn[j] = s;
    const double gn = -s * sg[j];
    g[j + 1] = gn;
    sg[j] = c * sg[j];
    g[j] = sg[j];
    ss[0] = fabs(gn) * recip(k.g_beta[q]);
  }
  __syncwarp();
  const double rel = ss[0];
  const bool stop = rel <= k.gtol || hn == 0.0 || j == M - 1;
  for (int i = lane; i <= j; i += 32) H[(size_t)j * (M + 1) + i] = col[i];
  if (stop) {  // back substitution H y = g into the combination coefficients, column by column
    for (int i = j; i >= 0; --i) {
      const double y = sg[i] * recip(col[i]);
      __syncwarp();
      if (lane == 0) cf[CO_Y + i] = y;
      for (int l = lane; l < i; l += 32) {
        sg[l] -= col[l] * y;
        col[l] = H[(size_t)(i - 1) * (M + 1) + l];
      }
      __syncwarp();
    }
  }
  if (lane != 0) return;
  k.g_rel[q] = rel;
  k.g_it[q] = j + 1;
  if (stop) {
    k.active[q] = 0;
    k.nrows[q] = j + 1;
    k.g_capped[q] = !(rel <= k.gtol) && j + 1 == M;
  } else {
    cf[CO_FAC] = recip(hn);
  }
}

// Start of a recurrence from z (every suspension): |z|, the scalar state, iteration 0.
template <typename T, bool GM>
__global__ void k_kr_start(KrArgs a, const T *z) {
  __shared__ double red[DOT_ROWS][DOT_NT / 32];
  const Chunk ch = chunk_of(a.va, blockIdx.x);
  const KDev &k = a.k;
  const int q = ch.s;
  T acc[DOT_ROWS];
  chunk_dots(ch, z, 0, 0, 1, z, acc);
  block_sums(acc, 1, a.partial, a.nblk, blockIdx.x, 0, red);
  const int b0 = a.va.blk0[q], b1 = a.va.blk0[q + 1];
  double *cf = k.coef + (size_t)q * COEF_STRIDE;
  if (last_block(a.done + q, b1 - b0)) {
    sum_partials(a, b0, b1, 1, cf + CO_NRM);
    if (threadIdx.x == 0) {
      const double b = root(fmax(cf[CO_NRM], 0.0));
      if (GM) {
        k.g_beta[q] = b;
        k.g_rel[q] = b > 0.0 ? 1.0 : 0.0;
        k.g_g[(size_t)q * (k.gmax + 1)] = b;
        k.g_it[q] = 0;
        k.g_capped[q] = 0;
      } else {
        k.l_b0[q] = b;
        k.l_err[q] = HUGE_VAL;
        k.l_it[q] = 0;
        k.l_capped[q] = 0;
      }
      k.nrows[q] = 0;
      k.active[q] = b > 0.0;
      cf[CO_FAC] = b > 0.0 ? recip(b) : 0.0;
    }
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) *k.iter = 0;
}

template <typename T>
__global__ void k_kr_dot(KrArgs a, const T *__restrict__ rows, const T *w) {
  __shared__ double red[DOT_ROWS][DOT_NT / 32];
  const Chunk ch = chunk_of(a.va, blockIdx.x);
  if (!a.va.active[ch.s]) return;
  const int nr = min(*a.k.iter + 1, MAX_ROWS);
  block_dots(a, ch, rows, nr, w, a.k.coef + (size_t)ch.s * COEF_STRIDE + CO_H1, red);
}

template <typename T>
__global__ void k_kr_sub_dot(KrArgs a, const T *__restrict__ rows, T *w) {
  __shared__ double red[DOT_ROWS][DOT_NT / 32];
  __shared__ T cs[MAX_ROWS];
  const Chunk ch = chunk_of(a.va, blockIdx.x);
  if (!a.va.active[ch.s]) return;
  const int nr = min(*a.k.iter + 1, MAX_ROWS);
  double *cf = a.k.coef + (size_t)ch.s * COEF_STRIDE;
  for (int r = threadIdx.x; r < nr; r += blockDim.x) cs[r] = (T)cf[CO_H1 + r];
  __syncthreads();
  chunk_sub(ch, w, rows, a.stride, nr, cs);
  block_dots(a, ch, rows, nr, w, cf + CO_H2, red);
}

// The loop continues while a suspension is active and fewer than `cap` iterations ran
// (so it always terminates); h: the while node's condition inside a graph.
template <typename T, bool GM>
__global__ void k_kr_finish(KrArgs a, const T *__restrict__ rows, T *w, int cap, cudaGraphConditionalHandle h,
                            int graph) {
  __shared__ double red[DOT_ROWS][DOT_NT / 32];
  __shared__ T cs[MAX_ROWS];
  __shared__ double sm[LZ_ROWS * 35];
  const KDev &k = a.k;
  const int solvers = GM ? 0 : k.nsys, b = (int)blockIdx.x - solvers;
  const Chunk ch = chunk_of(a.va, max(b, 0));
  const int q = b < 0 ? (int)blockIdx.x : ch.s, j = *k.iter;
  const int b0 = a.va.blk0[q], b1 = a.va.blk0[q + 1];
  bool last = (int)blockIdx.x == (GM ? b0 : q);  // an inactive suspension arrives with its first block
  if (a.va.active[q]) {
    if (b < 0) {
      if (threadIdx.x < 32) lz_solve(k, q, j, threadIdx.x, sm);
    } else {
      const int nr = min(j + 1, MAX_ROWS);
      const double *cf = k.coef + (size_t)q * COEF_STRIDE;
      for (int r = threadIdx.x; r < nr; r += blockDim.x) cs[r] = (T)cf[CO_H2 + r];
      __syncthreads();
      T acc[DOT_ROWS];
#pragma unroll
      for (int r = 0; r < DOT_ROWS; ++r) acc[r] = 0;
      acc[0] = chunk_sub(ch, w, rows, a.stride, nr, cs);
      block_sums(acc, 1, a.partial, a.nblk, b, 0, red);
    }
    last = last_block(a.done + q, b1 - b0 + (GM ? 0 : 1));
    if (last) {
      sum_partials(a, b0, b1, 1, k.coef + (size_t)q * COEF_STRIDE + CO_NRM);
      if (threadIdx.x < 32) {
        __syncwarp();
        if (GM) gm_step(k, q, j, threadIdx.x, sm);
        else lz_step(k, q, j, threadIdx.x);
      }
      __syncthreads();
    }
  }
  // loop control by the last suspension to arrive
  if (last && (k.nsys == 1 || last_block(a.done + k.nsys, k.nsys))) {
    int any = 0;
    for (int s = threadIdx.x; s < k.nsys; s += blockDim.x) any |= __ldcg(k.active + s);
    any = __syncthreads_or(any);
    if (threadIdx.x == 0) {
      const int cont = any && j + 1 < cap;
      *k.iter = j + 1;
      k.flag[0] = cont;
      if (graph) cudaGraphSetConditional(h, cont ? 1u : 0u);
    }
  }
}

// Basis row *iter = coef[s][CO_FAC] * src for the active suspensions, also into vin and,
// particle by particle, into the cell-list order of the pair sum's input (pos: a
// particle's place in that list).
template <typename T>
__global__ void k_kr_next(KrArgs a, T *basis, const T *src, T *vin, T *vcell, const int *__restrict__ pos) {
  using T4 = typename V4<T>::t;
  const Chunk ch = chunk_of(a.va, blockIdx.x);
  if (!a.va.active[ch.s]) return;
  const T f = (T)a.k.coef[(size_t)ch.s * COEF_STRIDE + CO_FAC];
  T *dst = basis + (int64_t)*a.k.iter * a.stride;
  for (int64_t i = ch.beg / 8 + threadIdx.x; i < ch.end / 8; i += blockDim.x) {  // a row of 8 per thread
    const int64_t p = pos[i];
    T4 lo, hi;
    load_row((const T4 *)src, i, lo, hi);
    lo.x *= f;
    lo.y *= f;
    lo.z *= f;
    lo.w *= f;
    hi.x *= f;
    hi.y *= f;
    hi.z *= f;
    hi.w *= f;
    store_row((T4 *)dst, i, lo, hi);
    store_row((T4 *)vin, i, lo, hi);
    cell_row(lo, hi);
    store_row((T4 *)vcell, p, lo, hi);
  }
}

// flag[0] = (any suspension active); inside a graph also the while condition.
__global__ void k_loop_begin(KDev k, cudaGraphConditionalHandle h, int graph) {
  int any = 0;
  for (int q = threadIdx.x; q < k.nsys; q += blockDim.x) any |= k.active[q];
  any = __syncthreads_or(any);
  if (threadIdx.x == 0) {
    k.flag[0] = any;
    if (graph) cudaGraphSetConditional(h, any ? 1u : 0u);
  }
}

__global__ void k_all_active(int nsys, int *active) {
  for (int q = blockIdx.x * blockDim.x + threadIdx.x; q < nsys; q += gridDim.x * blockDim.x) active[q] = 1;
}

unsigned sys_blocks(const pse_ctx *c) { return (unsigned)std::min<int64_t>(ceil_div(c->nsys, 128), 512); }

KrArgs kr_args(const pse_ctx *c) {
  KrArgs a;
  a.va = vec_args(c);
  a.k = c->kd;
  a.stride = 8 * c->p.N;
  a.nblk = c->nvblk;
  a.partial = c->d_dots;
  a.done = c->d_done;
  return a;
}

template <typename T>
void kr_start_t(pse_ctx *c, const void *z, bool gm, cudaStream_t s) {
  const unsigned nb = (unsigned)c->nvblk;
  if (gm) k_kr_start<T, true><<<nb, DOT_NT, 0, s>>>(kr_args(c), (const T *)z);
  else k_kr_start<T, false><<<nb, DOT_NT, 0, s>>>(kr_args(c), (const T *)z);
}

template <typename T>
void kr_step_t(pse_ctx *c, void *w, bool gm, int cap, cudaGraphConditionalHandle h, int graph, cudaStream_t s) {
  const unsigned nb = (unsigned)c->nvblk;
  const KrArgs a = kr_args(c);
  const T *V = (const T *)c->d_basis;
  k_kr_dot<T><<<nb, DOT_NT, 0, s>>>(a, V, (const T *)w);
  k_kr_sub_dot<T><<<nb, DOT_NT, 0, s>>>(a, V, (T *)w);
  if (gm) k_kr_finish<T, true><<<nb, DOT_NT, 0, s>>>(a, V, (T *)w, cap, h, graph);
  else k_kr_finish<T, false><<<nb + c->nsys, DOT_NT, 0, s>>>(a, V, (T *)w, cap, h, graph);
}

}  // namespace

// |z| and the scalar start of a Lanczos (gm = false) or GMRES recurrence.
pse_status kr_start(pse_ctx *c, const void *z, bool gm, cudaStream_t s) {
  StageTimer timer(c, PSE_STAGE_VECTOR, s);
  c->nlaunch += 1;
  if (c->prec == PSE_MIXED) kr_start_t<float>(c, z, gm, s);
  else kr_start_t<double>(c, z, gm, s);
  PSE_CUDA_TRY(c, cudaGetLastError());
  return PSE_OK;
}

// Orthogonalises w against basis rows 0 .. *iter (classical Gram-Schmidt twice, FP64
// coefficients), takes the scalar step of every active suspension and advances the loop.
pse_status kr_step(pse_ctx *c, void *w, bool gm, int cap, cudaGraphConditionalHandle h, int graph, cudaStream_t s) {
  StageTimer timer(c, PSE_STAGE_VECTOR, s);
  c->nlaunch += 3;
  if (c->prec == PSE_MIXED) kr_step_t<float>(c, w, gm, cap, h, graph, s);
  else kr_step_t<double>(c, w, gm, cap, h, graph, s);
  PSE_CUDA_TRY(c, cudaGetLastError());
  return PSE_OK;
}

// The next Krylov vector from src: basis row *iter, d_vin and d_vcell (the pair sum's input).
pse_status kr_next(pse_ctx *c, const void *src, cudaStream_t s) {
  StageTimer timer(c, PSE_STAGE_VECTOR, s);
  c->nlaunch += 1;
  const unsigned nb = (unsigned)c->nvblk;
  if (c->prec == PSE_MIXED)
    k_kr_next<float><<<nb, DOT_NT, 0, s>>>(kr_args(c), (float *)c->d_basis, (const float *)src, (float *)c->d_vin,
                                           (float *)c->d_vcell, c->d_cell_key);
  else
    k_kr_next<double><<<nb, DOT_NT, 0, s>>>(kr_args(c), (double *)c->d_basis, (const double *)src, (double *)c->d_vin,
                                            (double *)c->d_vcell, c->d_cell_key);
  PSE_CUDA_TRY(c, cudaGetLastError());
  return PSE_OK;
}

void kd_loop_begin(pse_ctx *c, cudaGraphConditionalHandle h, int graph, cudaStream_t s) {
  c->nlaunch += 1;
  k_loop_begin<<<1, 256, 0, s>>>(c->kd, h, graph);
}
void kd_all_active(pse_ctx *c, cudaStream_t s) {
  c->nlaunch += 1;
  k_all_active<<<sys_blocks(c), 128, 0, s>>>(c->nsys, c->d_active);
}

namespace {

__global__ void k_scalars(int n, const double *x, double *rec, double *rt) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  rec[i] = recip(x[i]);
  rt[i] = root(x[i]);
}

__global__ void __launch_bounds__(32) k_lz_solve(KDev k, int j) {
  __shared__ double sm[LZ_ROWS * 35];
  lz_solve(k, 0, j, threadIdx.x, sm);
}

}  // namespace

}  // namespace pse

// The device's scalar arithmetic and tridiagonal square root on host arrays (not on any
// product's path: the library's own checks call them).
extern "C" {

// rec = recip(x), rt = root(x); 0, or 1 on a CUDA error.
int pse_internal_device_scalars(int n, const double *x, double *rec, double *rt) {
  const size_t b = sizeof(double) * (size_t)n;
  double *d = nullptr;
  if (n < 1 || cudaMalloc(&d, 3 * b) != cudaSuccess) return 1;
  cudaError_t e = cudaMemcpy(d, x, b, cudaMemcpyHostToDevice);
  pse::k_scalars<<<(n + 127) / 128, 128>>>(n, d, d + n, d + 2 * n);
  if (e == cudaSuccess) e = cudaGetLastError();
  if (e == cudaSuccess) e = cudaMemcpy(rec, d + n, b, cudaMemcpyDeviceToHost);
  if (e == cudaSuccess) e = cudaMemcpy(rt, d + 2 * n, b, cudaMemcpyDeviceToHost);
  cudaFree(d);
  return e == cudaSuccess ? 0 : 1;
}

// c = T^{1/2} e1 as iteration m - 1 of the Lanczos kernel takes it (alpha[0..m), beta[0..m-1)):
// 0, 2 when the eigensolver gave up, 1 on a CUDA error.
int pse_internal_device_sqrt_e1(int m, const double *alpha, const double *beta, double *c) {
  if (m < 1 || m > 120) return 1;
  const size_t L = (size_t)m, nodes = 2 * pse::SQRT_NODES;
  std::vector<double> h(pse::COEF_STRIDE + 4 * L + 1 + nodes + 2 * L + L * L + 1, 0.0);
  double *p = nullptr;
  if (cudaMalloc(&p, sizeof(double) * h.size()) != cudaSuccess) return 1;
  pse::KDev k{};
  k.nsys = 1;
  k.lmax = m;
  k.coef = p;
  k.l_alpha = k.coef + pse::COEF_STRIDE;
  k.l_beta = k.l_alpha + L;
  k.l_cprev = k.l_beta + L;
  k.l_c = k.l_cprev + L;
  k.l_err = k.l_c + L;
  k.l_nodes = k.l_err + 1;
  k.l_work = k.l_err + 1 + nodes;
  k.l_capped = (int *)(k.l_work + 2 * L + L * L);
  h[pse::CO_H1 + m - 1] = alpha[m - 1];
  for (int i = 0; i + 1 < m; ++i) {
    h[pse::COEF_STRIDE + i] = alpha[i];
    h[pse::COEF_STRIDE + L + i] = beta[i];
  }
  double *hn = &h[pse::COEF_STRIDE + 4 * L + 1];
  pse::sqrt_nodes(pse::SQRT_NODES, pse::SQRT_WINDOW, hn, hn + pse::SQRT_NODES);
  int capped = 0;
  cudaError_t e = cudaMemcpy(p, h.data(), sizeof(double) * h.size(), cudaMemcpyHostToDevice);
  pse::k_lz_solve<<<1, 32>>>(k, m - 1);
  if (e == cudaSuccess) e = cudaGetLastError();
  if (e == cudaSuccess) e = cudaMemcpy(c, k.l_c, sizeof(double) * L, cudaMemcpyDeviceToHost);
  if (e == cudaSuccess) e = cudaMemcpy(&capped, k.l_capped, sizeof(int), cudaMemcpyDeviceToHost);
  cudaFree(p);
  return e != cudaSuccess ? 1 : (capped ? 2 : 0);
}

}  // extern "C"
