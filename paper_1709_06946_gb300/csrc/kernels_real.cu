// Real-space part of the split mobility (Sec. 2.3.1): for every particle the sum
// over neighbours closer than r_cut of the 8x8 real-space block (Eqs. MUFr-MDCr)
// applied to [F; S], plus the real-space self term (App. A, Case 3).
//
// G lanes per particle walk its slotted neighbour list.  Outputs are in sorted
// order (by suspension, then spreading tile); each neighbour record holds the
// neighbour's position in the cell list, and the input vector is first copied
// into cell-list order, so the lanes of a particle, walking consecutive entries
// of the list (runs of cells along x), read neighbouring rows of that copy and
// share cache lines.  A persistent grid takes blocks of particles from a work
// counter; particles of suspensions marked inactive are skipped.  The copy holds the
// stresslet as Cartesian components, and the strain rates are summed as Cartesian
// components and projected on the Y basis once per particle.
//
// The seven scalar functions, FP32: beyond contact a Gaussian times polynomials in 1/r
// (RealPoly, fitted per handle), below it a table on r with linear interpolation; FP64:
// cubic Lagrange interpolation of the table with one-sided stencils at the r = 2a node
// where the functions have a kink.
#include <algorithm>

#include "device_common.cuh"
#include "pse_internal.cuh"

namespace pse {
namespace {

struct RealArgs {
  int64_t Ntot;
  int nsys, len, k2;
  double inv_dr, self_uf, self_es;
};

// Where an FP32 product takes its scalar functions from.
enum { LK_TABLE = 0, LK_SMEM = 1, LK_POLY = 2 };

// 32 bytes (8 floats) from 32-byte aligned read-only global memory in one
// 256-bit load.
__device__ __forceinline__ void ldg8(const float *p, float4 &lo, float4 &hi) {
  asm("ld.global.nc.v8.f32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
      : "=f"(lo.x), "=f"(lo.y), "=f"(lo.z), "=f"(lo.w), "=f"(hi.x), "=f"(hi.y), "=f"(hi.z), "=f"(hi.w)
      : "l"(p));
}

// A neighbour record, brought from DRAM 256 bytes at a time (a particle's records are
// contiguous: its lanes' next four steps).  S -> E at 2^20 particles 435 -> 415 us; not
// allocating in L1 makes it 462 us.
__device__ __forceinline__ float4 ld_record(const float4 *p) {
  float4 v;
  asm("ld.global.nc.L2::256B.v4.f32 {%0,%1,%2,%3}, [%4];"
      : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
      : "l"(p));
  return v;
}
__device__ __forceinline__ double4_32a ld_record(const double4_32a *p) { return *p; }

// f[0..7) at r by linear interpolation.  The full product reads two 8-float
// entries (q and q + 1); the partial products read one 8-float interval record
// holding the values they need at both ends: f4..f6 (S -> E) or f0..f3
// ([F; S] -> U); the other functions are left unset.
template <bool SH = false, int MODE = M_FULL>
__device__ __forceinline__ void lookup(const float *tab, const RealArgs &a, float r, float f[7]) {
  float x = r * (float)a.inv_dr;
  int q = min((int)x, a.len - 2);
  float t = x - (float)q;
  const float4 *t4 = (const float4 *)tab;
  float4 a0, a1, b0, b1;
  if (!SH && MODE == M_SE) {
    ldg8(tab + 8 * q, a0, a1);  // f4 f5 f6 at q, then at q + 1
    f[4] = fmaf(t, a0.w - a0.x, a0.x);
    f[5] = fmaf(t, a1.x - a0.y, a0.y);
    f[6] = fmaf(t, a1.y - a0.z, a0.z);
    return;
  }
  if (!SH && (MODE == M_FSU || MODE == M_SU)) {
    ldg8(tab + 8 * q, a0, a1);  // f0..f3 at q, then at q + 1
    f[0] = fmaf(t, a1.x - a0.x, a0.x);
    f[1] = fmaf(t, a1.y - a0.y, a0.y);
    f[2] = fmaf(t, a1.z - a0.z, a0.z);
    f[3] = fmaf(t, a1.w - a0.w, a0.w);
    return;
  }
  if (SH) {  // table staged in shared memory
    a0 = t4[2 * q];
    a1 = t4[2 * q + 1];
    b0 = t4[2 * q + 2];
    b1 = t4[2 * q + 3];
  } else {  // entries are 8 floats (32 bytes): one 256-bit load each
    ldg8(tab + 8 * q, a0, a1);
    ldg8(tab + 8 * q + 8, b0, b1);
  }
  f[0] = fmaf(t, b0.x - a0.x, a0.x);
  f[1] = fmaf(t, b0.y - a0.y, a0.y);
  f[2] = fmaf(t, b0.z - a0.z, a0.z);
  f[3] = fmaf(t, b0.w - a0.w, a0.w);
  f[4] = fmaf(t, b1.x - a1.x, a1.x);
  f[5] = fmaf(t, b1.y - a1.y, a1.y);
  f[6] = fmaf(t, b1.z - a1.z, a1.z);
}

template <bool SH = false, int MODE = M_FULL>
__device__ __forceinline__ void lookup(const double *tab, const RealArgs &a, double r, double f[7]) {
  double x = r * a.inv_dr;
  int q = min((int)x, a.len - 2);
  int b = q - 1;
  if (q < a.k2) b = min(b, a.k2 - 3);
  else b = max(b, a.k2);
  b = max(0, min(b, a.len - 4));
  double t = x - (double)b;
  const double c6 = 1.0 / 6.0, u0 = t * (t - 1), u1 = (t - 2) * (t - 3);
  const double w0 = -c6 * (t - 1) * u1, w1 = 0.5 * t * u1, w2 = -0.5 * u0 * (t - 3), w3 = c6 * u0 * (t - 2);
  const double *r0 = tab + 8 * (size_t)b;
#pragma unroll
  for (int k = 0; k < 7; ++k)
    f[k] = w0 * __ldg(r0 + k) + w1 * __ldg(r0 + 8 + k) + w2 * __ldg(r0 + 16 + k) + w3 * __ldg(r0 + 24 + k);
}

// Function k of the fit: f_k = exp2(-cg (r - r0)^2) P_k(t), t = ta / r + tb in [-1, 1].
__device__ __forceinline__ float poly_at(const RealPoly &p, int k, float t) {
  float v = p.c[k][POLY_DEG];
#pragma unroll
  for (int d = POLY_DEG - 1; d >= 0; --d) v = fmaf(v, t, p.c[k][d]);
  return v;
}

// One neighbour's terms.  g: separation; row: [F, Sxx, Syy, Sxy, Sxz, Syz]; f: the scalar
// functions with f[1] - f[0] in place of f[1].  U += f2 v + f0 F + (f3 q + (f1 - f0) rf) rh with
// v = S rh, q = rh.v, rf = rh.F; the strain is sym(w, rh) + f4 S with
// w = f5 v - f2 F / 2 + (f6 q - f3 rf) / 2 rh; d holds half of its diagonal, o the rest.
template <typename T, int MODE>
__device__ __forceinline__ void pair_terms(const T rh[3], const T row[8], const T f[7], T U[3], T d[3], T o[3]) {
  constexpr bool HAS_F = MODE == M_FULL || MODE == M_FSU, WANT_U = MODE != M_SE;
  constexpr bool WANT_E = MODE == M_FULL || MODE == M_SE;
  const T szz = -(row[3] + row[4]);
  const T v[3] = {row[3] * rh[0] + row[5] * rh[1] + row[6] * rh[2], row[5] * rh[0] + row[4] * rh[1] + row[7] * rh[2],
                  row[6] * rh[0] + row[7] * rh[1] + szz * rh[2]};
  const T q = rh[0] * v[0] + rh[1] * v[1] + rh[2] * v[2];
  const T rf = HAS_F ? rh[0] * row[0] + rh[1] * row[1] + rh[2] * row[2] : (T)0;
  if (WANT_U) {
    T c = f[3] * q;
    if (HAS_F) c += f[1] * rf;
#pragma unroll
    for (int m = 0; m < 3; ++m) {
      U[m] += f[2] * v[m] + c * rh[m];
      if (HAS_F) U[m] += f[0] * row[m];
    }
  }
  if (WANT_E) {
    const T cy = (T)0.5 * (HAS_F ? f[6] * q - f[3] * rf : f[6] * q), h4 = (T)0.5 * f[4], h2 = (T)-0.5 * f[2];
    T w[3];
#pragma unroll
    for (int m = 0; m < 3; ++m) {
      w[m] = f[5] * v[m] + cy * rh[m];
      if (HAS_F) w[m] += h2 * row[m];
    }
    d[0] += h4 * row[3] + w[0] * rh[0];
    d[1] += h4 * row[4] + w[1] * rh[1];
    d[2] += h4 * szz + w[2] * rh[2];
    o[0] += f[4] * row[5] + w[0] * rh[1] + w[1] * rh[0];
    o[1] += f[4] * row[6] + w[0] * rh[2] + w[2] * rh[0];
    o[2] += f[4] * row[7] + w[1] * rh[2] + w[2] * rh[1];
  }
}

// G lanes share one particle: they walk its neighbour list with stride G (so
// the neighbours' records are fetched in parallel) and the partial sums are
// reduced with shuffles; the first lane of the group adds the self term.
//
// Bound: random 32-byte reads pass L1 at 64 bytes per clock and SM (1.95 lanes per clock
// measured), so a table entry per pair (two for the full product) cost as much as the
// neighbour's row; the polynomials take 9 FMAs per function instead, and the FMA pipe
// and L1 are then about equally busy.  The terms collected along rh and in Cartesian
// components take about 60 operations (110 in the Y basis).  At 2^20 particles, 105
// neighbours each: full product 886 -> 630 us, S -> E 648 -> 415, S -> U 594 -> 364;
// FP64 form at 11000 particles 630 -> 445 us.  Below 10^5 particles the few thousand warps
// wait on their records (S -> E at 64000 49 us, 67 before).
//
// FP32, polynomials: 48 registers so that five 256-thread CTAs fit an SM (four: S -> E 487
// us; six: full 751 us, spilled).  With the table 64 registers and four, as its lookups of the
// full product do not fit 48: per product 831 -> 803 us at 10^6 particles, 149 -> 140 at 10^5 and
// xi = 0.3, 27 -> 21 at 3000; S -> E the same.  A static split over warps instead of the work
// counter: full 737 us.  With LK_SMEM one 1024-thread CTA per SM first copies the table into
// shared memory.
template <typename T, int MODE, int G, int LK = LK_TABLE, int NT = LK == LK_SMEM ? 1024 : 256>
__global__ void __launch_bounds__(NT, sizeof(T) == 4 ? (LK == LK_SMEM ? 1 : (LK == LK_TABLE ? 4 : 5)) : 1)
    k_real(RealArgs a, RealPoly poly, const SysDev *__restrict__ sys, const int64_t *__restrict__ p0,
           const int *__restrict__ active, int *queue, int nitems, const int *__restrict__ nstart,
           const typename V4<T>::t *__restrict__ geo, const T *__restrict__ vin, const T *__restrict__ vcell,
           T *__restrict__ vout, const T *__restrict__ gtab) {
  extern __shared__ __align__(16) unsigned char tab_raw[];
  const T *tab = gtab;
  if (LK == LK_SMEM) {
    float4 *dst = (float4 *)tab_raw;
    const float4 *src = (const float4 *)gtab;
    for (int q = threadIdx.x; q < 2 * a.len; q += blockDim.x) dst[q] = src[q];
    __syncthreads();
    tab = (const T *)tab_raw;
  }
  constexpr bool HAS_F = MODE == M_FULL || MODE == M_FSU, WANT_U = MODE != M_SE;
  constexpr bool WANT_E = MODE == M_FULL || MODE == M_SE;
  using T4 = typename V4<T>::t;
  for_each_item(queue, nitems, [&](int item) {
    const int64_t gid = ((int64_t)item * NT + threadIdx.x) / G;
    const int sub = threadIdx.x % G;
    const int64_t i = gid < a.Ntot ? gid : a.Ntot - 1;
    const int si = find_sys(p0, a.nsys, i);
    const bool live = gid < a.Ntot && active[si];
    const SysDev &sd = sys[si];
    const T4 *v4 = (const T4 *)vin, *vc4 = (const T4 *)vcell;
    T U[3] = {0, 0, 0}, d[3] = {0, 0, 0}, o[3] = {0, 0, 0};
    // particle i's row of slots; an overflowed list is flagged and redone
    const int64_t k0 = sd.nbr0 + (i - sd.p0) * sd.slots;
    const int cnt = live ? min(nstart[i], sd.slots) : 0;
    T4 next;
    if (sub < cnt) next = ld_record(geo + k0 + sub);
    for (int n = sub; n < cnt; n += G) {
      const T4 gg = next;  // separation x_i - x_j and j, stored by the list build
      if (n + G < cnt) next = ld_record(geo + k0 + n + G);
      const int j = real_as_index<T>(gg.w);
      T4 q0, q1;
      if constexpr (sizeof(T) == 4) ldg8((const float *)vcell + 8 * (size_t)j, q0, q1);  // the 8 slots of row j
      else q0 = vc4[2 * j], q1 = vc4[2 * j + 1];
      const T r2 = gg.x * gg.x + gg.y * gg.y + gg.z * gg.z;
      const T ir = sizeof(T) == 4 ? (T)fast_rsqrt((float)r2) : (T)1 / sqrt(r2), r = r2 * ir;
      const T rh[3] = {gg.x * ir, gg.y * ir, gg.z * ir};
      T f[7];
      if (LK == LK_POLY && (float)r2 >= poly.r02) {
        const float t = fmaf(poly.ta, (float)ir, poly.tb), dr = (float)r - poly.r0, g = fast_exp2(-poly.cg * dr * dr);
        if (HAS_F) f[0] = (T)(g * poly_at(poly, 0, t));
        if (HAS_F) f[1] = (T)(g * poly_at(poly, 1, t));
        if (WANT_U || HAS_F) f[2] = (T)(g * poly_at(poly, 2, t));
        if (WANT_U || HAS_F) f[3] = (T)(g * poly_at(poly, 3, t));
        if (WANT_E) {
          f[4] = (T)(g * poly_at(poly, 4, t));
          f[5] = (T)(g * poly_at(poly, 5, t));
          f[6] = (T)(g * poly_at(poly, 6, t));
        }
      } else {
        lookup<LK == LK_SMEM, MODE>(tab, a, r, f);
        if (HAS_F) f[1] -= f[0];
      }
      const T row[8] = {q0.x, q0.y, q0.z, q0.w, q1.x, q1.y, q1.z, q1.w};
      pair_terms<T, MODE>(rh, row, f, U, d, o);
    }
    const T r2 = (T)1.4142135623730951;
    T E[5] = {r2 * (d[0] - d[1]), (T)0.81649658092772603 * (d[0] + d[1] - 2 * d[2]), r2 * o[0], r2 * o[1], r2 * o[2]};
#pragma unroll
    for (int s = G / 2; s > 0; s >>= 1) {
#pragma unroll
      for (int m = 0; m < 3; ++m)
        if (WANT_U) U[m] += __shfl_xor_sync(0xffffffffu, U[m], s, G);
#pragma unroll
      for (int m = 0; m < 5; ++m)
        if (WANT_E) E[m] += __shfl_xor_sync(0xffffffffu, E[m], s, G);
    }
    if (live && sub == 0) {
      T4 s0 = v4[2 * i], s1 = v4[2 * i + 1];
      if (WANT_U && HAS_F) {
        U[0] += (T)a.self_uf * s0.x;
        U[1] += (T)a.self_uf * s0.y;
        U[2] += (T)a.self_uf * s0.z;
      }
      if (WANT_E) {
        E[0] += (T)a.self_es * s0.w;
        E[1] += (T)a.self_es * s1.x;
        E[2] += (T)a.self_es * s1.y;
        E[3] += (T)a.self_es * s1.z;
        E[4] += (T)a.self_es * s1.w;
      }
      T4 o0, o1;
      o0.x = U[0];
      o0.y = U[1];
      o0.z = U[2];
      o0.w = E[0];
      o1.x = E[1];
      o1.y = E[2];
      o1.z = E[3];
      o1.w = E[4];
      T4 *o4 = (T4 *)vout;
      o4[2 * i] = o0;
      o4[2 * i + 1] = o1;
    }
  });
}

template <typename T, int MODE, int G, int LK>
void launch_real_k(pse_ctx *c, const RealArgs &a, const void *vin, void *vout, const void *tab, cudaStream_t s) {
  constexpr int NT = LK == LK_SMEM ? 1024 : 256;
  auto kern = k_real<T, MODE, G, LK>;
  const size_t sm = LK == LK_SMEM ? sizeof(T) * 8 * (size_t)a.len : 0;
  if (LK == LK_SMEM) {
    static std::once_flag once;
    std::call_once(once, [&] {
      cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)c->smem_optin);
      cudaGetLastError();
    });
  }
  static std::atomic<int> per_sm{0};
  const int64_t items = ceil_div(a.Ntot * G, NT);
  const unsigned grid = persistent_grid(c, kern, NT, sm, items, per_sm);
  int *q = next_queue(c);
  kern<<<grid, NT, sm, s>>>(a, c->poly, c->d_sys, c->d_p0, c->d_active, q, (int)items, c->d_nbr_start,
                            (const typename V4<T>::t *)c->d_nbr_geo, (const T *)vin, (const T *)c->d_vcell, (T *)vout,
                            (const T *)tab);
}

// FP32: the table in shared memory where the autotuner chose it, else the polynomial fit
// where it holds (RealPoly::ok), else the table; the partial products read their interval
// tables.
template <typename T, int MODE, int G>
void launch_real_m(pse_ctx *c, const RealArgs &a, const void *vin, void *vout, cudaStream_t s) {
  if constexpr (sizeof(T) == 4) {
    if (c->real_smem_table && sizeof(T) * 8 * (size_t)a.len <= c->smem_optin)
      return launch_real_k<T, MODE, G, LK_SMEM>(c, a, vin, vout, c->d_table, s);
    const void *tab = MODE == M_SE ? c->d_table_e : (MODE == M_FULL ? c->d_table : c->d_table_u);
    if (c->poly.ok) return launch_real_k<T, MODE, G, LK_POLY>(c, a, vin, vout, tab, s);
    return launch_real_k<T, MODE, G, LK_TABLE>(c, a, vin, vout, tab, s);
  }
  launch_real_k<T, MODE, G, LK_TABLE>(c, a, vin, vout, c->d_table, s);
}

template <typename T, int G>
void launch_real_g(pse_ctx *c, const RealArgs &a, const void *vin, void *vout, int mode, cudaStream_t s) {
  if (mode == M_FULL) launch_real_m<T, M_FULL, G>(c, a, vin, vout, s);
  else if (mode == M_SE) launch_real_m<T, M_SE, G>(c, a, vin, vout, s);
  else if (mode == M_SU) launch_real_m<T, M_SU, G>(c, a, vin, vout, s);
  else launch_real_m<T, M_FSU, G>(c, a, vin, vout, s);
}

template <typename T>
void launch_real(pse_ctx *c, const RealArgs &a, const void *vin, void *vout, int mode, cudaStream_t s) {
  // lanes per particle from the mean neighbour count of the current lists
  int g = c->opt.real_lanes;
  if (g <= 0) {
    const int64_t pairs = c->npairs > 0 ? c->npairs : c->npairs_est;  // before the first list: the estimate
    double mean = a.Ntot > 0 ? (double)pairs / a.Ntot : 0.0;
    g = mean >= 200.0 ? 8 : (mean >= 24.0 ? 4 : 1);  // 4 lanes measured fastest near 100 neighbours
  }
  switch (g) {
    case 32: launch_real_g<T, 32>(c, a, vin, vout, mode, s); break;
    case 16: launch_real_g<T, 16>(c, a, vin, vout, mode, s); break;
    case 8: launch_real_g<T, 8>(c, a, vin, vout, mode, s); break;
    case 4: launch_real_g<T, 4>(c, a, vin, vout, mode, s); break;
    default: launch_real_g<T, 1>(c, a, vin, vout, mode, s);
  }
}

// The three rotation scalars of the 11-moment form at r (4 reals per node): linear
// interpolation in FP32; in FP64 cubic Lagrange interpolation with the same
// one-sided stencils at the r = 2a node as lookup().
__device__ __forceinline__ void rot_lookup(const float *tab, const RealArgs &a, float r, float g[3]) {
  float x = r * (float)a.inv_dr;
  int q = min((int)x, a.len - 2);
  float t = x - (float)q;
  const float4 u = ((const float4 *)tab)[q], v = ((const float4 *)tab)[q + 1];
  g[0] = fmaf(t, v.x - u.x, u.x);
  g[1] = fmaf(t, v.y - u.y, u.y);
  g[2] = fmaf(t, v.z - u.z, u.z);
}
__device__ __forceinline__ void rot_lookup(const double *tab, const RealArgs &a, double r, double g[3]) {
  double x = r * a.inv_dr;
  int q = min((int)x, a.len - 2);
  int b = q - 1;
  if (q < a.k2) b = min(b, a.k2 - 3);
  else b = max(b, a.k2);
  b = max(0, min(b, a.len - 4));
  double t = x - (double)b;
  const double c6 = 1.0 / 6.0, u0 = t * (t - 1), u1 = (t - 2) * (t - 3);
  const double w0 = -c6 * (t - 1) * u1, w1 = 0.5 * t * u1, w2 = -0.5 * u0 * (t - 3), w3 = c6 * u0 * (t - 2);
  const double *r0 = tab + 4 * (size_t)b;
#pragma unroll
  for (int k = 0; k < 3; ++k)
    g[k] = w0 * __ldg(r0 + k) + w1 * __ldg(r0 + 4 + k) + w2 * __ldg(r0 + 8 + k) + w3 * __ldg(r0 + 12 + k);
}

// The 11-moment real-space product (Sec. 2.2.1 rigid-particle relation): rows of 12
// slots, [F(3), L(3), s(5), -] in and [U(3), Omega(3), e(5), -] out.  Per pair, the
// 8 x 8 force-stresslet terms of k_real plus the rotation couplings
//   U += gF rh x L,   Omega += gF rh x F + gL1 L + gL2 (rh.L) rh + 2 gL2 (S rh) x rh,
//   e += gL2 symY(rh x L, rh)
// (gF, gL1, gL2 the rotation scalars); self terms self_uf, self_ol, self_es.  G lanes
// per particle walk its neighbour records, neighbours' rows from the cell-ordered copy.
template <typename T, int G>
__global__ void __launch_bounds__(256) k_real11(RealArgs a, const SysDev *__restrict__ sys,
                                                const int64_t *__restrict__ p0, const int *__restrict__ active,
                                                int *queue, int nitems, const int *__restrict__ nstart,
                                                const typename V4<T>::t *__restrict__ geo,
                                                const T *__restrict__ vin, const T *__restrict__ vcell,
                                                T *__restrict__ vout, const T *__restrict__ tab,
                                                const T *__restrict__ rtab, T self_ol) {
  using T4 = typename V4<T>::t;
  for_each_item(queue, nitems, [&](int item) {
    const int64_t gid = ((int64_t)item * 256 + threadIdx.x) / G;
    const int sub = threadIdx.x % G;
    const int64_t i = gid < a.Ntot ? gid : a.Ntot - 1;
    const int si = find_sys(p0, a.nsys, i);
    const bool live = gid < a.Ntot && active[si];
    const SysDev &sd = sys[si];
    T o[11];
#pragma unroll
    for (int m = 0; m < 11; ++m) o[m] = 0;
    const int64_t k0 = sd.nbr0 + (i - sd.p0) * sd.slots;
    const int cnt = live ? min(nstart[i], sd.slots) : 0;
    for (int n = sub; n < cnt; n += G) {
      const T4 gg = geo[k0 + n];
      const int j = real_as_index<T>(gg.w);
      const T r2 = gg.x * gg.x + gg.y * gg.y + gg.z * gg.z;
      const T ir = sizeof(T) == 4 ? (T)rsqrtf((float)r2) : (T)1 / sqrt(r2), r = r2 * ir;
      const T rh[3] = {gg.x * ir, gg.y * ir, gg.z * ir};
      T f[7], gr[3];
      lookup<false, M_FULL>(tab, a, r, f);
      rot_lookup(rtab, a, r, gr);
      const T *row = vcell + 12 * (size_t)j;
      const T F[3] = {row[0], row[1], row[2]}, Lv[3] = {row[3], row[4], row[5]};
      const T s[5] = {row[6], row[7], row[8], row[9], row[10]};
      T v[3];
      Smul(s, rh, v);
      const T q = rh[0] * v[0] + rh[1] * v[1] + rh[2] * v[2];
      const T rf = rh[0] * F[0] + rh[1] * F[1] + rh[2] * F[2];
      const T rl = rh[0] * Lv[0] + rh[1] * Lv[1] + rh[2] * Lv[2];
      const T rxL[3] = {rh[1] * Lv[2] - rh[2] * Lv[1], rh[2] * Lv[0] - rh[0] * Lv[2], rh[0] * Lv[1] - rh[1] * Lv[0]};
      const T rxF[3] = {rh[1] * F[2] - rh[2] * F[1], rh[2] * F[0] - rh[0] * F[2], rh[0] * F[1] - rh[1] * F[0]};
      const T vxr[3] = {v[1] * rh[2] - v[2] * rh[1], v[2] * rh[0] - v[0] * rh[2], v[0] * rh[1] - v[1] * rh[0]};
      const T cu = f[3] * q + (f[1] - f[0]) * rf;
#pragma unroll
      for (int m = 0; m < 3; ++m) {
        o[m] += f[2] * v[m] + f[0] * F[m] + cu * rh[m] + gr[0] * rxL[m];
        o[3 + m] += gr[0] * rxF[m] + gr[1] * Lv[m] + gr[2] * rl * rh[m] + (T)2 * gr[2] * vxr[m];
      }
      T pv[3], sy[5], yr[5], yl[5];
#pragma unroll
      for (int m = 0; m < 3; ++m) pv[m] = f[5] * v[m] - (T)0.5 * f[2] * F[m];
      symY(pv, rh, sy);
      symY(rh, rh, yr);
      symY(rxL, rh, yl);
      const T cy = (T)0.5 * (f[6] * q - f[3] * rf);
#pragma unroll
      for (int m = 0; m < 5; ++m) o[6 + m] += f[4] * s[m] + sy[m] + cy * yr[m] + gr[2] * yl[m];
    }
#pragma unroll
    for (int off = G / 2; off > 0; off >>= 1)
#pragma unroll
      for (int m = 0; m < 11; ++m) o[m] += __shfl_xor_sync(0xffffffffu, o[m], off, G);
    if (live && sub == 0) {
      const T *me = vin + 12 * (size_t)i;
      T *out = vout + 12 * (size_t)i;
#pragma unroll
      for (int m = 0; m < 3; ++m) {
        out[m] = o[m] + (T)a.self_uf * me[m];
        out[3 + m] = o[3 + m] + self_ol * me[3 + m];
      }
#pragma unroll
      for (int m = 0; m < 5; ++m) out[6 + m] = o[6 + m] + (T)a.self_es * me[6 + m];
      out[11] = 0;
    }
  });
}

// vcell12[k] = vin12[list[k]] (12-real rows).
template <typename T>
__global__ void k_cell_gather12(int64_t N, const int *__restrict__ list, const T *__restrict__ vin,
                                T *__restrict__ vcell) {
  const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= 12 * N) return;
  const int64_t k = e / 12;
  vcell[e] = vin[12 * (int64_t)list[k] + (e - 12 * k)];
}

// vcell[k] = cell_row(vin[list[k]]): the rows of the input vector in cell-list order.
template <typename T>
__global__ void k_cell_gather(int64_t N, const int *__restrict__ list, const typename V4<T>::t *__restrict__ vin,
                              typename V4<T>::t *__restrict__ vcell) {
  const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= N) return;
  const int64_t j = list[k];
  typename V4<T>::t lo, hi;
  load_row(vin, j, lo, hi);
  cell_row(lo, hi);
  store_row(vcell, k, lo, hi);
}

// Harmonic overlap repulsion F_i = sum_j k (2a - r_ij) rh_ij over neighbours
// closer than 2a (from the list's separation records), written in user order.  OV_LANES
// lanes share a particle's list; a comparison in the record's own type, a rounding
// margin above contact, keeps the FP64 arithmetic to the few pairs near or in contact
// (all 105 neighbours in FP64 on one thread took 144 us at N = 3000; now 12 us).
constexpr int OV_LANES = 8;
template <typename T>
__global__ void k_overlap(const SysDev *__restrict__ sys, const int64_t *__restrict__ p0, int nsys, int64_t Ntot,
                          double contact, double kspring, const int *__restrict__ nstart,
                          const typename V4<T>::t *__restrict__ geo, const int *__restrict__ perm, T *F) {
  const int64_t gid = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) / OV_LANES;
  const int sub = threadIdx.x % OV_LANES;
  const bool live = gid < Ntot;
  const int64_t i = live ? gid : Ntot - 1;
  const SysDev &sd = sys[find_sys(p0, nsys, i)];
  const T near2 = (T)(contact * contact * 1.00001);
  double f[3] = {0, 0, 0};
  const int64_t k0 = sd.nbr0 + (i - sd.p0) * sd.slots;
  const int cnt = live ? min(nstart[i], sd.slots) : 0;
  for (int n = sub; n < cnt; n += OV_LANES) {
    const typename V4<T>::t g = geo[k0 + n];
    if (g.x * g.x + g.y * g.y + g.z * g.z > near2) continue;
    const double d[3] = {(double)g.x, (double)g.y, (double)g.z};
    double r = sqrt(d[0] * d[0] + d[1] * d[1] + d[2] * d[2]);
    if (r >= contact || r == 0.0) continue;
    double c = kspring * (contact - r) / r;
    for (int m = 0; m < 3; ++m) f[m] += c * d[m];
  }
#pragma unroll
  for (int o = OV_LANES / 2; o > 0; o >>= 1)
    for (int m = 0; m < 3; ++m) f[m] += __shfl_xor_sync(0xffffffffu, f[m], o);
  if (live && sub == 0) {
    const int64_t u = perm[i];
    for (int m = 0; m < 3; ++m) F[3 * u + m] = (T)f[m];
  }
}

}  // namespace

pse_status overlap_force(pse_ctx *c, double kspring, void *F, cudaStream_t s) {
  c->nlaunch += 1;
  const int64_t N = c->p.N;
  const unsigned nb = (unsigned)ceil_div(N * OV_LANES, 256);
  if (c->prec == PSE_MIXED)
    k_overlap<float><<<nb, 256, 0, s>>>(c->d_sys, c->d_p0, c->nsys, N, 2.0 * c->p.a, kspring, c->d_nbr_start,
                                        (const float4 *)c->d_nbr_geo, c->d_perm, (float *)F);
  else
    k_overlap<double><<<nb, 256, 0, s>>>(c->d_sys, c->d_p0, c->nsys, N, 2.0 * c->p.a, kspring, c->d_nbr_start,
                                         (const double4_32a *)c->d_nbr_geo, c->d_perm, (double *)F);
  PSE_CUDA_TRY(c, cudaGetLastError());
  return PSE_OK;
}

// vout = M_r vin for the current configuration (sorted order, [N][8]); rows of
// inactive suspensions are left untouched.
pse_status real_apply(pse_ctx *c, const void *vin, void *vout, int mode, cudaStream_t s, bool gathered) {
  StageTimer timer(c, PSE_STAGE_REAL, s, mode);
  c->nlaunch += 1;
  RealArgs a;
  a.Ntot = c->p.N;
  a.nsys = c->nsys;
  a.len = c->table_len;
  a.k2 = c->table_k2;
  a.inv_dr = 1.0 / c->table_dr;
  a.self_uf = c->self_uf;
  a.self_es = c->self_es;
  if (!gathered) c->nlaunch += 1;
  const unsigned nb = (unsigned)ceil_div(c->p.N, 256);
  if (c->prec == PSE_MIXED) {
    if (!gathered)
      k_cell_gather<float><<<nb, 256, 0, s>>>(c->p.N, c->d_cell_list, (const float4 *)vin, (float4 *)c->d_vcell);
    launch_real<float>(c, a, vin, vout, mode, s);
  } else {
    if (!gathered)
      k_cell_gather<double><<<nb, 256, 0, s>>>(c->p.N, c->d_cell_list, (const double4_32a *)vin,
                                               (double4_32a *)c->d_vcell);
    launch_real<double>(c, a, vin, vout, mode, s);
  }
  PSE_CUDA_TRY(c, cudaGetLastError());
  return PSE_OK;
}

// vout12 = M_r vin12 for the 11-moment form (12-slot rows, sorted order).
pse_status real_apply11(pse_ctx *c, const void *vin12, void *vout12, cudaStream_t s) {
  StageTimer timer(c, PSE_STAGE_REAL, s);
  c->nlaunch += 2;
  RealArgs a;
  a.Ntot = c->p.N;
  a.nsys = c->nsys;
  a.len = c->table_len;
  a.k2 = c->table_k2;
  a.inv_dr = 1.0 / c->table_dr;
  a.self_uf = c->self_uf;
  a.self_es = c->self_es;
  constexpr int G = 4;
  const int64_t items = ceil_div(a.Ntot * G, 256);
  const unsigned ng = (unsigned)ceil_div(12 * c->p.N, 256);
  int *q = next_queue(c);
  if (c->prec == PSE_MIXED) {
    static std::atomic<int> per_sm{0};
    k_cell_gather12<float><<<ng, 256, 0, s>>>(c->p.N, c->d_cell_list, (const float *)vin12, (float *)c->d_vcell12);
    auto kern = k_real11<float, G>;
    const unsigned grid = persistent_grid(c, kern, 256, 0, items, per_sm);
    kern<<<grid, 256, 0, s>>>(a, c->d_sys, c->d_p0, c->d_active, q, (int)items, c->d_nbr_start,
                              (const float4 *)c->d_nbr_geo, (const float *)vin12, (const float *)c->d_vcell12,
                              (float *)vout12, (const float *)c->d_table, (const float *)c->d_table_rot,
                              (float)c->self_ol);
  } else {
    static std::atomic<int> per_sm{0};
    k_cell_gather12<double><<<ng, 256, 0, s>>>(c->p.N, c->d_cell_list, (const double *)vin12,
                                               (double *)c->d_vcell12);
    auto kern = k_real11<double, G>;
    const unsigned grid = persistent_grid(c, kern, 256, 0, items, per_sm);
    kern<<<grid, 256, 0, s>>>(a, c->d_sys, c->d_p0, c->d_active, q, (int)items, c->d_nbr_start,
                              (const double4_32a *)c->d_nbr_geo, (const double *)vin12,
                              (const double *)c->d_vcell12, (double *)vout12, (const double *)c->d_table,
                              (const double *)c->d_table_rot, c->self_ol);
  }
  PSE_CUDA_TRY(c, cudaGetLastError());
  return PSE_OK;
}

}  // namespace pse
