// Configuration set-up: wrapping, binning by spreading tile, counting sort,
// per-particle spreading/real-space records, linked-cell list and neighbour list.
//
// Sorted order = by the spreading tile that holds the first grid index of a
// particle's Gaussian support; the spreading and interpolation kernels visit the
// 2x2x2 neighbouring bins of their tile, and the pair sum walks a neighbour list
// built from cells of side >= r_cut (Sec. 2.3.1, linked-cell lists).
#include <algorithm>
#include <cmath>

#include "device_common.cuh"
#include "pse_internal.cuh"

namespace pse {
namespace {

constexpr int SCAN_NT = 256, SCAN_IPT = 8, SCAN_BLK = SCAN_NT * SCAN_IPT;

// Exclusive scan of in[0..n) into out (in-place allowed) per block of SCAN_BLK items.
__global__ void k_scan_block(const int *in, int *out, int64_t n, int *block_sums) {
  __shared__ int warp_tot[SCAN_NT / 32];
  int64_t base = (int64_t)blockIdx.x * SCAN_BLK + (int64_t)threadIdx.x * SCAN_IPT;
  int v[SCAN_IPT], tot = 0;
#pragma unroll
  for (int i = 0; i < SCAN_IPT; ++i) {
    int64_t idx = base + i;
    v[i] = idx < n ? in[idx] : 0;
    tot += v[i];
  }
  int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  int incl = tot;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    int t = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += t;
  }
  if (lane == 31) warp_tot[w] = incl;
  __syncthreads();
  if (w == 0) {
    int x = lane < SCAN_NT / 32 ? warp_tot[lane] : 0, xi = x;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      int t = __shfl_up_sync(0xffffffffu, xi, o);
      if (lane >= o) xi += t;
    }
    if (lane < SCAN_NT / 32) warp_tot[lane] = xi - x;  // exclusive warp offsets
    if (lane == SCAN_NT / 32 - 1 && block_sums) block_sums[blockIdx.x] = xi;
  }
  __syncthreads();
  int run = warp_tot[w] + incl - tot;
#pragma unroll
  for (int i = 0; i < SCAN_IPT; ++i) {
    int64_t idx = base + i;
    if (idx < n) out[idx] = run;
    run += v[i];
  }
}

__global__ void k_scan_add(int *out, int64_t n, const int *offs) {
  int64_t base = (int64_t)blockIdx.x * SCAN_BLK;
  int add = offs[blockIdx.x];
  for (int64_t i = threadIdx.x; i < SCAN_BLK; i += blockDim.x) {
    int64_t idx = base + i;
    if (idx < n) out[idx] += add;
  }
}

__device__ __forceinline__ double wrap_coord(double x, double L) {
  if (__double2hiint(x) >= 0 && x < L) return x;  // already inside: fmod would return x itself
  x = fmod(x, L);
  if (x < 0) x += L;
  if (x >= L) x = 0.0;
  return x;
}

// floor(x / y) or rint(x / y) of the rounded FP64 quotient, for 0 <= x / y < 2^20, as an
// integer and as a double.  The reciprocal product q = x * (1/y) lies within 1e-9 of the
// rounded quotient, so its floor (rint) is the same unless q lies within 2^-19 of an
// integer (a half-integer); there the division decides.  At sm_103a's FP64 rate (one warp
// instruction per 16 cycles) the FP64 instructions of k_bin and k_derive are their time:
// adding 2^52 leaves the integer in the low word, and the closeness test reads the high
// word, so a quotient costs a product and three sums (2^20 particles: k_bin 93 -> 53 us,
// k_derive 144 -> 89 us; 1000: 5.4 -> 4.7 and 7.7 -> 5.7).
struct Quot {
  int n;
  double f;
};
__device__ __forceinline__ Quot quot_floor(double x, double y, double iy) {
  constexpr double M = 4503599627370496.0;  // 2^52
  const double q = x * iy, s = __dadd_rd(q, M), f = s - M;
  const int hi = __double2hiint(q - f);  // the fraction (exact) between 2^-19 and 1 - 2^-19?
  if (hi >= 0x3EC00000 && hi < 0x3FEFFFFC) return {__double2loint(s), f};
  const double e = floor(x / y);
  return {(int)e, e};
}
__device__ __forceinline__ Quot quot_rint(double x, double y, double iy) {
  constexpr double M = 6755399441055744.0;  // 1.5 * 2^52
  const double q = x * iy, s = q + M, f = s - M;
  const int hi = __double2hiint(q - f) & 0x7fffffff;  // the distance from f below 0.5 - 2^-19?
  if (hi < 0x3FDFFFF8) return {__double2loint(s), f};
  const double e = rint(x / y);
  return {(int)e, e};
}

// First grid index of the support of a particle at wrapped coordinate x.
__device__ __forceinline__ Quot support_start(double x, double h, double ih, int P) {
  Quot q = (P & 1) ? quot_rint(x, h, ih) : quot_floor(x, h, ih);
  const int below = (P - 1) / 2;
  q.n -= below;
  q.f -= (double)below;
  return q;
}

// Wraps particle u (user order) of its suspension into [0, L) and counts it in
// the spreading tile that holds the first grid index of its support, refined by
// the 4 x 4 x 4 sub-block of the tile (so that the sorted order is spatially
// coherent inside a tile: neighbours' records then lie close together).
__global__ void k_bin(const SysDev *__restrict__ sys, const int64_t *__restrict__ p0, int nsys, int64_t Ntot,
                      int P, const double *pos, double *posw, int *tile_key, int *rank, int *tile_cnt, int *bad) {
  int64_t u = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (u >= Ntot) return;
  const SysDev &b = sys[find_sys(p0, nsys, u)];
  int iw[3];
  double xin[3];
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    xin[d] = pos[3 * u + d];
    // not finite: the exponent bits of the high word are all set
    if ((__double2hiint(xin[d]) & 0x7ff00000) == 0x7ff00000) {
      atomicOr(bad, 1);
      xin[d] = 0.0;
    }
  }
  if (b.def) {  // lattice coordinates z = A^{-1} x (Sec. 2.3.3); everything below works on z
    const double z0 = b.Ai[0] * xin[0] + b.Ai[1] * xin[1] + b.Ai[2] * xin[2];
    const double z1 = b.Ai[3] * xin[0] + b.Ai[4] * xin[1] + b.Ai[5] * xin[2];
    const double z2 = b.Ai[6] * xin[0] + b.Ai[7] * xin[1] + b.Ai[8] * xin[2];
    xin[0] = z0;
    xin[1] = z1;
    xin[2] = z2;
  }
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    const double x = wrap_coord(xin[d], b.L);
    posw[3 * u + d] = x;
    iw[d] = wrapi(support_start(x, b.h, b.inv_h, P).n, b.Ng);
  }
  int tk = b.tile0 + ((iw[2] / b.T[2]) * b.nt[1] + iw[1] / b.T[1]) * b.nt[0] + iw[0] / b.T[0];
  int sub = (((iw[2] % b.T[2]) * SUB_SIDE / b.T[2]) * SUB_SIDE + (iw[1] % b.T[1]) * SUB_SIDE / b.T[1]) * SUB_SIDE +
            (iw[0] % b.T[0]) * SUB_SIDE / b.T[0];
  tk = tk * SUB_BLOCKS + sub;
  tile_key[u] = tk;
  rank[u] = atomicAdd(&tile_cnt[tk], 1);
}

// tile_start[t] = fine_start[t * SUB_BLOCKS] for t = 0 .. ntiles
__global__ void k_tile_starts(int64_t ntiles, const int *fine_start, int *tile_start) {
  int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t <= ntiles) tile_start[t] = fine_start[t * SUB_BLOCKS];
}

__global__ void k_scatter(int64_t N, const int *key, const int *start, const int *rank, int *perm, int *inv) {
  int64_t u = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (u >= N) return;
  const int i = start[key[u]] + rank[u];
  perm[i] = (int)u;
  inv[u] = i;
}

template <typename T>
__global__ void k_derive(const SysDev *__restrict__ sys, const int64_t *__restrict__ p0, int nsys, int64_t Ntot,
                         int P, const int *perm, const double *posw, int4 *sp_i0, typename V4<T>::t *sp_d0,
                         void *rs, int *cell_key, int *rank, int *cell_cnt) {
  int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= Ntot) return;
  const SysDev &b = sys[find_sys(p0, nsys, i)];
  int u = perm[i];
  double x[3], xc[3];  // position, offset from the cell's corner
  int iw[3], c[3];
  T d0[3];
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    x[d] = posw[3 * (int64_t)u + d];
    const Quot i0 = support_start(x[d], b.h, b.inv_h, P);
    iw[d] = wrapi(i0.n, b.Ng);
    d0[d] = (T)(i0.f * b.h - x[d]);
    Quot q = quot_floor(x[d], b.cs, b.inv_cs);
    if (q.n >= b.nc) q = {b.nc - 1, (double)(b.nc - 1)};
    c[d] = q.n;
    xc[d] = x[d] - q.f * b.cs;
  }
  sp_i0[i] = make_int4(iw[0], iw[1], iw[2], c[0] | (c[1] << 10) | (c[2] << 20));  // w: the cell, at most 1023 a side
  typename V4<T>::t dd;
  dd.x = d0[0];
  dd.y = d0[1];
  dd.z = d0[2];
  dd.w = 0;
  sp_d0[i] = dd;
  if (sizeof(T) == 4) {
    ((float4 *)rs)[i] = make_float4((float)xc[0], (float)xc[1], (float)xc[2], (float)c[0]);
  } else {
    ((double4_32a *)rs)[i] = make_double4_32a(x[0], x[1], x[2], 0.0);
  }
  int ck = b.cell0 + (c[2] * b.nc + c[1]) * b.nc + c[0];
  cell_key[i] = ck;
  rank[i] = atomicAdd(&cell_cnt[ck], 1);
}

// Cell list: the particles of every cell, and a copy of their records (cell
// offsets or positions) in the same order, so that the neighbour search reads
// contiguous records.
template <typename T>
__global__ void k_cell_scatter(int64_t N, int *cell_key, const int *start, const int *rank, int *list,
                               const typename V4<T>::t *rs, typename V4<T>::t *rs_cell) {
  int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= N) return;
  const int k = start[cell_key[i]] + rank[i];
  list[k] = (int)i;
  rs_cell[k] = rs[i];
  cell_key[i] = k;  // from here on: the particle's own position in the cell list
}

// Neighbour list in one pass, one warp per cell: for each particle i of the cell and
// each neighbour j (r < r_cut, minimum image within its own suspension) the separation
// x_i - x_j and j go into i's own row of slots, and the row's length into cnt[i]; per
// suspension the total and the largest count are accumulated for the host's capacity
// check.  The stencil is 5 x 5 x 5 cells (every cell once when there are fewer than 5
// per side): its 25 x runs of cells are ranges of the cell-ordered records, and the warp
// walks their concatenation 32 candidates at a time, one per lane (a reduced bit mask of
// the runs that start in the batch tells each lane its run), so the records are read
// coalesced once per cell and tested against all its particles, NP of them at a time in
// registers; a ballot places the hits in consecutive slots.  Runs that wrap around the
// box in x have a second part, walked in a second pass.
//
// Bound by instruction issue (about 60 % of the slots; a quarter of the candidates are
// neighbours, so the compaction and not the distance is most of a test).  One thread per
// particle, as before, read the candidates of 32 particles from 32 places (L1
// wavefronts) and left small systems with a few warps of a long serial loop; the FP64
// form also divided by L for every candidate.  Measured, before and after: N = 3000 155
// -> 23 us, 64 suspensions of 160000 284 -> 196, sheared cell of 150000 465 -> 294, 2^20
// (r_cut 7.07, 105 neighbours) 1180 -> 1037, FP64 form at 11000 1102 -> 125.  Dilute
// systems take k_nbr_sparse (use_sparse).
// DEF: deformed lattice (Sec. 2.3.3): records and cells hold lattice coordinates z,
// and each candidate's separation is mapped to x_i - x_j = A (z_i - z_j) before the
// test, so the stored separations are Cartesian as for the cube.
constexpr int NBR_NT = 256;

// Suspension of a cell (SysDev::cell0 increases).
__device__ __forceinline__ int find_cell_sys(const SysDev *sys, int nsys, int64_t cell) {
  int lo = 0, hi = nsys - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (sys[mid].cell0 <= cell) lo = mid;
    else hi = mid - 1;
  }
  return lo;
}

// Difference of two cell coordinates to the nearest image (unchanged in [-nc/2, nc/2]).
__device__ __forceinline__ int cell_offset(int t, int nc) {
  t -= t > nc / 2 ? nc : 0;
  return t + (t < -(nc / 2) ? nc : 0);
}

__device__ __forceinline__ void add_totals(unsigned long long *tot, int si, int lane, unsigned long long sum, int big) {
  if (lane == 0) {
    atomicAdd(&tot[2 * si], sum);
    atomicMax(&tot[2 * si + 1], (unsigned long long)big);
  }
}

// x_i - x_j for a particle's coordinates c and a candidate's record q; sx, sy, sz: cells (FP32) or
// box lengths (FP64) to the nearest image.
template <typename T, bool DEF, bool WIDE>
__device__ __forceinline__ typename V4<T>::t nbr_sep(const T c[3], const typename V4<T>::t &q, T sx, T sy, T sz, T cs,
                                                     T L, const T *A) {
  typename V4<T>::t rec;
  if (sizeof(T) == 4) {
    rec.x = fma(sx, cs, c[0] - q.x);
    rec.y = fma(sy, cs, c[1] - q.y);
    rec.z = fma(sz, cs, c[2] - q.z);
  } else {
    rec.x = c[0] - q.x;
    rec.y = c[1] - q.y;
    rec.z = c[2] - q.z;
    if (WIDE) {  // the nearest image is s box lengths away (pairs beyond it are further than r_cut)
      rec.x -= L * sx;
      rec.y -= L * sy;
      rec.z -= L * sz;
    }
  }
  if (!WIDE) {
    rec.x -= L * rint(rec.x / L);
    rec.y -= L * rint(rec.y / L);
    rec.z -= L * rint(rec.z / L);
  }
  if constexpr (DEF) {  // x_i - x_j = A (z_i - z_j)
    const T zx = rec.x, zy = rec.y, zz = rec.z;
    rec.x = A[0] * zx + A[1] * zy + A[2] * zz;
    rec.y = A[3] * zx + A[4] * zy + A[5] * zz;
    rec.z = A[6] * zx + A[7] * zy + A[8] * zz;
  }
  return rec;
}

// The runs of one pass (lane r: start, length and y / z offsets of run r) walked for up to
// NP particles of the cell.
template <typename T, bool DEF, bool WIDE, int NP>
struct NbrWalk {
  using T4 = typename V4<T>::t;
  const T4 *rs_cell;
  T4 *geo;
  int lane, np, kb;          // particles kb .. kb + np - 1 of the cell list
  T cx;                      // the cell's x index
  int icx, nc;
  T cs, L, A[DEF ? 9 : 1];   // suspension constants in registers (the stores of the records keep the
                             // compiler from holding values read through a reference)
  T ctr[NP][3];
  int at[NP], lim[NP];       // next free entry and end of each particle's row of slots

  // T4 record q of candidate k; sx, sy, sz: cells (FP32) or box lengths (FP64) to the nearest image
  __device__ __forceinline__ void test(const T4 &q, int k, bool live, T sx, T sy, T sz) {
    const unsigned below = (1u << lane) - 1u;
    if (sizeof(T) == 4) {
      if (WIDE) sx += cx - (T)q.w;
      else sx = (T)cell_offset(icx - (int)q.w, nc);
    }
#pragma unroll
    for (int p = 0; p < NP; ++p) {
      if (p < np) {
        T4 rec = nbr_sep<T, DEF, WIDE>(ctr[p], q, sx, sy, sz, cs, L, A);
        const bool hit = rec.x * rec.x + rec.y * rec.y + rec.z * rec.z < rc2 && live && k != kb + p;
        const unsigned hits = __ballot_sync(0xffffffffu, hit);
        const int to = at[p] + __popc(hits & below);
        if (hit && to < lim[p]) {  // separation x_i - x_j and the neighbour's cell-list position
          rec.w = index_as_real<T>(k);
          geo[to] = rec;
        }
        at[p] += __popc(hits);
      }
    }
  }
  T rc2;

  // total candidates in nruns runs; lane r < nruns: run r starts `beg` candidates in, at
  // record delta + beg
  __device__ __forceinline__ void walk(int total, int nruns, int beg, int delta, T ry, T rz, T wx) {
    int r0 = -1;  // the last run that starts before the batch
    for (int base = 0; base < total; base += 32) {
      const bool live = base + lane < total;
      const unsigned d = (unsigned)(beg - base);
      const unsigned marks = __reduce_or_sync(0xffffffffu, lane < nruns && d < 32u ? 1u << d : 0u);
      const int r = r0 + __popc(marks & (0xffffffffu >> (31 - lane)));
      r0 += __popc(marks);
      const int k = __shfl_sync(0xffffffffu, delta, r) + base + lane;
      const T sy = __shfl_sync(0xffffffffu, ry, r), sz = __shfl_sync(0xffffffffu, rz, r);
      T4 q = rs_cell[live ? k : 0];
      test(q, k, live, wx, sy, sz);
    }
  }
};

// One cell; done(i, n) receives each particle (sorted index) and its neighbour count.
template <typename T, bool DEF, bool WIDE, typename Done>
__device__ __forceinline__ void nbr_cell(const SysDev &a, int64_t cell, int k0, int k1, T rc2,
                                         const typename V4<T>::t *rs_cell, const int *__restrict__ cell_start,
                                         const int *__restrict__ cell_list, typename V4<T>::t *geo, int *s_run,
                                         Done &&done) {
  constexpr int NP = sizeof(T) == 4 ? 4 : 2;
  const int lane = threadIdx.x & 31;
  const int nc = a.nc, slots = a.slots, rel = (int)(cell - a.cell0);
  const int cx = rel % nc, cy = (rel / nc) % nc, cz = rel / (nc * nc);
  const int span = WIDE ? 5 : nc, x0 = WIDE ? cx - 2 : 0, x1 = WIDE ? cx + 2 : nc - 1;
  // lane r owns x run r of the stencil: its cells' y and z offsets from this cell
  // (nearest image, in cells; in box lengths for FP64) and its one or two ranges
  int part_s[2] = {0, 0}, part_n[2] = {0, 0};
  T oy = 0, oz = 0;
  if (lane < span * span) {
    int ry = lane % span, rz = lane / span;
    if (WIDE) {
      ry += cy - 2;
      rz += cz - 2;
    }
    const int wy = ry < 0 ? -1 : (ry >= nc ? 1 : 0), wz = rz < 0 ? -1 : (rz >= nc ? 1 : 0);
    const int row = a.cell0 + ((rz - wz * nc) * nc + (ry - wy * nc)) * nc;
    oy = sizeof(T) == 4 ? (T)cell_offset(cy - ry, nc) : (T)wy;
    oz = sizeof(T) == 4 ? (T)cell_offset(cz - rz, nc) : (T)wz;
    part_s[0] = cell_start[row + max(x0, 0)];
    part_n[0] = cell_start[row + min(x1, nc - 1) + 1] - part_s[0];
    if (x0 < 0) {  // cells [x0 + nc, nc)
      part_s[1] = cell_start[row + x0 + nc];
      part_n[1] = cell_start[row + nc] - part_s[1];
    } else if (x1 >= nc) {  // cells [0, x1 - nc]
      part_s[1] = cell_start[row];
      part_n[1] = cell_start[row + x1 - nc + 1] - part_s[1];
    }
  }
  const int nparts = x0 < 0 || x1 >= nc ? 2 : 1;
  NbrWalk<T, DEF, WIDE, NP> w;
  w.rs_cell = rs_cell;
  w.geo = geo;
  w.lane = lane;
  w.cx = (T)cx;
  w.icx = cx;
  w.nc = nc;
  w.cs = sizeof(T) == 4 ? (T)a.csf : (T)a.cs;
  w.L = sizeof(T) == 4 ? (T)a.Lf : (T)a.L;
  if constexpr (DEF) {
#pragma unroll
    for (int i = 0; i < 9; ++i) w.A[i] = sizeof(T) == 4 ? (T)a.Af[i] : (T)a.A[i];
  }
  w.rc2 = rc2;
  for (w.kb = k0; w.kb < k1; w.kb += NP) {
    w.np = min(NP, k1 - w.kb);
#pragma unroll
    for (int p = 0; p < NP; ++p) {
      const int k = min(w.kb + p, k1 - 1);
      const typename V4<T>::t c = rs_cell[k];
      w.ctr[p][0] = c.x;
      w.ctr[p][1] = c.y;
      w.ctr[p][2] = c.z;
      w.at[p] = (int)(a.nbr0 + ((int64_t)cell_list[k] - a.p0) * slots);
      w.lim[p] = w.at[p] + slots;
    }
    for (int part = 0; part < nparts; ++part) {
      // nonempty runs first, in order
      const int pn = part ? part_n[1] : part_n[0], ps = part ? part_s[1] : part_s[0];
      const unsigned have = __ballot_sync(0xffffffffu, pn > 0);
      const int nruns = __popc(have);
      __syncwarp();
      if (pn > 0) s_run[__popc(have & ((1u << lane) - 1u))] = lane;
      __syncwarp();
      const int from = lane < nruns ? s_run[lane] : 0;
      const int rn = __shfl_sync(0xffffffffu, pn, from), rs = __shfl_sync(0xffffffffu, ps, from);
      const T ry = __shfl_sync(0xffffffffu, oy, from), rz = __shfl_sync(0xffffffffu, oz, from);
      int inc = lane < nruns ? rn : 0;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int u = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += u;
      }
      const int total = __shfl_sync(0xffffffffu, inc, 31), beg = inc - rn;
      // the second part wraps in x: its cells lie nc cells (one box length) further
      const T wrap = part ? (x0 < 0 ? (T)1 : (T)-1) : (T)0;
      w.walk(total, nruns, beg, rs - beg, ry, rz, sizeof(T) == 4 ? wrap * (T)nc : -wrap);
    }
#pragma unroll
    for (int p = 0; p < NP; ++p)
      if (p < w.np) done(cell_list[w.kb + p], w.at[p] - (w.lim[p] - slots));
  }
}

// FP32: 64 registers, four 256-thread CTAs per SM (about 9 % faster than three, although
// the cell's set-up then spills).
template <typename T, bool DEF>
__global__ void __launch_bounds__(NBR_NT, sizeof(T) == 4 ? 4 : 1)
    k_nbr(const SysDev *__restrict__ sys, int nsys, int64_t ncells, float rc2f, double rc2, const void *rs_cell,
          const int *__restrict__ cell_start, const int *__restrict__ cell_list, int *cnt, typename V4<T>::t *geo,
          unsigned long long *tot, int *ovf) {
  using T4 = typename V4<T>::t;
  __shared__ int s_run[NBR_NT / 32][32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const T r2max = sizeof(T) == 4 ? (T)rc2f : (T)rc2;
  const int64_t step = (int64_t)gridDim.x * (NBR_NT / 32);
  int si = -1, big = 0;
  unsigned long long sum = 0;
  for (int64_t cell = (int64_t)blockIdx.x * (NBR_NT / 32) + warp; cell < ncells; cell += step) {
    const int k0 = cell_start[cell], k1 = cell_start[cell + 1];
    if (k0 == k1) continue;
    const int sn = find_cell_sys(sys, nsys, cell);
    if (sn != si) {  // the totals of the suspension just left
      if (si >= 0) add_totals(tot, si, lane, sum, big);
      si = sn;
      sum = 0;
      big = 0;
    }
    const SysDev &a = sys[si];
    const int slots = a.slots;
    auto done = [&](int i, int n) {
      if (lane == 0) {
        cnt[i] = n;
        if (n > slots) atomicOr(ovf, 1);
      }
      sum += (unsigned)n;
      big = max(big, n);
    };
    if (a.nc >= 5)
      nbr_cell<T, DEF, true>(a, cell, k0, k1, r2max, (const T4 *)rs_cell, cell_start, cell_list, geo, s_run[warp], done);
    else
      nbr_cell<T, DEF, false>(a, cell, k0, k1, r2max, (const T4 *)rs_cell, cell_start, cell_list, geo, s_run[warp], done);
  }
  if (si >= 0) add_totals(tot, si, lane, sum, big);
}

// The same list, one thread per particle, for systems of mostly empty cells (use_sparse):
// a thread streams through the cell-ordered records of its runs, NB of them loaded before
// the first is tested.  Bound by the latency of that walk; 10^6 particles at a volume fraction of
// 0.01 take 177 us, 983 with a warp per cell.  Returns the particle's neighbour count; self: its own
// cell-list position, packed: its cell.
template <typename T, bool DEF, bool WIDE>
__device__ __forceinline__ int nbr_particle(const SysDev &a, int self, int packed, T r2max,
                                            const typename V4<T>::t *__restrict__ rs_cell,
                                            const int *__restrict__ cell_start, typename V4<T>::t *row_geo) {
  using T4 = typename V4<T>::t;
  constexpr int NB = 4;
  const int nc = a.nc, slots = a.slots, cell0 = a.cell0;
  const T cs = sizeof(T) == 4 ? (T)a.csf : (T)a.cs, L = sizeof(T) == 4 ? (T)a.Lf : (T)a.L;
  T A[DEF ? 9 : 1];
  if constexpr (DEF) {
#pragma unroll
    for (int m = 0; m < 9; ++m) A[m] = sizeof(T) == 4 ? (T)a.Af[m] : (T)a.A[m];
  }
  const int cx = packed & 1023, cy = (packed >> 10) & 1023, cz = packed >> 20;
  const int span = WIDE ? 5 : nc, y0 = WIDE ? cy - 2 : 0, z0 = WIDE ? cz - 2 : 0;
  const int x0 = WIDE ? cx - 2 : 0, x1 = WIDE ? cx + 2 : nc - 1;
  const T4 own = rs_cell[self];
  const T ctr[3] = {own.x, own.y, own.z};
  int n = 0;
  for (int iz = 0; iz < span; ++iz)
    for (int iy = 0; iy < span; ++iy) {
      const int rz = z0 + iz, ry = y0 + iy;
      const int wz = rz < 0 ? -1 : (rz >= nc ? 1 : 0), wy = ry < 0 ? -1 : (ry >= nc ? 1 : 0);
      const int row = cell0 + ((rz - wz * nc) * nc + (ry - wy * nc)) * nc;
      const T sy = sizeof(T) == 4 ? (T)(WIDE ? 2 - iy : cell_offset(cy - ry, nc)) : (T)wy;
      const T sz = sizeof(T) == 4 ? (T)(WIDE ? 2 - iz : cell_offset(cz - rz, nc)) : (T)wz;
      // cells [x0, x1], in two ranges where they wrap
      for (int wx = x0 < 0 ? -1 : 0; wx <= (x1 >= nc ? 1 : 0); ++wx) {
        const int kb = cell_start[row + max(x0 - wx * nc, 0)];
        const int ke = cell_start[row + min(x1 - wx * nc, nc - 1) + 1];
        for (int k = kb; k < ke; k += NB) {
          T4 q[NB];
#pragma unroll
          for (int u = 0; u < NB; ++u)
            if (k + u < ke) q[u] = rs_cell[k + u];
#pragma unroll
          for (int u = 0; u < NB; ++u) {
            if (k + u >= ke) break;
            T sx = (T)wx;
            if (sizeof(T) == 4) sx = WIDE ? (T)(cx - wx * nc) - (T)q[u].w : (T)cell_offset(cx - (int)q[u].w, nc);
            T4 rec = nbr_sep<T, DEF, WIDE>(ctr, q[u], sx, sy, sz, cs, L, A);
            if (rec.x * rec.x + rec.y * rec.y + rec.z * rec.z < r2max && k + u != self) {
              if (n < slots) {
                rec.w = index_as_real<T>(k + u);
                row_geo[n] = rec;
              }
              ++n;
            }
          }
        }
      }
    }
  return n;
}

template <typename T, bool DEF>
__global__ void __launch_bounds__(128)
    k_nbr_sparse(const SysDev *__restrict__ sys, const int64_t *__restrict__ p0, int nsys, int64_t Ntot, float rc2f,
                 double rc2, const typename V4<T>::t *__restrict__ rs_cell, const int4 *__restrict__ sp_i0,
                 const int *__restrict__ cell_start, const int *__restrict__ cell_pos, int *cnt, typename V4<T>::t *geo,
                 unsigned long long *tot, int *ovf) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= Ntot) return;
  const int si = find_sys(p0, nsys, i), self = cell_pos[i], packed = sp_i0[i].w;
  const SysDev &a = sys[si];
  const T r2max = sizeof(T) == 4 ? (T)rc2f : (T)rc2;
  typename V4<T>::t *row_geo = geo + a.nbr0 + (i - a.p0) * a.slots;
  const int n = a.nc >= 5 ? nbr_particle<T, DEF, true>(a, self, packed, r2max, rs_cell, cell_start, row_geo)
                          : nbr_particle<T, DEF, false>(a, self, packed, r2max, rs_cell, cell_start, row_geo);
  cnt[i] = n;
  if (n > a.slots) atomicOr(ovf, 1);
  // one atomic addition per warp when its particles share a suspension
  const unsigned act = __activemask();
  const int leader = __ffs(act) - 1;
  if (__all_sync(act, si == __shfl_sync(act, si, leader))) {
    const unsigned sum = __reduce_add_sync(act, (unsigned)n), big = __reduce_max_sync(act, (unsigned)n);
    if ((int)(threadIdx.x & 31) == leader) add_totals(tot, si, 0, sum, (int)big);
  } else {
    add_totals(tot, si, 0, (unsigned)n, n);
  }
}

void *alloc_dev(pse_ctx *c, size_t bytes) {
  void *p = nullptr;
  if (cudaMalloc(&p, bytes) != cudaSuccess) return nullptr;
  c->allocs.push_back(p);
  c->dev_bytes += (int64_t)bytes;
  return p;
}

// One thread per particle where most cells hold one particle or none: a warp per cell then
// has few candidates for its lanes and few particles to test them against, and walks past
// the empty cells one after the other.  A thread's serial walk over 25 runs takes 20 us and more,
// so there have to be many cells for it (600 per SM).  Measured, us, warp / thread:
//   FP32  N = 10^6: 0.1 particles per cell 983 / 177, 0.86 708 / 346, 1.5 756 / 535, 2.2 860 / 734
//         300000: 0.02 850 / 63, 0.87 230 / 132, 1.5 243 / 204, 2.1 265 / 263;  200000: 1.5 167 / 163, 1.8 174 / 205
//         60000: 0.22 61 / 31, 0.87 55 / 51, 1.3 56 / 65;  30000: 0.11 44 / 26, 0.44 33 / 38;  10000: 0.11 21 / 23
//   FP64  300000: 0.11 477 / 489, 0.21 435 / 686;  100000: 0.02 499 / 103;  30000: 0.02 164 / 42, 0.11 74 / 81
bool use_sparse(const pse_ctx *c) {
  if (c->ncells < 600 * (int64_t)c->nsm) return false;
  return c->prec == PSE_MIXED ? 2 * c->ncells >= c->p.N + 65536 : c->ncells >= 16 * c->p.N;
}

// A warp per cell; beyond 16 blocks per SM each walks several cells, so the totals take
// one atomic addition per warp and not per cell.
template <typename T, bool DEF>
void launch_nbr(pse_ctx *c, double rc2, cudaStream_t s) {
  using T4 = typename V4<T>::t;
  if (use_sparse(c)) {
    k_nbr_sparse<T, DEF><<<(unsigned)ceil_div(c->p.N, 128), 128, 0, s>>>(
        c->d_sys, c->d_p0, c->nsys, c->p.N, (float)rc2, rc2, (const T4 *)c->d_rs_cell, (const int4 *)c->d_sp_i0,
        c->d_cell_start, c->d_cell_key, c->d_nbr_start, (T4 *)c->d_nbr_geo, c->d_nbr_tot, c->d_flag + 1);
    return;
  }
  auto kern = k_nbr<T, DEF>;
  const int64_t nb = std::min<int64_t>(ceil_div(c->ncells, NBR_NT / 32), (int64_t)c->nsm * 16);
  kern<<<(unsigned)nb, NBR_NT, 0, s>>>(c->d_sys, c->nsys, c->ncells, (float)rc2, rc2, c->d_rs_cell, c->d_cell_start,
                                       c->d_cell_list, c->d_nbr_start, (typename V4<T>::t *)c->d_nbr_geo,
                                       c->d_nbr_tot, c->d_flag + 1);
}

}  // namespace

// Exclusive scan of n+1 ints (in[n] must be 0) so that out[n] is the total.
pse_status exclusive_scan(pse_ctx *c, int *buf, int64_t n1, cudaStream_t s) {
  // level sizes
  int64_t sizes[8];
  int levels = 0;
  int64_t len = n1;
  while (true) {
    sizes[levels++] = len;
    if (len <= SCAN_BLK) break;
    len = ceil_div(len, SCAN_BLK);
    if (levels >= 7) break;
  }
  int *bufs[8];
  bufs[0] = buf;
  int64_t off = 0;
  for (int l = 1; l < levels; ++l) {
    bufs[l] = c->d_scan_tmp + off;
    off += sizes[l];
  }
  c->nlaunch += 2 * levels - 1;
  for (int l = 0; l < levels; ++l) {
    int64_t nb = ceil_div(sizes[l], SCAN_BLK);
    k_scan_block<<<(unsigned)nb, SCAN_NT, 0, s>>>(bufs[l], bufs[l], sizes[l], l + 1 < levels ? bufs[l + 1] : nullptr);
  }
  for (int l = levels - 2; l >= 0; --l) {
    int64_t nb = ceil_div(sizes[l], SCAN_BLK);
    k_scan_add<<<(unsigned)nb, SCAN_NT, 0, s>>>(bufs[l], sizes[l], bufs[l + 1]);
  }
  PSE_CUDA_TRY(c, cudaGetLastError());
  return PSE_OK;
}

int64_t scan_tmp_ints(int64_t n1) {
  int64_t tot = 0, len = n1;
  while (len > SCAN_BLK) {
    len = ceil_div(len, SCAN_BLK);
    tot += len;
  }
  return tot + 16;
}

// Slot layout of the neighbour list: per suspension `slots` entries per particle.
int64_t layout_neighbours(pse_ctx *c) {
  int64_t off = 0;
  for (int q = 0; q < c->nsys; ++q) {
    c->hs[q].nbr0 = off;
    off += (int64_t)c->hs[q].slots * c->hs[q].N;
  }
  return off;
}

// Builds the sorted configuration for positions d_pos (device, user order, FP64).
pse_status setup_config(pse_ctx *c, const double *d_pos, cudaStream_t s) {
  StageTimer timer(c, PSE_STAGE_SETUP, s);
  c->nlaunch += 5;  // bin, scatter, derive, cell scatter, neighbour list (+ scans)
  const Params &p = c->p;
  const int64_t N = p.N;
  const int ns = c->nsys;
  unsigned nb = (unsigned)ceil_div(N, 256);
  const int64_t nfine = c->ntiles * SUB_BLOCKS;
  // status words (a graph clears them once, for both of its builds), totals and counts
  char *clear = c->capturing ? (char *)c->d_nbr_tot : (char *)c->d_flag;
  PSE_CUDA_TRY(c, cudaMemsetAsync(clear, 0, (char *)(c->d_cell_start + c->ncells + 1) - clear, s));
  k_bin<<<nb, 256, 0, s>>>(c->d_sys, c->d_p0, ns, N, p.P, d_pos, c->d_posw, c->d_tile_key, c->d_rank, c->d_fine_start,
                           c->d_flag);
  PSE_TRY(exclusive_scan(c, c->d_fine_start, nfine + 1, s));
  k_scatter<<<nb, 256, 0, s>>>(N, c->d_tile_key, c->d_fine_start, c->d_rank, c->d_perm, c->d_inv);
  if (c->n_cubic < ns) {
    c->nlaunch += 1;
    k_tile_starts<<<(unsigned)ceil_div(c->ntiles + 1, 256), 256, 0, s>>>(c->ntiles, c->d_fine_start, c->d_tile_start);
  }
  if (c->prec == PSE_MIXED)
    k_derive<float><<<nb, 256, 0, s>>>(c->d_sys, c->d_p0, ns, N, p.P, c->d_perm, c->d_posw, (int4 *)c->d_sp_i0,
                                       (float4 *)c->d_sp_d0, c->d_rs, c->d_cell_key, c->d_rank, c->d_cell_start);
  else
    k_derive<double><<<nb, 256, 0, s>>>(c->d_sys, c->d_p0, ns, N, p.P, c->d_perm, c->d_posw, (int4 *)c->d_sp_i0,
                                        (double4_32a *)c->d_sp_d0, c->d_rs, c->d_cell_key, c->d_rank, c->d_cell_start);
  PSE_TRY(exclusive_scan(c, c->d_cell_start, c->ncells + 1, s));
  if (c->prec == PSE_MIXED)
    k_cell_scatter<float><<<nb, 256, 0, s>>>(N, c->d_cell_key, c->d_cell_start, c->d_rank, c->d_cell_list,
                                             (const float4 *)c->d_rs, (float4 *)c->d_rs_cell);
  else
    k_cell_scatter<double><<<nb, 256, 0, s>>>(N, c->d_cell_key, c->d_cell_start, c->d_rank, c->d_cell_list,
                                              (const double4_32a *)c->d_rs, (double4_32a *)c->d_rs_cell);
  const double rc2 = p.rcut * p.rcut;
  for (int attempt = 0; attempt < 2; ++attempt) {
    if (attempt > 0) PSE_CUDA_TRY(c, cudaMemsetAsync(c->d_nbr_tot, 0, 2 * sizeof(unsigned long long) * ns, s));
    const bool def = c->lattice != 0;
    if (c->prec == PSE_MIXED) def ? launch_nbr<float, true>(c, rc2, s) : launch_nbr<float, false>(c, rc2, s);
    else def ? launch_nbr<double, true>(c, rc2, s) : launch_nbr<double, false>(c, rc2, s);
    if (c->capturing) return PSE_OK;  // the graph's caller checks the flags and the totals afterwards
    PSE_CUDA_TRY(c, cudaMemcpyAsync(c->h_status, c->d_flag, 16 + 2 * sizeof(unsigned long long) * ns,
                                    cudaMemcpyDeviceToHost, s));
    PSE_CUDA_TRY(c, cudaGetLastError());
    PSE_CUDA_TRY(c, cudaStreamSynchronize(s));
    if (c->h_status[0]) {
      c->err = "non-finite particle position";
      return PSE_ERR_NONFINITE;
    }
    bool grow = false;
    c->npairs = 0;
    c->npairs_sys.assign(ns, 0);
    for (int q = 0; q < ns; ++q) {
      c->npairs_sys[q] = (int64_t)c->h_nbr_tot[2 * q];
      c->npairs += c->npairs_sys[q];
      int64_t mx = (int64_t)c->h_nbr_tot[2 * q + 1];
      if (mx > c->hs[q].slots) {
        c->hs[q].slots = (int)((mx + 15) / 8 * 8);  // a particle has more neighbours than slots
        grow = true;
      }
    }
    if (!grow) break;
    // enlarge the list and rebuild once
    int64_t cap = layout_neighbours(c);
    if ((double)cap > 2.0e9) {
      c->err = "neighbour list exceeds 2^31 entries";
      return PSE_ERR_INVALID_ARG;
    }
    void *gq = alloc_dev(c, 4 * c->ts * (size_t)cap);
    if (!gq) {
      c->err = "cannot allocate neighbour list";
      return PSE_ERR_OOM;
    }
    c->d_nbr_geo = gq;  // the old list stays in c->allocs and is freed at destroy
    c->nbr_cap = cap;
    ++c->layout_version;
    PSE_CUDA_TRY(c, cudaMemcpyAsync(c->d_sys, c->hs.data(), sizeof(SysDev) * ns, cudaMemcpyHostToDevice, s));
  }
  PSE_CUDA_TRY(c, cudaGetLastError());
  return PSE_OK;
}

}  // namespace pse
