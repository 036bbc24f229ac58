// Gaussian spreading Q (Sec. 2.3.2, Eq. WSops2).
//
// Persistent CTAs take output tiles (of any suspension) from a work counter.
// Warp w owns the tile's z-planes w, w + 16, ...: it scans the candidate
// particles whose support can cross its plane 32 at a time (a ballot picks the
// hits) and adds each hit's P x P footprint in the plane to the shared tile with
// plain read-modify-writes (each lane owns one (x, y) point of the footprint and
// updates all its components; no other warp touches the plane), so there are no
// atomics, the result is deterministic, and the warps never wait for one another
// between the clearing of a tile and its read-out.  The tile is then written
// once to the component-major grids with coalesced stores; no grid zeroing pass
// is needed because the tiles cover the grid.
#include "wave_common.cuh"

namespace pse {
namespace {

// moments [SLOT0, SLOT0 + C) of particle k (a ROW-slot row: 8, or 12 in the
// 11-moment product), read by the whole warp
template <typename T, int C, int SLOT0, int ROW = 8>
__device__ __forceinline__ void load_moments(const T *__restrict__ vin, int k, T mv[C]) {
  const T *row = vin + ROW * (size_t)k;
  if (sizeof(T) == 4 && SLOT0 == 3 && C == 5) {
    mv[0] = row[3];
    const float4 q = *(const float4 *)(row + 4);
    mv[1] = q.x;
    mv[2] = q.y;
    mv[3] = q.z;
    mv[4] = q.w;
  } else if (sizeof(T) == 4 && SLOT0 == 0 && C == 8) {
    const float4 q = *(const float4 *)row, r = *(const float4 *)(row + 4);
    mv[0] = q.x;
    mv[1] = q.y;
    mv[2] = q.z;
    mv[3] = q.w;
    mv[4] = r.x;
    mv[5] = r.y;
    mv[6] = r.z;
    mv[7] = r.w;
  } else {
#pragma unroll
    for (int c = 0; c < C; ++c) mv[c] = row[SLOT0 + c];
  }
}

// The one-dimensional Gaussian weights of a hit in one plane, one per lane: lanes [0, P)
// along x, [P, 2P) along y, lane 2P along z at the plane; exp(-alpha (d0 + j h)^2).
template <typename T>
__device__ __forceinline__ T plane_weight(int l, int P, int packed, T alpha, T hs, const typename V4<T>::t &d0) {
  if (l > 2 * P) return (T)0;
  int ex, ey, ez;
  unpack_offsets(packed, ex, ey, ez);
  const int j = l < P ? l : (l < 2 * P ? l - P : ez);
  const T o = (l < P ? d0.x : (l < 2 * P ? d0.y : d0.z)) + (T)j * hs;
  return exp(-alpha * o * o);
}

// ROW: slots per particle row of vin; COMP0: first grid component written.
//
// The FP64 form is bound by its FP64 instructions (one warp instruction per 16 cycles): per
// hit an exponential of about 25 and, per pass over the footprint, 2 + C.  A hit needs 2 P + 1
// weights, so for P <= 7 two hits share one exponential, and the few points that a whole
// pass would take beyond a multiple of 32 (4 at P = 6) go to a lane per component: 8
// components, P = 6, 11003 particles 375 -> 257 us (the shared exponential alone 291).
template <typename T, int C, int SLOT0, int PT, int ROW = 8, int COMP0 = 0>
__global__ void __launch_bounds__(WAVE_THREADS) k_spread(WaveArgs wa, int *queue, const int4 *__restrict__ sp_i0,
                                                         const typename V4<T>::t *__restrict__ sp_d0,
                                                         const T *__restrict__ vin, const int *__restrict__ fine_start,
                                                         T *__restrict__ grid_all) {
  // footprint points of a last pass that, with C lanes per point, fit one warp
  constexpr int LEFT = PT > 0 && PT * PT % 32 * C <= 32 ? PT * PT % 32 : 0;
  constexpr int NPASS = PT > 0 ? (PT * PT - LEFT + 31) / 32 : 1;
  constexpr int PZ = PT > 0 ? PT : 1;
  constexpr int HP = 2 * PZ + 1 <= 16 ? 2 : 1, HL = 32 / HP;
  using T4 = typename V4<T>::t;
  extern __shared__ __align__(32) unsigned char smem_raw[];
  for_each_item(queue, wa.ntiles, [&](int item) {
    const int si = find_sys(wa.tile0, wa.nsys, item);
    const SysDev &a = wa.sys[si];
    if (wave_skip(wa, si, a)) return;
    const int P = PT > 0 ? PT : wa.P, Ng = a.Ng, nitem = P * P;
    const int Tx = a.T[0], Ty = a.T[1], Tz = a.T[2];
    const int RX = tile_rx(Tx, P);
    const int npts = Tz * Ty * RX;
    TileL<T, C> tl;
    tl.init(smem_raw, npts);
    {
      T zero[C];
#pragma unroll
      for (int c = 0; c < C; ++c) zero[c] = (T)0;
      for (int q = threadIdx.x; q < npts; q += blockDim.x) tl.store(q, zero);
    }
    __syncthreads();  // cleared before any update or (for a tile with no particles) the read-out
    int t[3], t0[3], beg[8], cum[9];
    tile_of(a, item - a.tile0, t, t0);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const T alpha = sd_alpha<T>(a), hs = sd_h<T>(a), pref = sd_pref<T>(a);
    // this lane's (x, y) footprint point in every pass (fixed for the whole tile)
    int pjx[NPASS], pjy[NPASS];
    bool pok[NPASS];
#pragma unroll
    for (int ps = 0; ps < NPASS; ++ps) {
      int it = ps * 32 + lane;
      pok[ps] = it < nitem;
      pjx[ps] = pok[ps] ? it % P : 0;
      pjy[ps] = pok[ps] ? it / P : 0;
    }
    for (int lz = warp; lz < Tz; lz += WAVE_WARPS) {
      const int plane = lz * Ty * RX;
      const int nb = plane_bins(a, t, lz, P, fine_start, beg, cum);
      const int total = cum[nb];
      for (int base = 0; base < total; base += 32) {
        const int v = base + lane;
        int k = 0, ox = 0, oy = 0, jz = P;
        if (v < total) {
          k = candidate(v, nb, beg, cum);
          int oz;
          if (overlaps(a, P, t0, sp_i0[k], ox, oy, oz)) {
            jz = lz - oz;
            if (jz < 0) jz += Ng;
          }
        }
        // signed offsets fit the packing for any grid (a hit's offset is in (-P, T))
        const int pk = pack_offsets(signed_offset(ox, Ng, P), signed_offset(oy, Ng, P), jz < P ? jz : 0);
        unsigned hits = __ballot_sync(0xffffffffu, jz < P);
        while (hits) {
          if (PT > 0) {
            // HP hits at a time: HL lanes evaluate the 2 P + 1 weights of each
            int src[2];
            src[0] = __ffs(hits) - 1;
            hits &= hits - 1;
            const int nh = HP == 2 && hits ? 2 : 1;
            src[1] = nh == 2 ? __ffs(hits) - 1 : src[0];
            if (nh == 2) hits &= hits - 1;
            const int ms = lane < HL ? src[0] : src[1];
            const int km = __shfl_sync(0xffffffffu, k, ms), pm = __shfl_sync(0xffffffffu, pk, ms);
            const T wl = plane_weight(lane % HL, PZ, pm, alpha, hs, sp_d0[km]);
            for (int h = 0; h < nh; ++h) {
              const int l0 = h * HL;
              const int ke = __shfl_sync(0xffffffffu, km, l0);
              int ex, ey, ez;
              unpack_offsets(__shfl_sync(0xffffffffu, pm, l0), ex, ey, ez);
              ex += ex < 0 ? Ng : 0;  // back to offsets in [0, Ng)
              ey += ey < 0 ? Ng : 0;
              T mv[C];
              load_moments<T, C, SLOT0, ROW>(vin, ke, mv);
              const T wz = pref * __shfl_sync(0xffffffffu, wl, l0 + 2 * PZ);
#pragma unroll
              for (int ps = 0; ps < NPASS; ++ps) {
                const T wxy =
                    __shfl_sync(0xffffffffu, wl, l0 + pjx[ps]) * __shfl_sync(0xffffffffu, wl, l0 + PZ + pjy[ps]);
                int lx = ex + pjx[ps], ly = ey + pjy[ps];
                if (lx >= Ng) lx -= Ng;
                if (ly >= Ng) ly -= Ng;
                if (pok[ps] && lx < Tx && ly < Ty) {
                  const T wt = wxy * wz;
                  const int i = plane + ly * RX + lx;
                  T vv[C];
                  tl.load(i, vv);
#pragma unroll
                  for (int c = 0; c < C; ++c) vv[c] += wt * mv[c];
                  tl.store(i, vv);
                }
              }
              if (LEFT > 0) {  // the leftover points, a lane per point and component
                const int it = PZ * PZ - LEFT + min(lane / C, LEFT - 1), c = lane % C, jx = it % PZ, jy = it / PZ;
                const T wxy = __shfl_sync(0xffffffffu, wl, l0 + jx) * __shfl_sync(0xffffffffu, wl, l0 + PZ + jy);
                int lx = ex + jx, ly = ey + jy;
                if (lx >= Ng) lx -= Ng;
                if (ly >= Ng) ly -= Ng;
                if (lane < LEFT * C && lx < Tx && ly < Ty)
                  *tl.comp(plane + ly * RX + lx, c) += wxy * wz * vin[ROW * (size_t)ke + SLOT0 + c];
              }
              __syncwarp();  // the next particle may update the same points from other lanes
            }
          } else {  // any support size and any lattice: weights on the fly, exp(-alpha |A d|^2)
            const int src = __ffs(hits) - 1;
            hits &= hits - 1;
            const int ke = __shfl_sync(0xffffffffu, k, src);
            int ex, ey, ez;
            unpack_offsets(__shfl_sync(0xffffffffu, pk, src), ex, ey, ez);
            ex += ex < 0 ? Ng : 0;  // back to offsets in [0, Ng)
            ey += ey < 0 ? Ng : 0;
            const T4 d0 = sp_d0[ke];
            T mv[C];
            load_moments<T, C, SLOT0, ROW>(vin, ke, mv);
            const T dz = d0.z + (T)ez * hs;
            const T qz = sd_qa<T>(a, 2) * dz * dz, q4 = sd_qa<T>(a, 4) * dz, q5 = sd_qa<T>(a, 5) * dz;
            for (int ib = 0; ib < nitem; ib += 32) {
              const int it = ib + lane;
              const int jx = it % P, jy = it / P;
              int lx = ex + jx, ly = ey + jy;
              if (lx >= Ng) lx -= Ng;
              if (ly >= Ng) ly -= Ng;
              if (it < nitem && lx < Tx && ly < Ty) {
                const T dx = d0.x + (T)jx * hs, dy = d0.y + (T)jy * hs;
                const T q = sd_qa<T>(a, 0) * dx * dx + sd_qa<T>(a, 1) * dy * dy + sd_qa<T>(a, 3) * dx * dy + q4 * dx + q5 * dy + qz;
                const T wt = pref * exp(-q);
                const int i = plane + ly * RX + lx;
                T vv[C];
                tl.load(i, vv);
#pragma unroll
                for (int c = 0; c < C; ++c) vv[c] += wt * mv[c];
                tl.store(i, vv);
              }
            }
            __syncwarp();  // the next particle may update the same points from other lanes
          }
        }
      }
    }
    __syncthreads();
    T *grid = grid_all + a.grid0;
    const int tv = Tx * Ty * Tz;
    for (int q = threadIdx.x; q < tv; q += blockDim.x) {
      int x = q % Tx, y = (q / Tx) % Ty, z = q / (Tx * Ty);
      size_t g = ((size_t)(t0[2] + z) * Ng + (t0[1] + y)) * Ng + (t0[0] + x);
      T v[C];
      tl.load((z * Ty + y) * RX + x, v);
#pragma unroll
      for (int c = 0; c < C; ++c) grid[(COMP0 + c) * a.gstride + g] = v[c];
    }
    __syncthreads();  // the tile is read out before the next item clears it
  });
}

template <typename T, int C, int SLOT0, int PT, int ROW = 8, int COMP0 = 0>
void launch_spread(pse_ctx *c, const WaveArgs &a, const void *vin, cudaStream_t s) {
  static std::once_flag once;
  static OccCache occ;
  auto kern = k_spread<T, C, SLOT0, PT, ROW, COMP0>;
  set_smem(kern, once);
  size_t sm = wave_smem_max<T, C>(c, a.want);
  unsigned grid = wave_grid(c, kern, sm, a.ntiles, occ);
  int *q = next_queue(c);
  kern<<<grid, WAVE_THREADS, sm, s>>>(a, q, (const int4 *)c->d_sp_i0, (const typename V4<T>::t *)c->d_sp_d0,
                                      (const T *)vin, c->d_fine_start, (T *)c->d_grid);
}

template <typename T, int C, int SLOT0, int ROW = 8, int COMP0 = 0>
void spread_p(pse_ctx *c, const WaveArgs &a, const void *vin, cudaStream_t s) {
  if (c->lattice) return launch_spread<T, C, SLOT0, 0, ROW, COMP0>(c, a, vin, s);  // non-separable weights
  switch (a.P) {
    case 5: launch_spread<T, C, SLOT0, 5, ROW, COMP0>(c, a, vin, s); break;
    case 6: launch_spread<T, C, SLOT0, 6, ROW, COMP0>(c, a, vin, s); break;
    case 8: launch_spread<T, C, SLOT0, 8, ROW, COMP0>(c, a, vin, s); break;
    default: launch_spread<T, C, SLOT0, 0, ROW, COMP0>(c, a, vin, s);
  }
}

}  // namespace

// Suspensions with tiles of up to 16^3: grid columns in registers (default) or the
// shared-memory tile (bit 0 of option wave_kernel).
void spread_cubic(pse_ctx *c, const WaveArgs &a, const void *vin, int mode, cudaStream_t s) {
  if (c->opt.wave_kernel & 1) spread16_launch(c, a, vin, mode, s);
  else spread_col_launch(c, a, vin, mode, s);
}

void spread_launch(pse_ctx *c, const WaveArgs &a, const void *vin, int mode, cudaStream_t s) {
  if (c->n_cubic == c->nsys) return spread_cubic(c, a, vin, mode, s);
  WaveArgs ag = a;
  if (c->n_cubic > 0) {  // both kinds of suspensions: one launch each
    WaveArgs ac = a;
    ac.want = 1;
    ag.want = 0;
    spread_cubic(c, ac, vin, mode, s);
    c->nlaunch += 1;
  }
  if (c->prec == PSE_MIXED) {
    if (mode == M_SE || mode == M_SU) spread_p<float, 5, 3>(c, ag, vin, s);
    else spread_p<float, 8, 0>(c, ag, vin, s);
  } else {
    if (mode == M_SE || mode == M_SU) spread_p<double, 5, 3>(c, ag, vin, s);
    else spread_p<double, 8, 0>(c, ag, vin, s);
  }
}

// The 11 components [F, L, S] of 12-slot rows onto grids 0..10 of every suspension
// (two passes: 8 and 3 components).
void spread11_launch(pse_ctx *c, const void *vin12, cudaStream_t s) {
  WaveArgs a = wave_args(c);
  c->nlaunch += 2;
  if (c->n_cubic == c->nsys) return spread_col11_launch(c, a, vin12, s);
  if (c->prec == PSE_MIXED) {
    spread_p<float, 8, 0, 12, 0>(c, a, vin12, s);
    spread_p<float, 3, 8, 12, 8>(c, a, vin12, s);
  } else {
    spread_p<double, 8, 0, 12, 0>(c, a, vin12, s);
    spread_p<double, 3, 8, 12, 8>(c, a, vin12, s);
  }
}

}  // namespace pse
