// Interpolation sigma Q^T (Sec. 2.3.2, Eq. WSops2) for tiles of up to 16^3 points, mixed precision,
// with the whole support region of a group of particles staged in shared memory.
//
// Work item: one z-layer of a tile, i.e. the particles whose support starts lie in
// the tile and in one of its SUB_SIDE layers of at most 16/SUB_SIDE planes (one
// contiguous range of the sort by tile and sub-block).  Their supports lie inside the region
// [t0x, t0x + wx + P - 1) x [t0y, t0y + wy + P - 1) x [z0, z0 + planes + P - 1),
// which the CTA copies from the grid (periodic wrap) into shared memory in the
// TileL layout.  Each particle is then read out once and complete by one quarter
// warp: its 8 lanes take the P x P columns of the support (column l + 8 s on lane
// l), walk each column along z, and the quarter sums its lanes with three
// shuffles, so every output row is written by one lane with no atomic addition
// (the tile-owned kernel splits a support over up to 8 tiles and adds the parts).
// Against the general kernel on 12^3 tiles at N_g = 36: 5 components 54 -> 8.1 us, 8
// components 33 -> 7.7; the 11-moment product's at N_g = 128 188 -> 97 and 134 -> 50 us.
// Two CTAs share an SM (about 83 KB each for 5 components, P = 6), so one CTA's
// staging overlaps the other's read-out; where staging is most of the work an item is a whole
// tile whose planes pass through a ring (halo_may_ring).
//
// Bound by L1: two thirds of the shared-memory and copy wavefronts of the one-layer form
// are staging (8 per 32 four-byte copies; 3969 points for 64 particles), the rest the
// read-out's 16-byte reads.  Lanes over 4 components x 8 points (conflict-free stores)
// made the copies slower (574 -> 1411 us at 2^20), 16 lanes per particle the read-out
// (540 -> 600).
//
// The weights are exp, not exp2 with log2(e) in the exponent: the special-function unit's 2^x
// is low by 4.8e-8 on average (exp is high by 0.6e-8), and with three such weights to a grid
// point the wave part came out smaller by 0.8e-7 on average over 25 sizes, at an error of 3e-7.
// At no cost: a weight takes part in P^2 or more products.
#include "wave_common.cuh"

namespace pse {
namespace {

// One layer per work item: 512 threads, two CTAs per SM.  A whole tile per item: 1024 threads
// and a ring of planes, one CTA per SM.
constexpr int HALO_THREADS = 512, RING_THREADS = 1024;

// 4 bytes from global to shared memory without a register round trip (cp.async,
// cached in L1); completion is awaited with cp_async_wait before a barrier.
__device__ __forceinline__ void cp_async4(float *smem, const float *gmem) {
  const unsigned s = (unsigned)__cvta_generic_to_shared(smem);
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(s), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
// Waits until at most `n` of the thread's latest groups are in flight.
template <int n>
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;\n" ::"n"(n) : "memory");
}
constexpr int LAYER = CUBE / SUB_SIDE;  // planes of support starts per work item

template <int P, bool RING = false> struct Halo {
  static constexpr int R = CUBE + P - 1;           // region side along x and y
  static constexpr int RZ = LAYER + P - 1;         // region depth along z
  static constexpr int NZ = RING ? RZ + LAYER : RZ;  // planes held: a layer's region, and the next layer's new planes
  static constexpr int RX = tile_rx(R, P);         // padded row (RX = P mod 8: conflict-free quarter reads)
  static constexpr int ZS = R * RX;                // plane stride (points)
  static constexpr int NPT = NZ * ZS;              // points of the staged planes
  static constexpr int LP = 8;                      // lanes of a particle
  static constexpr int NCOL = (P * P + LP - 1) / LP;  // column passes per lane
};

// DEF: deformed lattice with z orthogonal to the sheared plane (as the
// register-column spreading): the x-y weight of each support column is its own
// exponential of the x-y quadratic form; the z weights use G_zz.
// COMP0: first grid component read (grid components COMP0 .. COMP0 + C - 1 go
// to output slots SLOT0 .. SLOT0 + C - 1).  ROW: slots per particle row of vout.
//
// RING: an item is a tile.  The planes stay in a ring of slots, so a layer stages only the planes that the one below it did not have (21
// planes for the four layers of a 16^3 tile at P = 6, not 36), and they are copied while
// the layer below is read out.
template <int C, int SLOT0, int P, bool DEF, int COMP0, int ROW, bool RING>
__global__ void __launch_bounds__(RING ? RING_THREADS : HALO_THREADS, RING ? 1 : 2)
    k_interp_halo(WaveArgs wa, int *queue, const int4 *__restrict__ sp_i0, const float4 *__restrict__ sp_d0,
                  const int *__restrict__ fine_start, const float *__restrict__ grid_all, float *__restrict__ vout) {
  using H = Halo<P, RING>;
  constexpr int R = H::R, NZ = H::NZ, RX = H::RX, ZS = H::ZS, LP = H::LP, NT = RING ? RING_THREADS : HALO_THREADS;
  extern __shared__ __align__(32) unsigned char smem_raw[];
  TileL<float, C> tl;
  tl.init(smem_raw, H::NPT);
  const int lane = threadIdx.x & 31, group = lane / LP, sub = lane % LP, warp = threadIdx.x >> 5;
  constexpr int per_tile = RING ? 1 : SUB_SIDE;
  for_each_item(queue, wa.ntiles * per_tile, [&](int item) {
    const int tile = item / per_tile, kz0 = item % per_tile, kz1 = RING ? SUB_SIDE : kz0 + 1;
    const int si = find_sys(wa.tile0, wa.nsys, tile);
    const SysDev &a = wa.sys[si];
    if (wave_skip(wa, si, a)) return;
    const int Ng = a.Ng;
    int t[3], t0[3];
    tile_of(a, tile - a.tile0, t, t0);
    const int *fs = fine_start + (int64_t)tile * SUB_BLOCKS;
    constexpr int LB = SUB_SIDE * SUB_SIDE;  // sub-blocks of a layer
    if (fs[kz0 * LB] == fs[kz1 * LB]) return;
    // layer kz holds the planes [first(kz), first(kz + 1)) of the tile: 4 z / T = kz
    const int wz = tile_width(a, t[2], 2);
    auto first = [&](int kz) { return min((kz * a.T[2] + SUB_SIDE - 1) / SUB_SIDE, wz); };
    const int rx = tile_width(a, t[0], 0) + P - 1, ry = tile_width(a, t[1], 1) + P - 1;
    const float *grid = grid_all + a.grid0 + COMP0 * a.gstride;
    const int64_t gs = a.gstride;  // in a register: the copies keep the compiler from holding values read through `a`
    const bool whole = rx == R && ry == R;
    // planes [za, zb) (from the tile's origin, periodic) into the tile layout; plane z lies in
    // slot z mod NZ: asynchronous 4-byte copies (no register round trip), or for 5 components,
    // small supports and one layer per item loads and vector stores, U points per thread in
    // flight.  Unrolled: the copies' addresses take longer than the copies (8 components, P = 8,
    // 4096 tiles: 1123 us as a loop with gstride read per copy, 1023 so, 1057 unrolled 4; one
    // layer of 5 components, P = 6: 422 -> 384; the ring of 5 at P = 10 3457 unrolled 2, 3070 by 4)
    auto stage = [&](int za, int zb) {
      constexpr bool REGS = C == 5 && P <= 6 && !RING;
      constexpr int U = REGS ? 2 : 1, UNROLL = REGS || (C == 5 && RING) ? 4 : 2;
      const int n = (zb - za) * R * R;
#pragma unroll UNROLL
      for (int q0 = threadIdx.x; q0 < n; q0 += U * NT) {
        float v[U][C];
        int d[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
          const int q = q0 + u * NT, x = q % R, y = (q / R) % R, dz = q / (R * R), z = za + dz;
          const bool in = q < n && (whole || (x < rx && y < ry));  // a tile of fewer than 16 points
          d[u] = in ? (RING ? z % NZ : dz) * ZS + y * RX + x : -1;
          int gx = t0[0] + x, gy = t0[1] + y, gz = t0[2] + z;
          gx -= gx >= Ng ? Ng : 0;
          gy -= gy >= Ng ? Ng : 0;
          gz -= gz >= Ng ? Ng : 0;
          const float *g = grid + ((size_t)gz * Ng + gy) * Ng + gx;
          if (in) {
#pragma unroll
            for (int c = 0; c < C; ++c) {
              if (REGS) v[u][c] = __ldg(g + c * gs);
              else cp_async4(tl.comp(d[u], c), g + c * gs);
            }
          }
        }
        if (REGS) {
#pragma unroll
          for (int u = 0; u < U; ++u)
            if (d[u] >= 0) tl.store(d[u], v[u]);
        }
      }
      cp_async_commit();
    };
    const float nal = -(float)a.alpha, hs = (float)a.h, pref = (float)a.pref;
    const float kxx = DEF ? -(float)a.qa[0] : nal, kyy = DEF ? -(float)a.qa[1] : nal;
    const float kxy = DEF ? -(float)a.qa[3] : 0.f, kzz = DEF ? -(float)a.qa[2] : nal;
    stage(first(kz0), first(kz0 + 1) + P - 1);
    for (int kz = kz0; kz < kz1; ++kz) {
      const int zl = first(kz);
      if (RING && kz + 1 < kz1) {
        stage(first(kz + 1) + P - 1, first(kz + 2) + P - 1);
        cp_async_wait<1>();
      } else {
        cp_async_wait<0>();
      }
      __syncthreads();  // the layer's planes are staged
      const int beg = fs[kz * LB], end = fs[(kz + 1) * LB];
      // 32 / LP particles per warp per round (warp-uniform loop: the shuffles below run on
      // all 32 lanes)
      for (int base = beg + (32 / LP) * warp; base < end; base += NT / LP) {
        const int k = base + group;
        const bool live = k < end;
        const int ke = live ? k : end - 1;
        const int4 i0 = sp_i0[ke];
        const float4 d0 = sp_d0[ke];
        const int ex = i0.x - t0[0], ey = i0.y - t0[1], ez = i0.z - t0[2];  // in [0, 16), ez in the layer
        // 1D weights: lane sub < P holds the x, y and z weights of point sub (P <= 8,
        // the first lanes of a particle); a larger support has every lane form its own
        float wz[P], wx = 0.f, wy = 0.f;
        if constexpr (P <= 8) {
          const float f = (float)(sub < P ? sub : 0) * hs;
          const float ox = d0.x + f, oy = d0.y + f, oz = d0.z + f;
          wx = expf(nal * ox * ox);
          wy = expf(nal * oy * oy);
          const float wzl = expf(kzz * oz * oz);
#pragma unroll
          for (int j = 0; j < P; ++j) wz[j] = __shfl_sync(0xffffffffu, wzl, j, LP);
        } else {
#pragma unroll
          for (int j = 0; j < P; ++j) {
            const float oz = d0.z + (float)j * hs;
            wz[j] = expf(kzz * oz * oz);
          }
        }
        float acc[C];
#pragma unroll
        for (int c = 0; c < C; ++c) acc[c] = 0.f;
        const int s0 = RING ? ez % NZ : ez - zl, pb = ey * RX + ex;  // slot of the support's first plane
        constexpr int CU = P >= 8 ? 2 : H::NCOL;  // P = 8: partial unroll (register pressure)
#pragma unroll CU
        for (int s = 0; s < H::NCOL; ++s) {
          // this lane's column (px, py) = (c mod P, c / P) of the support, c = sub + LP s
          const int cc = sub + LP * s, px = cc % P, py = cc < P * P ? cc / P : 0;
          float wxy;
          if (DEF || P > 8) {  // the column's own x-y weight
            const float cx = d0.x + (float)px * hs, cy = d0.y + (float)py * hs;
            wxy = expf(kxx * cx * cx + kxy * cx * cy + kyy * cy * cy);
          } else {
            wxy = __shfl_sync(0xffffffffu, wx, px, LP) * __shfl_sync(0xffffffffu, wy, py, LP);
          }
          if (cc < P * P) {
            const int col = pb + py * RX + px;
#pragma unroll
            for (int jz = 0; jz < P; ++jz) {
              int sl = s0 + jz;
              if (RING) sl -= sl >= NZ ? NZ : 0;
              float vv[C];
              tl.load(col + sl * ZS, vv);
              const float w = wxy * wz[jz];
#pragma unroll
              for (int c = 0; c < C; ++c) acc[c] = fmaf(w, vv[c], acc[c]);
            }
          }
        }
#pragma unroll
        for (int o = LP / 2; o > 0; o >>= 1)
#pragma unroll
          for (int c = 0; c < C; ++c) acc[c] += __shfl_xor_sync(0xffffffffu, acc[c], o);
        // lane c of the particle adds component c
        float mine = acc[0];
#pragma unroll
        for (int c = 1; c < C; ++c) mine = sub == c ? acc[c] : mine;
        if (live && sub < C) {
          float *o = vout + ROW * (size_t)k + SLOT0 + sub;
          *o += pref * mine;
        }
      }
      __syncthreads();  // the planes are no longer read when the next ones overwrite them
    }
  });
}

// Staged bytes of C components with support P; a CTA may take 223 KB.
template <int C, int P, bool RING>
constexpr size_t halo_bytes() {
  return (size_t)Halo<P, RING>::NPT * (16 + (C == 5 ? 4 : (C == 8 ? 16 : 0)));
}

template <int C, int SLOT0, int P, bool DEF, int COMP0, int ROW, bool RING>
void launch_interp_halo_k(pse_ctx *c, const WaveArgs &a, void *vout, cudaStream_t s) {
  constexpr int NT = RING ? RING_THREADS : HALO_THREADS;
  static_assert(halo_bytes<C, P, RING>() <= 223 * 1024, "staged planes");
  static std::once_flag once;
  static OccCache occ;
  const size_t sm = TileL<float, C>::bytes((size_t)Halo<P, RING>::NPT);
  auto kern = k_interp_halo<C, SLOT0, P, DEF, COMP0, ROW, RING>;
  set_smem(kern, once);
  const unsigned grid = wave_grid(c, kern, sm, a.ntiles * (RING ? 1 : SUB_SIDE), occ, NT);
  int *q = next_queue(c);
  kern<<<grid, NT, sm, s>>>(a, q, (const int4 *)c->d_sp_i0, (const float4 *)c->d_sp_d0, c->d_fine_start,
                            (const float *)c->d_grid, (float *)vout);
}

// Whether an item is a whole tile (ring) or a layer.  A layer of a ring holds about 64
// particles for 128 places, so the ring gains where staging is most of the work: 8
// components, and 5 with large supports, from two tiles per SM on.  Measured, us, one layer
// / ring: 8 components, P = 6 69 / 60 at 343 tiles, 119 / 99 at 512, 931 / 673 at 4096
// (2^20 particles); 5 components, P = 8 98 / 86 at 512 and 1234 / 950 at 5832, P = 10 139 /
// 133 and 1847 / 1527; but P = 6 64 / 78 at 512, 384 / 446 at 4096 with 300000 particles,
// 499 / 528 with 2^20, and P = 5 538 / 595 at 5832; 3 components 420 / 467 at 4096.
template <int C, int P>
constexpr bool halo_may_ring() {
  return (C == 8 || (C == 5 && P >= 8)) && halo_bytes<C, P, true>() <= 223 * 1024;
}

template <int C, int SLOT0, int P, bool DEF, int COMP0, int ROW>
void launch_interp_halo(pse_ctx *c, const WaveArgs &a, void *vout, cudaStream_t s) {
  if constexpr (C == 8 && halo_bytes<C, P, false>() > 223 * 1024) {
    // the staged region of all components does not fit: components 0-4 and 5-7 in two passes
    launch_interp_halo<5, SLOT0, P, DEF, COMP0, ROW>(c, a, vout, s);
    launch_interp_halo<3, SLOT0 + 5, P, DEF, COMP0 + 5, ROW>(c, a, vout, s);
    c->nlaunch += 1;
  } else {
    if constexpr (halo_may_ring<C, P>())
      if (a.ntiles >= 2 * c->nsm) return launch_interp_halo_k<C, SLOT0, P, DEF, COMP0, ROW, true>(c, a, vout, s);
    launch_interp_halo_k<C, SLOT0, P, DEF, COMP0, ROW, false>(c, a, vout, s);
  }
}

template <int C, int SLOT0, bool DEF, int COMP0, int ROW>
void interp_halo_pd(pse_ctx *c, const WaveArgs &a, void *vout, cudaStream_t s) {
  switch (a.P) {
    case 5: launch_interp_halo<C, SLOT0, 5, DEF, COMP0, ROW>(c, a, vout, s); break;
    case 6: launch_interp_halo<C, SLOT0, 6, DEF, COMP0, ROW>(c, a, vout, s); break;
    case 10: launch_interp_halo<C, SLOT0, 10, DEF, COMP0, ROW>(c, a, vout, s); break;
    default: launch_interp_halo<C, SLOT0, 8, DEF, COMP0, ROW>(c, a, vout, s);
  }
}

template <int C, int SLOT0, int COMP0 = 0, int ROW = 8>
void interp_halo_p(pse_ctx *c, const WaveArgs &a, void *vout, cudaStream_t s) {
  if (c->lattice) interp_halo_pd<C, SLOT0, true, COMP0, ROW>(c, a, vout, s);
  else interp_halo_pd<C, SLOT0, false, COMP0, ROW>(c, a, vout, s);
}

}  // namespace

// Grids 0 .. 10 added to the 11 components of 12-slot rows.
void interp_halo11_launch(pse_ctx *c, const WaveArgs &a, void *vout12, cudaStream_t s) {
  interp_halo_p<8, 0, 0, 12>(c, a, vout12, s);
  interp_halo_p<3, 8, 8, 12>(c, a, vout12, s);
}

void interp_halo_launch(pse_ctx *c, const WaveArgs &a, void *vout, int mode, cudaStream_t s) {
  if (mode == M_FULL) interp_halo_p<8, 0>(c, a, vout, s);
  else if (mode == M_SE) interp_halo_p<5, 3>(c, a, vout, s);
  else interp_halo_p<3, 0>(c, a, vout, s);
}

}  // namespace pse
