// Kernels of the relativistic lattice Boltzmann update (arXiv 2205.04658) and the
// host launchers of one storage type.  Included once per storage type by
// rlbm_kernels_<type>.cu.
#pragma once

#include "rlbm_device.cuh"
#include "rlbm_launch.h"
#include "rlbm_stages.h"
#include "rlbm_tma.cuh"

#include <climits>
#include <type_traits>

namespace rlbm {

// The ghost column a cell at x also writes (INT_MIN: none): with x periodic, its image
// beyond the opposite edge; in an open channel, the last column repeats itself beyond the
// outflow edge and nothing is written into the inflow column.
__device__ __forceinline__ int ghost_col(int x, int nx, int walls) {
  if (walls & OPEN_X) return x == nx - 1 ? nx : INT_MIN;
  return x == 0 ? nx : (x == nx - 1 ? -1 : INT_MIN);
}
__device__ __forceinline__ int ghost_row(int y, int ny, int walls) {
  return (walls & (WALLS_Y | STRIP_Y)) ? INT_MIN : (y == 0 ? ny : (y == ny - 1 ? -1 : INT_MIN));
}
constexpr long long WAIT_CYCLES = 4000000000ll;  // ~2 s at 2 GHz: bounded TMA waits

// Bytes of the two buffers, ghosts and padding included, from which odd steps walk the lattice backwards
// (step_kernel).  The line lies between 724^2 FP32 (76 MB: no effect; 512^2, 40 MB, lost 4 %) and 896^2
// (117 MB: 22.7 -> 21.5 us per step); 1024^2 (152 MB) 29.1 -> 28.0, 4096^2 and FP16 within 1 %.
constexpr long long BACKWARDS_BYTES = 90000000ll;

template <typename S, int VS> struct Tile {
  static constexpr int Q = VSet<VS>::Q, TY = TileRows<S>::value;
  static constexpr int V = PadLayout<S>::V;
  static constexpr int XOFF = PadLayout<S>::XOFF;
  static constexpr int TXB = TILE_X + 2 * V;         // staged columns (16-byte granules on both sides)
  static constexpr int TYB = TY + 2;             // staged rows (one halo row each side)
  static constexpr int IN_BYTES = Q * TYB * TXB * (int)sizeof(S);
  static constexpr int IN_STRIDE = (IN_BYTES + 127) / 128 * 128;
  // stirring rows of the tile (at most MAX_SROWS k_y rows): G[row][TILE_X] (R4) and EY[row][TY]
  // (R2) after the populations; their size follows the shell at run time
  using R = typename RealOf<S>::type;
  static constexpr int MAX_SROWS = 16;
  static constexpr int G_ROW = TILE_X * 4 * (int)sizeof(R);
  static constexpr int EY_ROW = TY * 2 * (int)sizeof(R);
  static_assert(IN_STRIDE % 128 == 0 && G_ROW % 128 == 0, "TMA shared-memory destinations are 128-byte aligned");
  __host__ __device__ static constexpr int g_bytes(int rows) { return (rows * G_ROW + 127) / 128 * 128; }
  __host__ __device__ static constexpr int ey_bytes(int rows) { return (rows * EY_ROW + 127) / 128 * 128; }
  __host__ __device__ static constexpr int stage(int rows) { return IN_STRIDE + g_bytes(rows) + ey_bytes(rows); }
  __host__ __device__ static constexpr int smem(int nst, int rows) { return nst * stage(rows) + 64 + 128; }
};

// One cell per thread: the FP64 path.
// `release` is called once the staged tile has been read (by every thread); false: wind down.
template <typename S, int VS, bool MASK, bool FORCE, int CPT, class G, class W, class F>
__device__ __forceinline__ typename std::enable_if<CPT == 1, bool>::type
tile_cells(const unsigned char *stg, int ey_off, S *fout, int x0, int y0, int tid, const G &g, const W &wts,
           const Physics<typename RealOf<S>::type> &p, const Stir<typename RealOf<S>::type> &st, bool staged,
           unsigned *err, typename RealOf<S>::type *macro_out, F release) {
  using R = typename RealOf<S>::type;
  using V = VSet<VS>;
  using TL = Tile<S, VS>;
  constexpr int Q = V::Q;
    const int lx = tid % TILE_X, ly = tid / TILE_X;
    const int x = x0 + lx, y = y0 + ly;
    const S *tile = reinterpret_cast<const S *>(stg);
    const bool inside = x < g.nx && y < g.ny;
    const bool border = x0 == 0 || y0 == 0 || x0 + TILE_X >= g.nx || y0 + TL::TY >= g.ny;  // the tile's
    unsigned nb = 0;
    if (MASK && g.nbmask && inside) nb = g.nbmask[(long long)y * g.nx + x];
    const bool fluid = inside && !(MASK && (nb & 16u));
    R hn[Q], h[Q], Fx = p.body_x, Fy = p.body_y;
    if (fluid) {
      // pull-streaming from the staged tile: cell (lx, ly) at row ly + 1, column lx + V
      const int b0 = (ly + 1) * TL::TXB + lx + TL::V;
#pragma unroll
      for (int q = 0; q < Q; ++q) {
        const S *pl = tile + q * TL::TYB * TL::TXB + b0;
        const int sx = sgnx<VS>(q), sy = sgny<VS>(q);
        const R c = load_h_s<S, R>(pl);
        R acc = wts.beta[q][0] * c;
        if (sx != 0) {
          R v = load_h_s<S, R>(pl - sx);
          if (MASK && ((nb >> (4 - sx)) & 1u)) v = load_h_s<S, R>(tile + V::opp(q) * TL::TYB * TL::TXB + b0);
          acc = fma(wts.beta[q][1], v, acc);
        }
        if (sy != 0) {
          R v = load_h_s<S, R>(pl - sy * TL::TXB);
          if (MASK && ((nb >> (4 - 3 * sy)) & 1u)) v = load_h_s<S, R>(tile + V::opp(q) * TL::TYB * TL::TXB + b0);
          acc = fma(wts.beta[q][2], v, acc);
        }
        if (sx != 0 && sy != 0) {
          R v = load_h_s<S, R>(pl - sy * TL::TXB - sx);
          if (MASK && ((nb >> (4 - 3 * sy - sx)) & 1u)) v = load_h_s<S, R>(tile + V::opp(q) * TL::TYB * TL::TXB + b0);
          acc = fma(wts.beta[q][3], v, acc);
        }
        h[q] = acc;
      }
      if (FORCE) {  // F = sum_r Re[G_r(x) EY_r(y)], the table holding (Re, -Im)
        R Fx2 = R(0), Fy2 = R(0);
        for (int r = 0; r < st.nrows; ++r) {
          R4<R> G;
          R2<R> E;
          if (staged) {
            G = reinterpret_cast<const R4<R> *>(stg + TL::IN_STRIDE)[r * TILE_X + lx];
            E = reinterpret_cast<const R2<R> *>(stg + ey_off)[r * TL::TY + ly];
          } else {
            G = st.G_cur[(long long)r * g.nx + x];
            E = st.EY[(long long)r * st.eyp + y];
          }
          Fx = fma(G.x, E.x, Fx);
          Fx2 = fma(G.y, E.y, Fx2);
          Fy = fma(G.z, E.x, Fy);
          Fy2 = fma(G.w, E.y, Fy2);
        }
        Fx += Fx2;
        Fy += Fy2;
      }
    }
    if (!release()) return false;
    if (fluid) {
      const Mom<R> M = moments_of<R, R, VS, FORCE>(h);
      const Macro<R> m = cell_macro<R, VS>(h, M, p.vmax2);
      if (!m.ok) atomicOr(err, cell_error(m));
      if (macro_out) {  // the cell's Landau solution, force and streamed h, kept for the reverse sweep
        const long long nc = (long long)g.nx * g.ny, c = (long long)y * g.nx + x;
        macro_out[c] = m.eps_m1;
        macro_out[nc + c] = m.vx;
        macro_out[2 * nc + c] = m.vy;
        macro_out[3 * nc + c] = Fx;
        macro_out[4 * nc + c] = Fy;
#pragma unroll
        for (int q = 0; q < Q; ++q) macro_out[(5 + q) * nc + c] = h[q];
      }
      const Coll<R> cf = coll_coeffs<R, VS, FORCE>(M, m, p.omega0, p.fpref, Fx, Fy);
      collide_all<R, VS, FORCE>(cf, h, hn);
    } else {
#pragma unroll
      for (int q = 0; q < Q; ++q) hn[q] = R(0);
    }
    if (inside) {  // coalesced stores straight from registers (one 128-byte line per warp and plane)
      S *o = fout + (long long)(y + 1) * g.pitch + x + TL::XOFF;
#pragma unroll
      for (int q = 0; q < Q; ++q) o[q * g.plane] = store_h<S, R>(hn[q]);
    }
    // ghost copies of the periodic neighbours (boundary cells only)
    if (inside && border) {
      const int gxv = ghost_col(x, g.nx, g.walls);
      const int gyv = ghost_row(y, g.ny, g.walls);
      if (gxv != INT_MIN || gyv != INT_MIN) {
        const int px[3] = {gxv, x, gxv}, py[3] = {y, gyv, gyv};
        for (int a = 0; a < 3; ++a) {
          if (px[a] == INT_MIN || py[a] == INT_MIN) continue;
          S *o = fout + (long long)(py[a] + 1) * g.pitch + px[a] + TL::XOFF;
#pragma unroll
          for (int q = 0; q < Q; ++q) o[q * g.plane] = store_h<S, R>(hn[q]);
        }
      }
    }
    return true;
}

// Two cells per thread: cells (x, y) and (x, y + 1) of the 32 x 8 tile (y
// even), all per-cell arithmetic on packed FP32 pairs.  The FP32, FP16 and BF16 paths.  The
// two cells are adjacent rows, so the classes that move in y pull one of their rows for
// both (each such value is read from shared memory and converted once).
template <typename S, int VS, bool MASK, bool FORCE, int CPT, class G, class W, class F>
__device__ __forceinline__ typename std::enable_if<CPT == 2, bool>::type
tile_cells(const unsigned char *stg, int ey_off, S *fout, int x0, int y0, int tid, const G &g, const W &wts,
           const Physics<float> &p, const Stir<float> &st, bool staged, unsigned *err, float *macro_out, F release) {
  using V = VSet<VS>;
  using TL = Tile<S, VS>;
  using T = F2;
  constexpr int Q = V::Q;
  constexpr int DB = TL::TXB;  // smem offset of the second cell
  const int lx = tid % TILE_X, ly = tid / TILE_X;
  const int x = x0 + lx, yA = y0 + 2 * ly, yB = yA + 1;
  const S *tile = reinterpret_cast<const S *>(stg);
  const bool inA = x < g.nx && yA < g.ny, inB = x < g.nx && yB < g.ny;
  // whether the tile holds boundary cells
  const bool border = x0 == 0 || y0 == 0 || x0 + TILE_X >= g.nx || y0 + TL::TY >= g.ny;
  unsigned nbA = 0, nbB = 0;
  if (MASK && g.nbmask) {
    if (inA) nbA = g.nbmask[(long long)yA * g.nx + x];
    if (inB) nbB = g.nbmask[(long long)yB * g.nx + x];
  }
  const bool flA = inA && !(MASK && (nbA & 16u)), flB = inB && !(MASK && (nbB & 16u));
  const bool both = flA && flB;
  T hn[Q];
  {
    T Fx(p.body_x), Fy(p.body_y);
    if (FORCE) {
      // (before the pull: four rows of loads in flight need registers that h and its moments take later)
      // F = sum_r Re[G_r(x) EY_r(y)]: the pairs are (Re, -Im) of the table and (Re, Im) of the phase as
      // they lie in memory, so a row costs four multiply-adds and two 16-byte loads for both cells
      // (pairs over the two cells took a copy of each table value into both lanes and two negations)
      T axA(0.0f), ayA(0.0f), axB(0.0f), ayB(0.0f);
      auto add = [&](const float4 &G, const float4 &E) {
        const T gx(G.x, G.y), gy(G.z, G.w), eA(E.x, E.y), eB(E.z, E.w);
        axA = fma(gx, eA, axA);
        ayA = fma(gy, eA, ayA);
        axB = fma(gx, eB, axB);
        ayB = fma(gy, eB, ayB);
      };
      if (staged) {
        const float4 *Gs = reinterpret_cast<const float4 *>(stg + TL::IN_STRIDE) + lx;
        const float4 *Es = reinterpret_cast<const float4 *>(stg + ey_off) + ly;
#pragma unroll 4
        for (int r = 0; r < st.nrows; ++r) add(Gs[r * TILE_X], Es[r * (TL::TY / 2)]);
      } else if (flA || flB) {
        // (yA is even: yA and yA + 1 share 16 bytes of the phase table)
        const float4 *Gg = reinterpret_cast<const float4 *>(st.G_cur) + x;
        const float4 *Eg = reinterpret_cast<const float4 *>(st.EY) + yA / 2;
        for (int r = 0; r < st.nrows; ++r) add(Gg[(long long)r * g.nx], Eg[(long long)r * (st.eyp / 2)]);
      }
      Fx += T(axA.v.x + axA.v.y, axB.v.x + axB.v.y);
      Fy += T(ayA.v.x + ayA.v.y, ayB.v.x + ayB.v.y);
    }
    // (lanes without fluid, outside the lattice or solid, pull what the stage holds there and drop it)
    const int b0 = (2 * ly + 1) * TL::TXB + lx + TL::V;
    T h[Q];
    auto pull = [&](auto masked) {
      constexpr bool M = decltype(masked)::value;
#pragma unroll
    for (int q = 0; q < Q; ++q) {
      const S *pl = tile + q * TL::TYB * TL::TXB + b0;
      const S *own = tile + V::opp(q) * TL::TYB * TL::TXB + b0;
      const int sx = sgnx<VS>(q), sy = sgny<VS>(q);
      T acc = T(wts.beta2[q][0]) * T(load_s_raw<S>(pl), load_s_raw<S>(pl + DB));
      if (sx != 0) {
        float vA = load_s_raw<S>(pl - sx), vB = load_s_raw<S>(pl + DB - sx);
        if (M && ((nbA >> (4 - sx)) & 1u)) vA = load_s_raw<S>(own);
        if (M && ((nbB >> (4 - sx)) & 1u)) vB = load_s_raw<S>(own + DB);
        acc = fma(T(wts.beta2[q][1]), T(vA, vB), acc);
      }
      if (sy != 0) {
        float vA = load_s_raw<S>(pl - sy * TL::TXB), vB = load_s_raw<S>(pl + DB - sy * TL::TXB);
        if (M && ((nbA >> (4 - 3 * sy)) & 1u)) vA = load_s_raw<S>(own);
        if (M && ((nbB >> (4 - 3 * sy)) & 1u)) vB = load_s_raw<S>(own + DB);
        acc = fma(T(wts.beta2[q][2]), T(vA, vB), acc);
      }
      if (sx != 0 && sy != 0) {
        float vA = load_s_raw<S>(pl - sy * TL::TXB - sx), vB = load_s_raw<S>(pl + DB - sy * TL::TXB - sx);
        if (M && ((nbA >> (4 - 3 * sy - sx)) & 1u)) vA = load_s_raw<S>(own);
        if (M && ((nbB >> (4 - 3 * sy - sx)) & 1u)) vB = load_s_raw<S>(own + DB);
        acc = fma(T(wts.beta2[q][3]), T(vA, vB), acc);
      }
      h[q] = acc;
    }
    };
    // warps none of whose cells has a solid neighbour skip the substitutions (a third of an open
    // channel's instructions; at 15 % discs a third of the warps)
    if (MASK && __any_sync(0xffffffffu, ((nbA | nbB) & 0x1efu) != 0)) pull(std::true_type());
    else pull(std::false_type());
    if (!release()) return false;
    if (!both) {  // a lane without fluid (outside the lattice or solid) computes the rest state
#pragma unroll
      for (int q = 0; q < Q; ++q) h[q] = T(flA ? h[q].v.x : 0.0f, flB ? h[q].v.y : 0.0f);
    }
    const Mom<T> M = moments_of<T, T, VS, FORCE>(h);
    const Macro<T> m = cell_macro_pair<VS>(h, M, p.vmax2);
    if (!m.ok) atomicOr(err, cell_error(m));
    if (macro_out) {  // the cells' Landau solutions, forces and streamed h, kept for the reverse sweep
      const long long nc = (long long)g.nx * g.ny;
      if (flA) {
        const long long c = (long long)yA * g.nx + x;
        macro_out[c] = m.eps_m1.v.x;
        macro_out[nc + c] = m.vx.v.x;
        macro_out[2 * nc + c] = m.vy.v.x;
        macro_out[3 * nc + c] = Fx.v.x;
        macro_out[4 * nc + c] = Fy.v.x;
#pragma unroll
        for (int q = 0; q < Q; ++q) macro_out[(5 + q) * nc + c] = h[q].v.x;
      }
      if (flB) {
        const long long c = (long long)yB * g.nx + x;
        macro_out[c] = m.eps_m1.v.y;
        macro_out[nc + c] = m.vx.v.y;
        macro_out[2 * nc + c] = m.vy.v.y;
        macro_out[3 * nc + c] = Fx.v.y;
        macro_out[4 * nc + c] = Fy.v.y;
#pragma unroll
        for (int q = 0; q < Q; ++q) macro_out[(5 + q) * nc + c] = h[q].v.y;
      }
    }
    // the output in the stored scale (FP16: 2^8 h)
    constexpr float up = HScale<S>::up;
    const Coll<T> cf = coll_coeffs<T, VS, FORCE>(M, m, T(p.omega0 * up), T(p.fpref * up), Fx, Fy, T(up));
    collide_all<T, VS, FORCE>(cf, h, hn);
  }
  // a lane without fluid stores the rest state (0)
  if (!both) {
#pragma unroll
    for (int q = 0; q < Q; ++q) hn[q] = T(flA ? hn[q].v.x : 0.0f, flB ? hn[q].v.y : 0.0f);
  }
  // round once to the storage type (the ghost images below repeat the same values)
  S sA[Q], sB[Q];
  {
    const bool sr = sizeof(S) == 2 && p.stochastic;
    uint32_t rA = sr ? cell_hash(x, yA + p.y_off, p.step, p.round_key) : 0u;
    uint32_t rB = sr ? cell_hash(x, yB + p.y_off, p.step, p.round_key) : 0u;
    if constexpr (std::is_same<S, __half>::value) {
      if (sr) {
#pragma unroll
        for (int q = 0; q < Q; ++q) {
          rA = next_bits(rA);
          rB = next_bits(rB);
          const uint32_t d = round_pair_f16_sr(hn[q].v.x, hn[q].v.y, rA, rB);
          sA[q] = __ushort_as_half((unsigned short)(d & 0xffffu));
          sB[q] = __ushort_as_half((unsigned short)(d >> 16));
        }
      } else {
#pragma unroll
        for (int q = 0; q < Q; ++q) {
          const uint32_t d = round_pair_f16_rn(hn[q].v.x, hn[q].v.y);
          sA[q] = __ushort_as_half((unsigned short)(d & 0xffffu));
          sB[q] = __ushort_as_half((unsigned short)(d >> 16));
        }
      }
    } else {
#pragma unroll
      for (int q = 0; q < Q; ++q) {
        rA = next_bits(rA);
        rB = next_bits(rB);
        sA[q] = store_round<S>(hn[q].v.x, sr, rA);
        sB[q] = store_round<S>(hn[q].v.y, sr, rB);
      }
    }
  }
  {  // coalesced stores straight from registers (one 128-byte line per warp, row and plane)
    S *oA = fout + (long long)(yA + 1) * g.pitch + x + TL::XOFF;
    S *oB = oA + g.pitch;
    if (inA) {
#pragma unroll
      for (int q = 0; q < Q; ++q) oA[q * g.plane] = sA[q];
    }
    if (inB) {
#pragma unroll
      for (int q = 0; q < Q; ++q) oB[q * g.plane] = sB[q];
    }
  }
  // ghost copies of the periodic neighbours (boundary cells only)
  if (!border) return true;
#pragma unroll
  for (int lane = 0; lane < 2; ++lane) {
    const int y = lane ? yB : yA;
    if (!(lane ? inB : inA)) continue;
    const int gxv = ghost_col(x, g.nx, g.walls);
    const int gyv = ghost_row(y, g.ny, g.walls);
    if (gxv == INT_MIN && gyv == INT_MIN) continue;
    const int px[3] = {gxv, x, gxv}, py[3] = {y, gyv, gyv};
    for (int a = 0; a < 3; ++a) {
      if (px[a] == INT_MIN || py[a] == INT_MIN) continue;
      S *o = fout + (long long)(py[a] + 1) * g.pitch + px[a] + TL::XOFF;
#pragma unroll
      for (int q = 0; q < Q; ++q) o[q * g.plane] = lane ? sB[q] : sA[q];
    }
  }
  return true;
}

// ---------------------------------------------------------------------------
// The fused step (procedure items 2-5 of Sec. "The Standard/Classical LBM", with the
// driving term of Sec. "The Driving Term").  Persistent CTAs walk the tiles of the
// lattice.  Per tile, one 3-D TMA copy stages all Q planes of the tile plus a
// one-cell halo (ghost rows/columns carry the periodic wrap) into shared memory, with
// the tile's stirring rows; NST stages rotate on mbarriers (NST = 2: the next tile is
// in flight while this one is computed; NST = 1: its copy starts after the pull of this one
// and hides behind the arithmetic, and more CTAs fit on an SM: 512^2 FP32 12.0 -> 10.0 us).
// Each thread pull-streams its cell(s) from shared memory (bilinear weights, bounce-back
// substitution from the mask), takes the moments, Landau-matches, relaxes, adds the force
// and stores the Q results with coalesced stores, refreshing the ghost copies of boundary
// cells.
// ---------------------------------------------------------------------------
template <typename S, int VS, bool MASK, bool FORCE, int CPT, int NST, bool STORE>
__global__ void __launch_bounds__(TILE_THREADS)
step_kernel(const __grid_constant__ CUtensorMap tin, const __grid_constant__ CUtensorMap tG,
            const __grid_constant__ CUtensorMap tEY, S *__restrict__ fout,
            const Geometry<typename RealOf<S>::type> g, const Physics<typename RealOf<S>::type> p,
            const Stir<typename RealOf<S>::type> st, int srows_in, int *__restrict__ tile_ctr, unsigned seq,
            unsigned *__restrict__ err, typename RealOf<S>::type *__restrict__ macro_out) {
  using R = typename RealOf<S>::type;
  using TL = Tile<S, VS>;
  constexpr int NT = TILE_THREADS;
  const int wid = blockIdx.x, nworkers = gridDim.x;
  extern __shared__ __align__(128) unsigned char smem_raw[];
  // every TMA box lands on a 128-byte boundary of this aligned base
  unsigned char *smem = smem_raw + ((128u - (smem_u32(smem_raw) & 127u)) & 127u);
  // stirring rows staged with the tile (srows_in > 0) or read from global memory (L2)
  const bool staged = FORCE && srows_in > 0;
  const int srows = staged ? srows_in : 0;
  const int stage_stride = TL::stage(srows), ey_off = TL::IN_STRIDE + TL::g_bytes(srows);
  // barriers, one per stage; then the work item of each stage and the tile's column | row << 16
  uint64_t *bar = reinterpret_cast<uint64_t *>(smem + NST * stage_stride);
  int *item_of = reinterpret_cast<int *>(smem + NST * stage_stride + 32);
  int *tile_xy = item_of + NST;

  const int tid = threadIdx.x;
  const int ntx = (g.nx + TILE_X - 1) / TILE_X, nty = (g.ny + TL::TY - 1) / TL::TY;
  const int ntiles = ntx * nty;
  const float rcp_ntx = 1.0f / (float)ntx;
  const uint32_t stage_bytes = TL::IN_BYTES + srows * (TL::G_ROW + TL::EY_ROW);
  // Work items: the chunks of the next step's stirring table, one per warp, then the tiles.  On
  // small lattices CTAs of their own build the table while the others compute.  (A share of the
  // table for every CTA, in the shadow of its first copy, was longer than the copy and cost about
  // 1 us of every step; chunks behind the tiles made the launch's end 1.5 us longer at 1024^2.)
  const int chunks = (g.nx + stir_chunk<R>() - 1) / stir_chunk<R>();
  const int nprep = FORCE && st.G_next ? st.nrows * chunks : 0;
  const int tile0 = (nprep + NT / 32 - 1) / (NT / 32), nitems = tile0 + ntiles;
  // Items are handed out by a counter of this launch (launches alternate between two; the first
  // CTA clears the other one for the next launch).  Every item is computed the same way by whichever
  // CTA takes it, so the results do not depend on it.  With a CTA for every item its number is
  // the item, without the counter's round trip before the first copy (0.7 us).  (Larger grids
  // started that way were 3 % slower at 4096^2.)
  int *ctr = tile_ctr + (seq & 1u);
  const bool one_each = nitems <= nworkers;
  // When the two buffers are larger than L2, odd steps walk the lattice backwards: what the step before
  // wrote (and read) last is then still in L2 when it is read (and overwritten); one way every time
  // misses on nearly all of it.
  const bool backwards = (p.step & 1u) && 2ll * VSet<VS>::Q * g.plane * (long long)sizeof(S) > BACKWARDS_BYTES;

  if (tid == 0) {
    for (int s = 0; s < NST; ++s) mbar_init(&bar[s], 1);
    fence_mbar_init();
    prefetch_map(&tin);
    if (staged) {
      prefetch_map(&tG);
      prefetch_map(&tEY);
    }
  }
  // A launch chained to the previous step (programmatic dependent launch) may start while
  // that step's grid drains: the state, the stirring tables and the counters it wrote are
  // touched only after it has completed and its writes are visible.
  griddep_wait();
  if (tid == 0 && wid == 0) tile_ctr[(seq + 1u) & 1u] = 0;
  // thread 0: stage s takes item t (only tiles are copied; the barrier of another item, or of
  // none, completes at once: with t past the end this CTA takes nothing further, and the next
  // step's grid, when chained, may be scheduled once every CTA has come this far)
  auto fill = [&](int s, int t) {
    uint64_t *b = &bar[s];
    item_of[s] = t < nitems ? t : -1;
    if (t < tile0 || t >= nitems) {
      mbar_arrive(b);
      if (t >= nitems) griddep_launch_dependents();
      return;
    }
    t -= tile0;
    if (backwards) t = ntiles - 1 - t;
    // row = t / ntx, column = t mod ntx: the float quotient corrected exactly (t < 2^24)
    int row = (int)((float)t * rcp_ntx), col = t - row * ntx;
    while (col < 0) { --row; col += ntx; }
    while (col >= ntx) { ++row; col -= ntx; }
    tile_xy[s] = col | (row << 16);
    const int x0 = col * TILE_X, y0 = row * TL::TY;
    unsigned char *st0 = smem + s * stage_stride;
    mbar_expect_tx(b, stage_bytes);
    tma_load_3d(st0, &tin, b, x0 + TL::XOFF - TL::V, y0, 0);
    if (staged) {
      tma_load_2d(st0 + TL::IN_STRIDE, &tG, b, 4 * x0, 0);
      tma_load_2d(st0 + ey_off, &tEY, b, 2 * y0, 0);
    }
  };
  int pending = 0;  // thread 0: the item the next refill will take (fetched one ahead)
  if (tid == 0) {
    for (int s = 0; s < NST; ++s) fill(s, one_each ? wid + s * nworkers : atomicAdd(ctr, 1));
    pending = one_each ? nitems : atomicAdd(ctr, 1);
  }
  __syncthreads();

  // Every thread waits for the staged tile (bounded); a vote in a barrier makes the whole CTA
  // wind down together if a copy never lands.
  bool alive = true, ok = true;
  if (NST >= 2) {
    ok = mbar_wait_bounded(&bar[0], 0, WAIT_CYCLES);
    if (__syncthreads_or(!ok)) alive = false;
  }
  int k = 0;
  for (; alive; ++k) {
    const int s = k % NST;
    if (NST == 1) ok = mbar_wait_bounded(&bar[0], k & 1, WAIT_CYCLES);
    const int t = item_of[s];
    if (NST >= 2 && t < 0) break;
    // NST = 1: the stage is free, and the next tile's copy starts, once every thread has read its tile
    // (the barrier also carries the vote); all that follows the pull hides that copy
    auto release = [&]() {
      if (NST == 1) {
        if (__syncthreads_or(!ok)) return false;
        if (tid == 0 && t >= 0) {
          fill(0, pending);
          if (!one_each) pending = atomicAdd(ctr, 1);
        }
      }
      return true;
    };
    if (t >= tile0) {
      const int xy = tile_xy[s];
      alive = tile_cells<S, VS, MASK, FORCE, CPT>(smem + s * stage_stride, ey_off, fout, (xy & 0xffff) * TILE_X,
                                                  (xy >> 16) * TL::TY, tid, g, g, p, st, staged, err,
                                                  STORE ? macro_out : static_cast<R *>(nullptr), release);
    } else {
      alive = release();
      if (NST == 1 && t < 0) break;
      const int i = t * (NT / 32) + tid / 32;
      if (FORCE && alive && i < nprep) {
        const int r = i / chunks;
        stir_row_chunk<R>(st.modes, st.step_next, r, i - r * chunks, g.nx, tid & 31, st.G_next + (long long)r * g.nx);
      }
    }
    if (NST >= 2) {
      // the next stage's barrier completes with its tile, or at once when it has none
      const int sn = (k + 1) % NST;
      ok = mbar_wait_bounded(&bar[sn], ((k + 1) / NST) & 1, WAIT_CYCLES);
      if (__syncthreads_or(!ok)) {  // (also the barrier after which stage s is free)
        alive = false;
        break;
      }
      if (tid == 0) {
        fill(s, pending);
        if (!one_each) pending = atomicAdd(ctr, 1);
      }
    }
  }
  if (!alive && tid == 0) {
    // a staged copy did not land in time: latch the error and wait (bounded) once more
    // for this CTA's copies still in flight before returning
    atomicOr(err, ERR_TIMEOUT);
    // fills so far: NST = 1 fails behind the wait for item k - 1 (the last item, of none, has no copy)
    // and refills after it, NST = 2 has refilled at the end of k items
    wind_down(NST == 1 ? k : NST + k, NST, [&](int s, int parity) { mbar_wait_bounded(&bar[s], parity, WAIT_CYCLES); });
  }
}

// ---------------------------------------------------------------------------
// The batched step: one persistent launch advances every lattice of a batch (an
// ensemble of stirred realisations or impurity samples, uneven sizes) by one step.
// The tiles of all members form one list (member m owns tiles tile0[m] .. tile0[m+1]);
// CTAs walk it exactly as the single-lattice kernel walks one lattice (tiles handed out
// by a counter, cleared between launches by the kernel that advances the step), and take
// each tile's member (searched forward from the CTA's previous tile's member), buffers and
// TMA descriptors from the member table; the thread that stages a tile resolves it once
// and leaves what the tile needs in shared memory beside the stage.
// The per-member step is step0 + *bstep, so a captured CUDA graph of launches can
// replay with the counter advanced by a one-thread kernel between launches.  All members
// share the velocity set, storage type, dt/a, eta/s, eps0, the force shell and the
// rounding mode; they differ in size, walls, solids, seeds and initial fields.
// ---------------------------------------------------------------------------
struct BatchDims {
  int nx, ny, pitch, walls;
  long long plane;
  const uint16_t *nbmask;
};

// What the cells of a staged tile need of its member (written by the staging thread).
struct alignas(16) TileInfo {
  BatchDims dims;
  void *fout;          // the buffer this step writes
  unsigned *err;
  long long n;         // the member's step index
  int x0, y0, m;
  unsigned round_key;
};

template <typename R> __device__ __forceinline__ Stir<R> member_stir(const MemberDesc &d, long long n, double amp) {
  Stir<R> s;
  s.nrows = d.nrows; s.eyp = d.eyp;
  s.G_cur = (const R4<R> *)d.G[n & 1];
  s.EY = (const R2<R> *)d.EY;
  s.G_next = (R4<R> *)d.G[(n + 1) & 1];
  s.step_next = n + 1;
  s.modes = StirModes{d.mode_kx, d.row_start, d.tw, d.mode_scale, d.seed, amp};
  return s;
}

template <typename S, int VS, bool MASK, bool FORCE, int CPT, int NST>
__global__ void __launch_bounds__(TILE_THREADS, CPT == 2 ? 4 : 1)  // two-cell paths: 4 CTAs/SM
batch_step_kernel(const BatchTables bt, const Geometry<typename RealOf<S>::type> wts,
                  const Physics<typename RealOf<S>::type> p0, const int srows_in, const double amp,
                  const long long *__restrict__ bstep_ptr) {
  using R = typename RealOf<S>::type;
  using TL = Tile<S, VS>;
  constexpr int NT = TILE_THREADS;
  extern __shared__ __align__(128) unsigned char smem_raw[];
  unsigned char *smem = smem_raw + ((128u - (smem_u32(smem_raw) & 127u)) & 127u);
  const bool staged = FORCE && srows_in > 0;
  const int srows = staged ? srows_in : 0;
  const int stage_stride = TL::stage(srows), ey_off = TL::IN_STRIDE + TL::g_bytes(srows);
  uint64_t *bar = reinterpret_cast<uint64_t *>(smem + NST * stage_stride);
  TileInfo *info = reinterpret_cast<TileInfo *>(smem + NST * stage_stride + 64);
  const uint32_t stage_bytes = TL::IN_BYTES + srows * (TL::G_ROW + TL::EY_ROW);
  const long long bstep = *bstep_ptr;

  const int tid = threadIdx.x, wid = blockIdx.x, nworkers = gridDim.x;
  const int ntiles = bt.tile0[bt.n];
  if (tid == 0) {
    for (int s = 0; s < NST; ++s) mbar_init(&bar[s], 1);
    fence_mbar_init();
  }
  __syncthreads();
  // thread 0: stage s takes tile t of the list (handed out by the launch's counter, so a
  // CTA that runs ahead takes more tiles), or, with t past the end, only completes its
  // barrier; the tile's member is resolved here, once, into the stage's TileInfo.  A CTA's
  // tiles only increase, so the member search starts at the previous tile's member.
  int m_last = 0;
  auto fill = [&](int s, int t) {
    TileInfo &ti = info[s];
    uint64_t *b = &bar[s];
    if (t >= ntiles) {
      ti.m = -1;
      mbar_arrive(b);
      return;
    }
    int m = m_last;
    while (bt.tile0[m + 1] <= t) ++m;  // tile0[n] = ntiles > t ends the search
    m_last = m;
    const MemberDesc &d = bt.mem[m];
    const int lt = t - bt.tile0[m];
    // row = lt / ntx, column = lt mod ntx: the float quotient is within a unit or two of
    // the exact one (lt < 2^24), then corrected exactly
    int row = (int)((float)lt * d.rcp_ntx), col = lt - row * d.ntx;
    while (col < 0) { --row; col += d.ntx; }
    while (col >= d.ntx) { ++row; col -= d.ntx; }
    const int x0 = col * TILE_X, y0 = row * TL::TY;
    const long long n = d.step0 + bstep;
    const int cur = (d.cur0 + (int)(bstep & 1)) & 1;
    ti.dims = BatchDims{d.nx, d.ny, d.pitch, d.walls, d.plane, d.nbmask};
    ti.fout = d.f[cur ^ 1];
    ti.err = d.err;
    ti.n = n;
    ti.x0 = x0;
    ti.y0 = y0;
    ti.m = m;
    ti.round_key = d.round_key;
    unsigned char *st0 = smem + s * stage_stride;
    mbar_expect_tx(b, stage_bytes);
    tma_load_3d(st0, &d.tin[cur], b, x0 + TL::XOFF - TL::V, y0, 0);
    if (staged) {
      tma_load_2d(st0 + TL::IN_STRIDE, &d.tG[n & 1], b, 4 * x0, 0);
      tma_load_2d(st0 + ey_off, &d.tEY, b, 2 * y0, 0);
    }
  };
  int pending = 0;  // thread 0: the tile the next refill will stage (fetched one tile ahead)
  if (tid == 0) {
    for (int s = 0; s < NST; ++s) fill(s, atomicAdd(bt.tile_ctr, 1));
    pending = atomicAdd(bt.tile_ctr, 1);
  }
  bool alive = true, ok = true;
  if (NST >= 2) {
    ok = mbar_wait_bounded(&bar[0], 0, WAIT_CYCLES);
    if (__syncthreads_or(!ok)) alive = false;
  }
  int k = 0;
  for (; alive; ++k) {
    const int s = k % NST;
    if (NST == 1) ok = mbar_wait_bounded(&bar[0], k & 1, WAIT_CYCLES);
    const TileInfo ti = info[s];
    auto release = [&]() {  // (as in step_kernel)
      if (NST == 1) {
        if (__syncthreads_or(!ok)) return false;
        if (tid == 0 && ti.m >= 0) {
          fill(0, pending);
          pending = atomicAdd(bt.tile_ctr, 1);
        }
      }
      return true;
    };
    if (ti.m < 0) {
      if (NST == 1) alive = release();
      break;
    }
    Physics<R> p = p0;
    p.round_key = ti.round_key;
    p.step = (unsigned)(ti.n & 0xffffffffll);
    // staged stirring rows need only their count (the shell is shared by all members)
    Stir<R> st{};
    if (FORCE && staged) st.nrows = srows;
    else if (FORCE) st = member_stir<R>(bt.mem[ti.m], ti.n, amp);
    alive = tile_cells<S, VS, MASK, FORCE, CPT>(smem + s * stage_stride, ey_off, (S *)ti.fout, ti.x0, ti.y0, tid, ti.dims,
                                                wts, p, st, staged, ti.err, static_cast<R *>(nullptr), release);
    if (NST >= 2) {
      // the next stage's barrier completes with its tile, or at once when it has none
      const int sn = (k + 1) % NST;
      ok = mbar_wait_bounded(&bar[sn], ((k + 1) / NST) & 1, WAIT_CYCLES);
      if (__syncthreads_or(!ok)) {  // (also the barrier after which stage s is free)
        alive = false;
        break;
      }
      if (tid == 0) {
        fill(s, pending);
        pending = atomicAdd(bt.tile_ctr, 1);
      }
    }
  }
  if (!alive && tid == 0) {
    atomicOr(bt.mem[0].err, ERR_TIMEOUT);
    // (as in step_kernel)
    wind_down(NST == 1 ? k : NST + k, NST, [&](int s, int parity) { mbar_wait_bounded(&bar[s], parity, WAIT_CYCLES); });
  }
  if (!alive) return;  // copies may still be in flight: stage 0 is not free
  // The stirring tables of the next step, after the tiles: chunks of rows, members in order, one
  // per warp.
  if (FORCE && bt.mem[0].nrows) {
    const int total = bt.prep0[bt.n], warps = nworkers * (NT / 32);
    int m = 0;
    for (int e = wid * (NT / 32) + tid / 32; e < total; e += warps) {
      while (bt.prep0[m + 1] <= e) ++m;  // prep0[n] = total > e ends the search
      const MemberDesc &d = bt.mem[m];
      const Stir<R> st = member_stir<R>(d, d.step0 + bstep, amp);
      const int chunks = (d.nx + stir_chunk<R>() - 1) / stir_chunk<R>();
      const int i = e - bt.prep0[m], r = i / chunks;
      stir_row_chunk<R>(st.modes, st.step_next, r, i - r * chunks, d.nx, tid & 31, st.G_next + (long long)r * d.nx);
    }
  }
}

// ---------------------------------------------------------------------------
// Observation of the current state f_n = stream(f*_n) (procedure item 3) straight from
// global memory (ghost-padded planes), in one of three forms:
//   OBS_FIELDS  eps, u^x, u^y per cell (each pointer may be NULL) and the totals T^00, T^0x,
//               T^0y, 1/2 |v|^2 in `totals`;
//   OBS_V       z = v_x + i v_y per cell, the input of the spectrum's transform;
//   OBS_COLS    the column means of v in totals[0 .. nx) (x) and totals[nx .. 2 nx) (y).
// FP64 storage matches and sums in FP64; the others (FP32 state) match in FP32, as the step
// kernel does, on packed pairs of cells (x, y), (x, y + 1).
//
// What bounds it: DRAM at large sizes (17 planes read, 24 bytes of fields written per cell),
// so no other pipe may come near that: GB300 runs FP64 and the FP32 -> FP64 conversions at
// 1/64 of FP32's rate, and the former kernel's five FP64-pipe operations per cell alone took
// as long as the memory.  The values are widened with integer operations instead (exact),
// one FP64 addition per cell is left (eps = eps0 (1 + e)), and the totals and column sums of
// FP32 states are carried in pairs of FP32 numbers (48 bits), FP64 from the block's sum on.
// The last block to finish adds the blocks' partial sums in a fixed order; a second launch
// with one serial block took 12-130 us for that.
// ---------------------------------------------------------------------------
constexpr int OBS_FIELDS = 0, OBS_V = 1, OBS_COLS = 2;
// cells of a thread (rows y, y + 1) and rows of an observation tile (32 columns; 8 thread rows)
template <typename S> constexpr int obs_cells() { return sizeof(S) == 8 ? 1 : 2; }
template <typename S> constexpr int obs_rows() { return 8 * obs_cells<S>(); }

// FP32 to FP64 by moving the fields of the IEEE formats (exact); zeros, subnormals,
// infinities and NaN take the conversion instruction.
__device__ __forceinline__ double widen(float f) {
  const uint32_t u = __float_as_uint(f), a = u & 0x7fffffffu;
  if (a < 0x00800000u || a >= 0x7f800000u) return (double)f;
  return __hiloint2double((int)((u & 0x80000000u) | ((a >> 3) + 0x38000000u)), (int)(u << 29));
}
__device__ __forceinline__ double widen(double f) { return f; }

template <typename S, typename R, int VS, bool MASK>
__device__ __forceinline__ void pull_global(const S *__restrict__ fin, const Geometry<R> &g, int x, int y,
                                            unsigned nb, R h[VSet<VS>::Q]) {
  constexpr int Q = VSet<VS>::Q;
  const long long o = (long long)(y + 1) * g.pitch + x + PadLayout<S>::XOFF;
#pragma unroll
  for (int q = 0; q < Q; ++q) {
    const S *pl = fin + q * g.plane + o;
    const int sx = sgnx<VS>(q), sy = sgny<VS>(q);
    R acc = g.beta[q][0] * load_h<S, R>(pl);
    const R own = MASK ? load_h<S, R>(fin + VSet<VS>::opp(q) * g.plane + o) : R(0);
    if (sx != 0) acc += g.beta[q][1] * ((MASK && ((nb >> (4 - sx)) & 1u)) ? own : load_h<S, R>(pl - sx));
    if (sy != 0) acc += g.beta[q][2] * ((MASK && ((nb >> (4 - 3 * sy)) & 1u)) ? own : load_h<S, R>(pl - (long long)sy * g.pitch));
    if (sx != 0 && sy != 0)
      acc += g.beta[q][3] * ((MASK && ((nb >> (4 - 3 * sy - sx)) & 1u)) ? own : load_h<S, R>(pl - (long long)sy * g.pitch - sx));
    h[q] = acc;
  }
}

// The pulls of the cells (x, y) and (x, y + 1) as a pair (lanes without fluid are not pulled).
template <typename S, int VS, bool MASK>
__device__ __forceinline__ void pull_global_pair(const S *__restrict__ fin, const Geometry<float> &g, int x, int y,
                                                 unsigned nbA, unsigned nbB, bool flA, bool flB, F2 h[VSet<VS>::Q]) {
  float a[VSet<VS>::Q], b[VSet<VS>::Q];
#pragma unroll
  for (int q = 0; q < VSet<VS>::Q; ++q) a[q] = b[q] = 0.0f;
  if (flA) pull_global<S, float, VS, MASK>(fin, g, x, y, nbA, a);
  if (flB) pull_global<S, float, VS, MASK>(fin, g, x, y + 1, nbB, b);
#pragma unroll
  for (int q = 0; q < VSet<VS>::Q; ++q) h[q] = F2(a[q], b[q]);
}

struct ObsOut {
  double *eps, *ux, *uy;  // OBS_FIELDS (each may be NULL)
  double2 *z;             // OBS_V (FP32 states: float4 of the high and low parts of v_x, v_y, times zscale);
                          // OBS_COLS: the blocks' partial column sums (the same two forms)
  double *partials;       // [blocks][4]
  double *totals;         // [4]; OBS_COLS: [2 nx]
  unsigned *sync;         // zeroed counters of finished blocks: 1, or one per tile column (OBS_COLS)
  double *bins;           // OBS_V: nbins values cleared for the spectrum's sums
  int nbins;
  float zscale;           // OBS_V, FP32 states: the factor of z
};

// v = u / u^0 = u / sqrt(1 + u^2) of two cells in pairs: the root from the FP32 approximation by one Newton
// step, its residual 1 - s y^2 in two-float arithmetic.
__device__ __forceinline__ void over_u0(F2 ux, F2 uy, DF2 &vx, DF2 &vy) {
  const F2 xx = ux * ux, yy = uy * uy;
  const DF2 s = df_add(df_add(DF2{xx, fma(ux, ux, -xx)}, DF2{yy, fma(uy, uy, -yy)}), F2(1.0f));
  const F2 y = FM<F2>::rsqrt(s.h), t = y * y, tl = fma(y, y, -t);
  const F2 r = fma(s.h, t, F2(-1.0f)) + fma(s.h, tl, s.l * t);  // s y^2 - 1
  const F2 c = F2(-0.5f) * y * r;
  const F2 hx = ux * y, hy = uy * y;
  vx = df_norm(hx, fma(ux, c, fma(ux, y, -hx)));
  vy = df_norm(hy, fma(uy, c, fma(uy, y, -hy)));
}

template <typename S, int VS, bool MASK, int MODE>
__global__ void __launch_bounds__(256)
observe_kernel(const S *__restrict__ fin, const Geometry<typename RealOf<S>::type> g, double eps0, float vmax2,
               const ObsOut out, unsigned *__restrict__ err) {
  using R = typename RealOf<S>::type;
  constexpr int Q = VSet<VS>::Q;
  constexpr bool F64 = sizeof(R) == 8;
  constexpr int NC = obs_cells<S>(), OBS_ROWS = obs_rows<S>();
  const int lx = threadIdx.x, ly = threadIdx.y, tid = ly * 32 + lx;
  const int ntx = (g.nx + 31) / 32, nty = (g.ny + OBS_ROWS - 1) / OBS_ROWS, ntiles = ntx * nty;
  __shared__ double redd[8][4];
  __shared__ float4 redf[8][4];         // FP32 state: the warps' sums (high x, y, low x, y) of the four terms
  __shared__ double2 cols[8][32];
  __shared__ int cnt[8];
  __shared__ bool last;
  if (MODE == OBS_V && blockIdx.x == 0)
    for (int i = tid; i < out.nbins; i += 256) out.bins[i] = 0.0;
  double acc[4] = {0.0, 0.0, 0.0, 0.0};
  const DF2 zero{F2(0.0f), F2(0.0f)};
  DF2 accf[4] = {zero, zero, zero, zero};
  int fluid = 0;
  for (int t = blockIdx.x; t < ntiles; t += gridDim.x) {
    const int tx = t % ntx, ty = t / ntx;
    const int x = tx * 32 + lx, y = ty * OBS_ROWS + NC * ly;
    unsigned nb[NC];
    bool in[NC], fl[NC];
#pragma unroll
    for (int k = 0; k < NC; ++k) {
      in[k] = x < g.nx && y + k < g.ny;
      nb[k] = 0u;
      if (MASK && in[k]) nb[k] = g.nbmask[(long long)(y + k) * g.nx + x];
      fl[k] = in[k] && !(MASK && (nb[k] & 16u));
    }
    R e[NC], ux[NC], uy[NC], vx[NC], vy[NC];
    float wx[NC], wy[NC];  // FP32 state: the low parts of v
#pragma unroll
    for (int k = 0; k < NC; ++k) {
      e[k] = ux[k] = uy[k] = vx[k] = vy[k] = R(0);
      wx[k] = wy[k] = 0.0f;
    }
    if constexpr (F64) {
#pragma unroll
      for (int k = 0; k < NC; ++k) {
        if (!fl[k]) continue;
        R h[Q];
        pull_global<S, R, VS, MASK>(fin, g, x, y + k, nb[k], h);
        const Mom<double> M = moments_of<double, R, VS, false>(h);
        const Macro<double> m = macro_from<double, VS>(M, 40, 1e-12);
        if (!m.ok) atomicOr(err, cell_error(m));
        e[k] = m.eps_m1; ux[k] = m.ux; uy[k] = m.uy; vx[k] = m.vx; vy[k] = m.vy;
        if (MODE == OBS_FIELDS) {
          acc[0] += eps0 * (1.0 + M.e);
          acc[1] += eps0 * M.mx;
          acc[2] += eps0 * M.my;
          acc[3] += 0.5 * (m.vx * m.vx + m.vy * m.vy);
        }
      }
    } else {
      if (fl[0] || fl[1]) {
        F2 h[Q];
        pull_global_pair<S, VS, MASK>(fin, g, x, y, nb[0], nb[1], fl[0], fl[1], h);
        const Mom<F2> M = moments_of<F2, F2, VS, false>(h);
        const Macro<F2> m = cell_macro_pair<VS>(h, M, vmax2);  // (a lane without fluid matches the rest state)
        if (!m.ok) atomicOr(err, cell_error(m));
        e[0] = m.eps_m1.v.x; e[1] = m.eps_m1.v.y;
        ux[0] = m.ux.v.x; ux[1] = m.ux.v.y; uy[0] = m.uy.v.x; uy[1] = m.uy.v.y;
        if (MODE != OBS_FIELDS) {
          // v of the fields u that OBS_FIELDS hands out, to 45 bits: the v that Landau matching ends with lies
          // up to 3e-8 |v| to one side (its last step is not iterated), which a mean over cells keeps
          DF2 px, py;
          over_u0(m.ux, m.uy, px, py);
          vx[0] = px.h.v.x; vx[1] = px.h.v.y; vy[0] = py.h.v.x; vy[1] = py.h.v.y;
          wx[0] = px.l.v.x; wx[1] = px.l.v.y; wy[0] = py.l.v.x; wy[1] = py.l.v.y;
        }
        if (MODE == OBS_FIELDS) {
          // the deviations e, m_x, m_y (order u) beside the exact count of fluid cells
          // (T^00 = eps0 (1 + e))
          fluid += (fl[0] ? 1 : 0) + (fl[1] ? 1 : 0);
          accf[0] = df_add(accf[0], M.e);
          accf[1] = df_add(accf[1], M.mx);
          accf[2] = df_add(accf[2], M.my);
          accf[3] = df_add(accf[3], F2(0.5f) * fma(m.vx, m.vx, m.vy * m.vy));
        }
      }
    }
    if (MODE == OBS_COLS) {
      // column sums of the tile's rows, then (the last block of this tile column) of the row blocks
      if constexpr (F64) {
        cols[ly][lx] = make_double2(vx[0], vy[0]);
        __syncthreads();
        if (ly == 0 && x < g.nx) {
          double2 a = cols[0][lx];
          for (int j = 1; j < 8; ++j) { a.x += cols[j][lx].x; a.y += cols[j][lx].y; }
          out.z[(long long)ty * g.nx + x] = a;
        }
      } else {
        float4 *cf = reinterpret_cast<float4 *>(&cols[0][0]), *zf = reinterpret_cast<float4 *>(out.z);
        DF2 a = df_add(DF2{F2(vx[0], vy[0]), F2(wx[0], wy[0])}, DF2{F2(vx[NC - 1], vy[NC - 1]), F2(wx[NC - 1], wy[NC - 1])});
        cf[ly * 32 + lx] = make_float4(a.h.v.x, a.h.v.y, a.l.v.x, a.l.v.y);
        __syncthreads();
        if (ly == 0 && x < g.nx) {
          for (int j = 1; j < 8; ++j) {
            const float4 v = cf[j * 32 + lx];
            a = df_add(a, DF2{F2(v.x, v.y), F2(v.z, v.w)});
          }
          zf[(long long)ty * g.nx + x] = make_float4(a.h.v.x, a.h.v.y, a.l.v.x, a.l.v.y);
        }
      }
      __threadfence();
      __syncthreads();
      if (tid == 0) last = atomicInc(out.sync + tx, nty - 1) == (unsigned)(nty - 1);
      __syncthreads();
      if (last) {
        __threadfence();
        double2 a = make_double2(0.0, 0.0);
        if constexpr (F64) {
          if (x < g.nx)
            for (int j = ly; j < nty; j += 8) {
              const double2 v = __ldcg(&out.z[(long long)j * g.nx + x]);
              a.x += v.x;
              a.y += v.y;
            }
          cols[ly][lx] = a;
          __syncthreads();
          if (ly == 0)
            for (int j = 1; j < 8; ++j) { a.x += cols[j][lx].x; a.y += cols[j][lx].y; }
        } else {
          float4 *cf = reinterpret_cast<float4 *>(&cols[0][0]);
          const float4 *zf = reinterpret_cast<const float4 *>(out.z);
          DF2 d = zero;
          if (x < g.nx)
            for (int j = ly; j < nty; j += 8) {
              const float4 v = __ldcg(&zf[(long long)j * g.nx + x]);
              d = df_add(d, DF2{F2(v.x, v.y), F2(v.z, v.w)});
            }
          cf[ly * 32 + lx] = make_float4(d.h.v.x, d.h.v.y, d.l.v.x, d.l.v.y);
          __syncthreads();
          if (ly == 0) {
            for (int j = 1; j < 8; ++j) {
              const float4 v = cf[j * 32 + lx];
              d = df_add(d, DF2{F2(v.x, v.y), F2(v.z, v.w)});
            }
            a = make_double2(widen(d.h.v.x) + widen(d.l.v.x), widen(d.h.v.y) + widen(d.l.v.y));
          }
        }
        if (ly == 0 && x < g.nx) {
          out.totals[x] = a.x / g.ny;
          out.totals[g.nx + x] = a.y / g.ny;
        }
      }
      __syncthreads();
      continue;
    }
#pragma unroll
    for (int k = 0; k < NC; ++k) {
      if (!in[k]) continue;
      const long long c = (long long)(y + k) * g.nx + x;
      if (MODE == OBS_FIELDS) {
        if (out.eps) {
          double v = 1.0 + widen(e[k]);
          if (eps0 != 1.0) v *= eps0;
          out.eps[c] = fl[k] ? v : 0.0;
        }
        if (out.ux) out.ux[c] = widen(ux[k]);  // (0 at solid cells)
        if (out.uy) out.uy[c] = widen(uy[k]);
      } else if constexpr (F64) {
        out.z[c] = make_double2(vx[k], vy[k]);
      } else {
        const float s = out.zscale;
        reinterpret_cast<float4 *>(out.z)[c] = make_float4(s * vx[k], s * vy[k], s * wx[k], s * wy[k]);
      }
    }
  }
  if (MODE != OBS_FIELDS) return;
  // this block's partial sums, then (the last block) those of all blocks in a fixed order
  __syncthreads();
  if constexpr (F64) {
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      double v = acc[k];
      for (int off = 16; off > 0; off >>= 1) v += __shfl_down_sync(0xffffffffu, v, off);
      if (lx == 0) redd[ly][k] = v;
    }
    __syncthreads();
    if (tid < 4) {
      double v = 0.0;
      for (int w = 0; w < 8; ++w) v += redd[w][tid];
      out.partials[(long long)blockIdx.x * 4 + tid] = v;
    }
  } else {
#pragma unroll
    for (int k = 0; k < 4; ++k) {
#pragma unroll
      for (int off = 16; off > 0; off >>= 1) accf[k] = df_add(accf[k], df_shfl_xor(accf[k], off));
      if (lx == 0) redf[ly][k] = make_float4(accf[k].h.v.x, accf[k].h.v.y, accf[k].l.v.x, accf[k].l.v.y);
    }
    for (int off = 16; off > 0; off >>= 1) fluid += __shfl_down_sync(0xffffffffu, fluid, off);
    if (lx == 0) cnt[ly] = fluid;
    __syncthreads();
    if (ly == 0) {  // lane: term lx & 3 of warp lx >> 2
      const float4 f = redf[lx >> 2][lx & 3];
      double v = (widen(f.x) + widen(f.y)) + (widen(f.z) + widen(f.w));
      for (int off = 16; off >= 4; off >>= 1) v += __shfl_down_sync(0xffffffffu, v, off);  // lanes of a term are 4 apart
      if (lx == 0) {
        int n = 0;
        for (int w = 0; w < 8; ++w) n += cnt[w];
        v += (double)n;
      }
      if (lx < 4) out.partials[(long long)blockIdx.x * 4 + lx] = lx == 3 ? v : eps0 * v;
    }
  }
  __threadfence();
  __syncthreads();
  if (tid == 0) last = atomicInc(out.sync, gridDim.x - 1) == gridDim.x - 1;
  __syncthreads();
  if (!last) return;
  __threadfence();
  {  // term tid & 3; blocks tid >> 2, + 64, ...
    double v = 0.0;
    for (int i = tid >> 2; i < (int)gridDim.x; i += 64) v += __ldcg(&out.partials[(long long)i * 4 + (tid & 3)]);
    for (int off = 16; off >= 4; off >>= 1) v += __shfl_down_sync(0xffffffffu, v, off);
    if (lx < 4) redd[ly][lx] = v;
    __syncthreads();
    if (tid < 4) {
      double w = 0.0;
      for (int j = 0; j < 8; ++j) w += redd[j][tid];
      out.totals[tid] = w;
    }
  }
}

// ---------------------------------------------------------------------------
// Initial state f*_0 = f_eq(eps, u) (procedure item 1); NULL fields mean eps0 at rest.
// Writes the interior; ghost copies come from fill_ghosts.
// ---------------------------------------------------------------------------
template <typename S, int VS>
__global__ void init_kernel(S *__restrict__ fout, const Geometry<typename RealOf<S>::type> g, double eps0,
                            const double *__restrict__ eps, const double *__restrict__ ux,
                            const double *__restrict__ uy) {
  using V = VSet<VS>;
  const int x = blockIdx.x * blockDim.x + threadIdx.x;
  const int y = blockIdx.y * blockDim.y + threadIdx.y;
  if (x >= g.nx || y >= g.ny) return;
  const long long c = (long long)y * g.nx + x;
  const double e = eps ? eps[c] / eps0 : 1.0;
  const double ax = ux ? ux[c] : 0.0, ay = uy ? uy[c] : 0.0;
  const double u2 = ax * ax + ay * ay, u0 = sqrt(1.0 + u2);
  const bool solid = g.nbmask && (g.nbmask[c] & 16u);
  const long long o = (long long)(y + 1) * g.pitch + x + PadLayout<S>::XOFF;
#pragma unroll
  for (int q = 0; q < V::Q; ++q) {
    const double uv = ax * V::vx(q) + ay * V::vy(q);
    const double heq = (e - 1.0) + V::CA * e * u0 * uv + V::CB * e * uv * uv - V::CC * e * u2;
    fout[q * g.plane + o] = store_h<S, typename RealOf<S>::type>((typename RealOf<S>::type)(solid ? 0.0 : heq));
  }
}

// Ghost columns (x = -1, nx) and, for periodic y, ghost rows (y = -1, ny) and corners:
// copies of the wrapped interior.  With walls the ghost rows stay zero.
template <typename S, int VS>
__global__ void fill_ghosts_kernel(S *__restrict__ f, const Geometry<typename RealOf<S>::type> g) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  const int q = blockIdx.y;
  const int nper = 2 * (g.ny + 2) + 2 * g.nx;
  if (i >= nper) return;
  int gx, gy;  // ghost coordinate in cell units (-1 .. nx, -1 .. ny)
  if (i < 2 * (g.ny + 2)) { gx = (i & 1) ? g.nx : -1; gy = i / 2 - 1; }
  else { const int j = i - 2 * (g.ny + 2); gx = j / 2; gy = (j & 1) ? g.ny : -1; }
  S *pl = f + q * g.plane;
  const long long dst = (long long)(gy + 1) * g.pitch + gx + PadLayout<S>::XOFF;
  const bool yghost = gy < 0 || gy >= g.ny;
  if (yghost && (g.walls & STRIP_Y)) return;  // a strip's ghost rows come from the halo exchange
  if (yghost && (g.walls & WALLS_Y)) { pl[dst] = store_h<S, typename RealOf<S>::type>(0); return; }
  const int sx = (gx + g.nx) % g.nx, sy = (gy + g.ny) % g.ny;
  pl[dst] = pl[(long long)(sy + 1) * g.pitch + sx + PadLayout<S>::XOFF];
}

// Open channel (walls bit OPEN_X): the column left of x = 0 holds the inflow equilibrium
// (eps0, u^x = ux_in; written here once and never by the step kernel) and the column right
// of x = nx - 1 repeats that column (zero-gradient outflow; the step kernel keeps it up).
// Rows of bounce-back walls stay zero.  One thread per padded row, one grid row per plane.
template <typename S, int VS>
__global__ void open_ghosts_kernel(S *__restrict__ f, const Geometry<typename RealOf<S>::type> g, double ux_in) {
  using V = VSet<VS>;
  using R = typename RealOf<S>::type;
  const int row = blockIdx.x * blockDim.x + threadIdx.x;  // padded row 0 .. ny + 1
  const int q = blockIdx.y;
  if (row >= g.ny + 2) return;
  S *pl = f + q * g.plane + (long long)row * g.pitch + PadLayout<S>::XOFF;
  pl[g.nx] = pl[g.nx - 1];
  const bool wall_row = (g.walls & WALLS_Y) && (row == 0 || row == g.ny + 1);
  const double u0 = sqrt(1.0 + ux_in * ux_in), uv = ux_in * V::vx(q);
  const double heq = V::CA * u0 * uv + V::CB * uv * uv - V::CC * ux_in * ux_in;  // eps / eps0 = 1
  pl[-1] = store_h<S, R>((R)(wall_row ? 0.0 : heq));
}

// The stirring tables of steps n .. n + count - 1, one after the other at G (one warp per chunk of a
// row, as the step launches build the next step's).
template <typename R>
__global__ void stir_tables_kernel(const StirModes sm, R4<R> *G, long long table, int nrows, int nx, long long n, int count) {
  const int chunks = (nx + stir_chunk<R>() - 1) / stir_chunk<R>();
  const long long i = (long long)blockIdx.x * (blockDim.x / 32) + threadIdx.x / 32;
  if (i >= (long long)count * nrows * chunks) return;
  const int j = (int)(i / (nrows * chunks)), r = (int)(i / chunks) % nrows, chunk = (int)(i % chunks);
  stir_row_chunk<R>(sm, n + j, r, chunk, nx, threadIdx.x & 31, G + j * table + (long long)r * nx);
}

// ---------------------------------------------------------------------------
// Host launchers for this storage type
// ---------------------------------------------------------------------------
// beta2, the pull weights of the paired kernels, carries 1 / HScale<S>::up: those kernels
// convert the stored values without the scale.
template <typename S> static Geometry<typename RealOf<S>::type> to_geom(const HostGeom &h) {
  using R = typename RealOf<S>::type;
  Geometry<R> g;
  g.nx = h.nx; g.ny = h.ny; g.pitch = h.pitch; g.plane = h.plane; g.walls = h.walls; g.nbmask = h.nbmask;
  for (int q = 0; q < 17; ++q)
    for (int k = 0; k < 4; ++k) {
      g.beta[q][k] = (R)h.beta[q][k];
      const float b = (float)h.beta[q][k] * HScale<S>::down;
      g.beta2[q][k] = make_float2(b, b);
    }
  return g;
}

static StirModes to_modes(const HostStir &h) {
  return StirModes{h.mode_kx, h.row_start, h.tw, h.mode_scale, h.seed, h.amp};
}

template <typename R> static Stir<R> to_stir(const HostStir &h) {
  Stir<R> s;
  s.nrows = h.nrows;
  s.G_cur = (const R4<R> *)h.G_cur; s.EY = (const R2<R> *)h.EY; s.G_next = (R4<R> *)h.G_next;
  s.eyp = h.eyp;
  s.step_next = h.step_next;
  s.modes = to_modes(h);
  return s;
}

// STORE: the variant that also keeps each fluid cell's Landau solution, force and streamed
// deviations h (5 + Q planes of nx * ny values; the gradient's recomputation); the regular
// kernel is compiled without that store.
template <typename S, int VS, bool MASK, bool FORCE, int NST, bool STORE>
static cudaError_t launch_step_k(const CUtensorMap &tin, const CUtensorMap &tG, const CUtensorMap &tEY, void *fout,
                                 const Geometry<typename RealOf<S>::type> &g, const Physics<typename RealOf<S>::type> &p,
                                 const Stir<typename RealOf<S>::type> &s, unsigned *err, int grid_limit,
                                 int stir_rows, int *tile_ctr, unsigned seq, bool chained, void *macro_out,
                                 cudaStream_t stream) {
  using TL = Tile<S, VS>;
  using R = typename RealOf<S>::type;
  constexpr int CPT = sizeof(S) == 8 ? 1 : 2;
  constexpr int NT = TILE_THREADS;
  auto kern = step_kernel<S, VS, MASK, FORCE, CPT, NST, STORE>;
  const int srows = (FORCE && s.nrows > 0 && s.nrows <= TL::MAX_SROWS && stir_rows != 2) ? s.nrows : 0;
  const int smem = TL::smem(NST, srows);
  static int configured_dev = -1, configured_smem = -1, max_blocks = 0, sms = 0;
  int dev = 0;
  cudaGetDevice(&dev);
  if (configured_dev != dev || configured_smem != smem) {
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
    if (e != cudaSuccess) return e;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&max_blocks, kern, NT, smem);
    if (e != cudaSuccess) return e;
    e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    configured_dev = dev;
    configured_smem = smem;
  }
  int items = ((g.nx + TILE_X - 1) / TILE_X) * ((g.ny + TL::TY - 1) / TL::TY);
  if (FORCE && s.G_next) items += (s.nrows * ((g.nx + stir_chunk<R>() - 1) / stir_chunk<R>()) + NT / 32 - 1) / (NT / 32);
  int workers = max_blocks * sms;
  if (grid_limit > 0 && grid_limit < workers) workers = grid_limit;
  if (workers > items) workers = items;
  if (workers < 1) workers = 1;
  if (chained) {
    // a step right after the previous one on the same stream: programmatic dependent
    // launch lets its CTAs be scheduled while that step's last tiles finish
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(workers);
    cfg.blockDim = dim3(NT);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kern, tin, tG, tEY, (S *)fout, g, p, s, srows, tile_ctr, seq, err,
                              static_cast<R *>(macro_out));
  }
  kern<<<workers, NT, smem, stream>>>(tin, tG, tEY, (S *)fout, g, p, s, srows, tile_ctr, seq, err,
                                      static_cast<R *>(macro_out));
  return cudaGetLastError();
}

template <typename S, int VS, bool MASK, bool FORCE, int NST>
static cudaError_t launch_step_v(const CUtensorMap &tin, const CUtensorMap &tG, const CUtensorMap &tEY, void *fout,
                                 const Geometry<typename RealOf<S>::type> &g, const Physics<typename RealOf<S>::type> &p,
                                 const Stir<typename RealOf<S>::type> &s, unsigned *err, int grid_limit,
                                 int stir_rows, int *tile_ctr, unsigned seq, bool chained, void *macro_out,
                                 cudaStream_t stream) {
  if constexpr (sizeof(S) >= 4) {  // the gradient runs on FP32 and FP64 states only
    if (macro_out)
      return launch_step_k<S, VS, MASK, FORCE, NST, true>(tin, tG, tEY, fout, g, p, s, err, grid_limit, stir_rows,
                                                           tile_ctr, seq, chained, macro_out, stream);
  }
  return launch_step_k<S, VS, MASK, FORCE, NST, false>(tin, tG, tEY, fout, g, p, s, err, grid_limit, stir_rows,
                                                        tile_ctr, seq, chained, nullptr, stream);
}

template <typename S, int NST>
static cudaError_t launch_step_n(int vset, const CUtensorMap &mi, const CUtensorMap &mg, const CUtensorMap &me,
                                 void *fout, const Geometry<typename RealOf<S>::type> &g,
                                 const Physics<typename RealOf<S>::type> &p, const Stir<typename RealOf<S>::type> &s,
                                 bool mask, bool force, unsigned *err, int grid_limit, int stir_rows,
                                 int *ctr, unsigned seq, bool chained, void *macro_out, cudaStream_t stream) {
  if (vset == 3) {
    if (force) {
      if (mask) return launch_step_v<S, 3, true, true, NST>(mi, mg, me, fout, g, p, s, err, grid_limit, stir_rows, ctr, seq, chained, macro_out, stream);
      return launch_step_v<S, 3, false, true, NST>(mi, mg, me, fout, g, p, s, err, grid_limit, stir_rows, ctr, seq, chained, macro_out, stream);
    }
    if (mask) return launch_step_v<S, 3, true, false, NST>(mi, mg, me, fout, g, p, s, err, grid_limit, stir_rows, ctr, seq, chained, macro_out, stream);
    return launch_step_v<S, 3, false, false, NST>(mi, mg, me, fout, g, p, s, err, grid_limit, stir_rows, ctr, seq, chained, macro_out, stream);
  }
  if (mask) return launch_step_v<S, 2, true, false, NST>(mi, mg, me, fout, g, p, s, err, grid_limit, stir_rows, ctr, seq, chained, macro_out, stream);
  return launch_step_v<S, 2, false, false, NST>(mi, mg, me, fout, g, p, s, err, grid_limit, stir_rows, ctr, seq, chained, macro_out, stream);
}

template <typename S>
static cudaError_t launch_step_t(int vset, const void *tin, const void *tg, const void *tey, void *fout,
                                 const HostGeom &hg, const HostPhys &hp, const HostStir &hs, unsigned *err,
                                 int grid_limit, int stages, int stir_rows, int *ctr, unsigned seq,
                                 bool chained, void *macro_out, cudaStream_t stream) {
  using R = typename RealOf<S>::type;
  const Geometry<R> g = to_geom<S>(hg);
  Physics<R> p;
  p.omega0 = (R)hp.omega0; p.fpref = (R)hp.fpref; p.body_x = (R)hp.body_x; p.body_y = (R)hp.body_y;
  p.vmax2 = (R)hp.vmax2;
  p.stochastic = hp.stochastic;
  p.round_key = hp.round_key;
  p.step = (unsigned)(hp.step & 0xffffffffll);
  p.y_off = hp.y_off;
  const Stir<R> s = to_stir<R>(hs);
  const CUtensorMap &mi = *(const CUtensorMap *)tin, &mg = *(const CUtensorMap *)tg, &me = *(const CUtensorMap *)tey;
  const bool mask = hg.nbmask != nullptr, force = hp.has_force != 0;
  if (stages == 1)
    return launch_step_n<S, 1>(vset, mi, mg, me, fout, g, p, s, mask, force, err, grid_limit, stir_rows, ctr, seq, chained, macro_out, stream);
  return launch_step_n<S, 2>(vset, mi, mg, me, fout, g, p, s, mask, force, err, grid_limit, stir_rows, ctr, seq, chained, macro_out, stream);
}

template <typename S, int VS, bool MASK, bool FORCE, int NST>
static cudaError_t launch_batch_v(const BatchTables &bt, const Geometry<typename RealOf<S>::type> &w,
                                  const Physics<typename RealOf<S>::type> &p, int srows, double amp,
                                  const long long *bstep, int grid_limit, int ntiles, cudaStream_t stream) {
  using TL = Tile<S, VS>;
  constexpr int CPT = sizeof(S) == 8 ? 1 : 2;
  constexpr int NT = TILE_THREADS;
  auto kern = batch_step_kernel<S, VS, MASK, FORCE, CPT, NST>;
  const int smem = TL::smem(NST, FORCE ? srows : 0) + NST * (int)sizeof(TileInfo);
  static int configured_dev = -1, configured_smem = -1, max_blocks = 0, sms = 0;
  int dev = 0;
  cudaGetDevice(&dev);
  if (configured_dev != dev || configured_smem != smem) {
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
    if (e != cudaSuccess) return e;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&max_blocks, kern, NT, smem);
    if (e != cudaSuccess) return e;
    e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    configured_dev = dev;
    configured_smem = smem;
  }
  int workers = max_blocks * sms;
  if (grid_limit > 0 && grid_limit < workers) workers = grid_limit;
  if (workers > ntiles) workers = ntiles;
  if (workers < 1) workers = 1;
  kern<<<workers, NT, smem, stream>>>(bt, w, p, FORCE ? srows : 0, amp, bstep);
  return cudaGetLastError();
}

template <typename S, int NST>
static cudaError_t launch_batch_n(int vset, const BatchTables &bt, const Geometry<typename RealOf<S>::type> &w,
                                  const Physics<typename RealOf<S>::type> &p, int srows, double amp,
                                  const long long *bstep, bool mask, bool force, int grid_limit, int ntiles,
                                  cudaStream_t st) {
  if (vset == 3) {
    if (force) {
      if (mask) return launch_batch_v<S, 3, true, true, NST>(bt, w, p, srows, amp, bstep, grid_limit, ntiles, st);
      return launch_batch_v<S, 3, false, true, NST>(bt, w, p, srows, amp, bstep, grid_limit, ntiles, st);
    }
    if (mask) return launch_batch_v<S, 3, true, false, NST>(bt, w, p, srows, amp, bstep, grid_limit, ntiles, st);
    return launch_batch_v<S, 3, false, false, NST>(bt, w, p, srows, amp, bstep, grid_limit, ntiles, st);
  }
  if (mask) return launch_batch_v<S, 2, true, false, NST>(bt, w, p, srows, amp, bstep, grid_limit, ntiles, st);
  return launch_batch_v<S, 2, false, false, NST>(bt, w, p, srows, amp, bstep, grid_limit, ntiles, st);
}

template <typename S>
static cudaError_t launch_batch_t(int vset, const BatchTables &bt, const HostGeom &hw, const HostPhys &hp, int srows,
                                  double amp, const long long *bstep, bool mask, int stages, int grid_limit,
                                  int ntiles, cudaStream_t stream) {
  using R = typename RealOf<S>::type;
  const Geometry<R> w = to_geom<S>(hw);
  Physics<R> p;
  p.omega0 = (R)hp.omega0; p.fpref = (R)hp.fpref; p.body_x = (R)hp.body_x; p.body_y = (R)hp.body_y;
  p.vmax2 = (R)hp.vmax2;
  p.stochastic = hp.stochastic;
  p.round_key = 0;
  p.step = 0;
  p.y_off = 0;
  const bool force = hp.has_force != 0;
  if (stages == 1)
    return launch_batch_n<S, 1>(vset, bt, w, p, srows, amp, bstep, mask, force, grid_limit, ntiles, stream);
  return launch_batch_n<S, 2>(vset, bt, w, p, srows, amp, bstep, mask, force, grid_limit, ntiles, stream);
}

template <typename S, int VS, bool MASK, int MODE>
static cudaError_t launch_observe_k(const S *fin, const Geometry<typename RealOf<S>::type> &g, double eps0, double vmax2,
                                    const ObsOut &o, unsigned *err, int blocks, cudaStream_t stream) {
  observe_kernel<S, VS, MASK, MODE><<<blocks, dim3(32, 8), 0, stream>>>(fin, g, eps0, (float)vmax2, o, err);
  return cudaGetLastError();
}

template <typename S, int VS, bool MASK>
static cudaError_t launch_observe_v(int mode, const S *fin, const Geometry<typename RealOf<S>::type> &g, double eps0,
                                    double vmax2, const ObsOut &o, unsigned *err, int sms, cudaStream_t stream) {
  const int ntiles = ((g.nx + 31) / 32) * ((g.ny + obs_rows<S>() - 1) / obs_rows<S>());
  // the fields' totals: at most 6 blocks per SM, which add up their tiles (fewer partial sums)
  if (mode == OBS_FIELDS) return launch_observe_k<S, VS, MASK, OBS_FIELDS>(fin, g, eps0, vmax2, o, err, ntiles < 6 * sms ? ntiles : 6 * sms, stream);
  if (mode == OBS_V) return launch_observe_k<S, VS, MASK, OBS_V>(fin, g, eps0, vmax2, o, err, ntiles, stream);
  return launch_observe_k<S, VS, MASK, OBS_COLS>(fin, g, eps0, vmax2, o, err, ntiles, stream);
}

template <typename S>
static cudaError_t launch_observe_t(int vset, int mode, const void *fin, const HostGeom &hg, double eps0, double vmax2,
                                    const HostObs &ho, unsigned *err, int sms, cudaStream_t stream) {
  using R = typename RealOf<S>::type;
  const Geometry<R> g = to_geom<S>(hg);
  const ObsOut o{ho.eps, ho.ux, ho.uy, ho.z, ho.partials, ho.totals, ho.sync, ho.bins, ho.nbins, ho.zscale};
  const bool mask = hg.nbmask != nullptr;
  const S *a = (const S *)fin;
  if (vset == 3) {
    if (mask) return launch_observe_v<S, 3, true>(mode, a, g, eps0, vmax2, o, err, sms, stream);
    return launch_observe_v<S, 3, false>(mode, a, g, eps0, vmax2, o, err, sms, stream);
  }
  if (mask) return launch_observe_v<S, 2, true>(mode, a, g, eps0, vmax2, o, err, sms, stream);
  return launch_observe_v<S, 2, false>(mode, a, g, eps0, vmax2, o, err, sms, stream);
}

template <typename S>
static cudaError_t launch_ghosts_t(int vset, void *f, const HostGeom &hg, cudaStream_t stream) {
  using R = typename RealOf<S>::type;
  const Geometry<R> g = to_geom<S>(hg);
  const int nper = 2 * (hg.ny + 2) + 2 * hg.nx;
  const dim3 grid((nper + 255) / 256, vset == 3 ? VSet<3>::Q : VSet<2>::Q);
  if (vset == 3) fill_ghosts_kernel<S, 3><<<grid, 256, 0, stream>>>((S *)f, g);
  else fill_ghosts_kernel<S, 2><<<grid, 256, 0, stream>>>((S *)f, g);
  return cudaGetLastError();
}

template <typename S>
static cudaError_t launch_init_t(int vset, void *fout, const HostGeom &hg, double eps0, const double *eps,
                                 const double *ux, const double *uy, cudaStream_t stream) {
  using R = typename RealOf<S>::type;
  const Geometry<R> g = to_geom<S>(hg);
  const dim3 block(32, 8);
  const dim3 grid((hg.nx + 31) / 32, (hg.ny + 7) / 8);
  if (vset == 3) init_kernel<S, 3><<<grid, block, 0, stream>>>((S *)fout, g, eps0, eps, ux, uy);
  else init_kernel<S, 2><<<grid, block, 0, stream>>>((S *)fout, g, eps0, eps, ux, uy);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  return launch_ghosts_t<S>(vset, fout, hg, stream);
}

template <typename S>
static cudaError_t launch_open_ghosts_t(int vset, void *f, const HostGeom &hg, double ux_in, cudaStream_t stream) {
  using R = typename RealOf<S>::type;
  const Geometry<R> g = to_geom<S>(hg);
  const dim3 grid((hg.ny + 2 + 127) / 128, vset == 3 ? VSet<3>::Q : VSet<2>::Q);
  if (vset == 3) open_ghosts_kernel<S, 3><<<grid, 128, 0, stream>>>((S *)f, g, ux_in);
  else open_ghosts_kernel<S, 2><<<grid, 128, 0, stream>>>((S *)f, g, ux_in);
  return cudaGetLastError();
}

template <typename S>
static cudaError_t launch_stir_tables_t(const HostStir &hs, void *G, long long table, int nx, long long n, int count,
                                        cudaStream_t stream) {
  using R = typename RealOf<S>::type;
  const int chunks = (nx + stir_chunk<R>() - 1) / stir_chunk<R>();
  const long long warps = (long long)count * hs.nrows * chunks;
  if (warps == 0) return cudaSuccess;
  stir_tables_kernel<R><<<(unsigned)((warps + 3) / 4), 128, 0, stream>>>(to_modes(hs), (R4<R> *)G, table, hs.nrows, nx, n, count);
  return cudaGetLastError();
}

}  // namespace rlbm

#define RLBM_DEFINE_LAUNCHERS(S, SUF)                                                                    \
  namespace rlbm {                                                                                       \
  cudaError_t launch_step_##SUF(int vset, const void *tin, const void *tg, const void *tey, void *fout,     \
                                const HostGeom &g, const HostPhys &p, const HostStir &s, unsigned *err, \
                                int grid_limit, int stages, int stir_rows, int *ctr, unsigned seq,      \
                                bool chained, void *macro_out, cudaStream_t st) {                        \
    return launch_step_t<S>(vset, tin, tg, tey, fout, g, p, s, err, grid_limit, stages, stir_rows, ctr, seq, \
                            chained, macro_out, st);                                                    \
  }                                                                                                      \
  cudaError_t launch_batch_step_##SUF(int vset, const BatchTables &bt, const HostGeom &w, const HostPhys &p, \
                                      int srows, double amp, const long long *bstep, bool mask, int stages, \
                                      int grid_limit, int ntiles, cudaStream_t st) {                        \
    return launch_batch_t<S>(vset, bt, w, p, srows, amp, bstep, mask, stages, grid_limit, ntiles, st);    \
  }                                                                                                      \
  cudaError_t launch_observe_##SUF(int vset, int mode, const void *fin, const HostGeom &g, double eps0,   \
                                   double vmax2, const HostObs &o, unsigned *err, int sms, cudaStream_t st) { \
    return launch_observe_t<S>(vset, mode, fin, g, eps0, vmax2, o, err, sms, st);                         \
  }                                                                                                      \
  cudaError_t launch_init_##SUF(int vset, void *fout, const HostGeom &g, double eps0, const double *e,  \
                                const double *ux, const double *uy, cudaStream_t st) {                   \
    return launch_init_t<S>(vset, fout, g, eps0, e, ux, uy, st);                                         \
  }                                                                                                      \
  cudaError_t launch_ghosts_##SUF(int vset, void *f, const HostGeom &g, cudaStream_t st) {              \
    return launch_ghosts_t<S>(vset, f, g, st);                                                           \
  }                                                                                                      \
  cudaError_t launch_open_ghosts_##SUF(int vset, void *f, const HostGeom &g, double ux_in, cudaStream_t st) { \
    return launch_open_ghosts_t<S>(vset, f, g, ux_in, st);                                               \
  }                                                                                                      \
  cudaError_t launch_stir_tables_##SUF(const HostStir &s, void *G, long long table, int nx, long long n,  \
                                       int count, cudaStream_t st) {                                     \
    return launch_stir_tables_t<S>(s, G, table, nx, n, count, st);                                        \
  }                                                                                                      \
  }
