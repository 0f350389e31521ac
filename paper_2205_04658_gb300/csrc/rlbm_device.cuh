// Device side of the relativistic lattice Boltzmann update (arXiv 2205.04658).
//
// State: normalised deviations h_i = f_i / (w_i eps0) - 1 of the post-collision
// populations f*_i, one SoA plane per folded velocity class, row pitch `pitch`.
//
// The paper's momentum set is the 26 unit vectors along the D3Q27 neighbour
// directions (Part I "Model and Methods"; Sec. "Boltzmann to Lattice Boltzmann").
// On a lattice one node thick in z, every population is even in v_z, so the pair
// (v_x, v_y, +v_z), (v_x, v_y, -v_z) is carried as one class with the summed weight
// and its v_z^2; this folds 26 directions into 17 classes exactly.
#pragma once

#include <cuda_runtime.h>
#include <cuda_fp16.h>
#include <cuda_bf16.h>
#include <stdint.h>

namespace rlbm {

// keep the scalar math overloads visible next to the packed-pair ones defined below
using ::fma;
using ::fmax;

enum : unsigned { ERR_UNSTABLE = 1u, ERR_UNPHYSICAL = 2u, ERR_TIMEOUT = 4u };

// ---------------------------------------------------------------------------
// Velocity classes.  VS = 3: the paper's set folded to 17 in-plane classes
// (weights 1/21, 4/105, 9/280 per 3-D direction, degree-7 spherical rule);
// VS = 2: 8 directions on the unit circle, weights 1/8.
// ---------------------------------------------------------------------------
#define RLBM_S2 0.70710678118654752440
#define RLBM_S3 0.57735026918962576451

template <int VS> struct VSet;

template <> struct VSet<3> {
  static constexpr int Q = 17;
  static constexpr int DP = 3;
  __host__ __device__ static constexpr double vx(int q) {
    return q == 1 ? 1.0 : q == 3 ? -1.0
         : (q == 5 || q == 8 || q == 9) ? RLBM_S2 : (q == 6 || q == 7 || q == 11) ? -RLBM_S2
         : (q == 13 || q == 16) ? RLBM_S3 : (q == 14 || q == 15) ? -RLBM_S3 : 0.0;
  }
  __host__ __device__ static constexpr double vy(int q) {
    return q == 2 ? 1.0 : q == 4 ? -1.0
         : (q == 5 || q == 6 || q == 10) ? RLBM_S2 : (q == 7 || q == 8 || q == 12) ? -RLBM_S2
         : (q == 13 || q == 14) ? RLBM_S3 : (q == 15 || q == 16) ? -RLBM_S3 : 0.0;
  }
  __host__ __device__ static constexpr double vz2(int q) {
    return q == 0 ? 1.0 : (q >= 9 && q <= 12) ? 0.5 : (q >= 13) ? (1.0 / 3.0) : 0.0;
  }
  __host__ __device__ static constexpr double w(int q) {
    return q == 0 ? 2.0 / 21.0 : q <= 4 ? 1.0 / 21.0 : q <= 8 ? 4.0 / 105.0
         : q <= 12 ? 8.0 / 105.0 : 9.0 / 140.0;
  }
  __host__ __device__ static constexpr int opp(int q) {
    return q == 0 ? 0 : q <= 4 ? ((q - 1 + 2) % 4) + 1 : q <= 8 ? ((q - 5 + 2) % 4) + 5
         : q <= 12 ? ((q - 9 + 2) % 4) + 9 : ((q - 13 + 2) % 4) + 13;
  }
  // f_eq coefficients: h_eq = (eps^ - 1) + CA eps^ u0 (u.v) + CB eps^ (u.v)^2 - CC eps^ |u|^2
  static constexpr double CA = 4.0, CB = 10.0, CC = 2.0;
  static constexpr double TAU_NUM = 5.0;  // tau_R = 5 (eta/s) / T
};

template <> struct VSet<2> {
  static constexpr int Q = 8;
  static constexpr int DP = 2;
  __host__ __device__ static constexpr double vx(int q) {
    return q == 0 ? 1.0 : q == 4 ? -1.0 : (q == 1 || q == 7) ? RLBM_S2 : (q == 3 || q == 5) ? -RLBM_S2 : 0.0;
  }
  __host__ __device__ static constexpr double vy(int q) {
    return q == 2 ? 1.0 : q == 6 ? -1.0 : (q == 1 || q == 3) ? RLBM_S2 : (q == 5 || q == 7) ? -RLBM_S2 : 0.0;
  }
  __host__ __device__ static constexpr double vz2(int) { return 0.0; }
  __host__ __device__ static constexpr double w(int) { return 0.125; }
  __host__ __device__ static constexpr int opp(int q) { return (q + 4) % 8; }
  static constexpr double CA = 3.0, CB = 6.0, CC = 1.5;
  static constexpr double TAU_NUM = 4.0;
};

// sign of the streaming displacement of class q (compile time)
template <int VS> __host__ __device__ constexpr int sgnx(int q) {
  return VSet<VS>::vx(q) > 1e-12 ? 1 : VSet<VS>::vx(q) < -1e-12 ? -1 : 0;
}
template <int VS> __host__ __device__ constexpr int sgny(int q) {
  return VSet<VS>::vy(q) > 1e-12 ? 1 : VSet<VS>::vy(q) < -1e-12 ? -1 : 0;
}

// ---------------------------------------------------------------------------
// Storage conversions
// ---------------------------------------------------------------------------
// Scale of the stored deviations.  FP16 storage holds 2^8 h: the deviations down to 2^-22
// (not 2^-14) then lie in FP16's normal range, where the stochastic rounding of the stores
// is unbiased, and |h| up to 255 stays below FP16's largest value.  Powers of two, so the
// scaling itself is exact.
template <typename S> struct HScale {
  static constexpr float up = 1.0f, down = 1.0f;
};
template <> struct HScale<__half> {
  static constexpr float up = 256.0f, down = 1.0f / 256.0f;
};

// h of one stored value (load_h: global memory through the read-only path; load_h_s:
// shared memory) and h to its stored form.
template <typename S, typename R> __device__ __forceinline__ R load_h(const S *p) { return (R)__ldg(p); }
template <> __device__ __forceinline__ float load_h<__half, float>(const __half *p) {
  return __half2float(__ldg(p)) * HScale<__half>::down;
}
template <> __device__ __forceinline__ float load_h<__nv_bfloat16, float>(const __nv_bfloat16 *p) {
  return __bfloat162float(__ldg(p));
}
template <typename S, typename R> __device__ __forceinline__ R load_h_s(const S *p) { return (R)*p; }
template <> __device__ __forceinline__ float load_h_s<__half, float>(const __half *p) {
  return __half2float(*p) * HScale<__half>::down;
}
template <> __device__ __forceinline__ float load_h_s<__nv_bfloat16, float>(const __nv_bfloat16 *p) {
  return __bfloat162float(*p);
}
// A stored value as FP32 without the storage scale (the paired step kernels fold 1 / up
// into their pull weights).
template <typename S> __device__ __forceinline__ float load_s_raw(const S *p) { return load_h_s<S, float>(p); }
template <> __device__ __forceinline__ float load_s_raw<__half>(const __half *p) { return __half2float(*p); }
template <typename S, typename R> __device__ __forceinline__ S store_h(R v) { return (S)v; }
template <> __device__ __forceinline__ __half store_h<__half, float>(float v) {
  return __float2half_rn(v * HScale<__half>::up);
}
template <> __device__ __forceinline__ __nv_bfloat16 store_h<__nv_bfloat16, float>(float v) {
  return __float2bfloat16_rn(v);
}

template <typename S> struct RealOf { using type = float; };
template <> struct RealOf<double> { using type = double; };

// ---------------------------------------------------------------------------
// Storage layout.  Each population plane holds (ny + 2) rows of `pitch` elements:
// interior cell (x, y) sits at row y + 1, column x + XOFF; column XOFF - 1 and XOFF + nx
// and rows 0 and ny + 1 are ghost copies of the periodic neighbours (solid walls keep
// zero ghost rows).  XOFF is 128 bytes, so interior rows start on a 128-byte line.
// ---------------------------------------------------------------------------
template <typename S> struct PadLayout {
  static constexpr int XOFF = 128 / (int)sizeof(S);
  static constexpr int V = 16 / (int)sizeof(S);  // TMA x granule (16 bytes)
};

// ---------------------------------------------------------------------------
// Tiles: 32 columns by 8 rows, two rows per thread, for the FP32-compute paths; by 4 rows, one per
// thread, for FP64.  Either way a CTA has four warps, one on each quarter of the SM: a warp's
// FP64 instruction takes 64 cycles whatever its lanes, and eight warps of an SM share the FP64
// units (74 ns per instruction instead of 37), so FP64 tiles of 8 rows left half the rate unused
// on lattices of fewer tiles than SMs.
// ---------------------------------------------------------------------------
template <typename S> struct TileRows { static constexpr int value = 8; };
template <> struct TileRows<double> { static constexpr int value = 4; };
constexpr int TILE_X = 32, TILE_THREADS = 128;

// ---------------------------------------------------------------------------
// Parameters
// ---------------------------------------------------------------------------
template <typename R> struct alignas(16) R4 { R x, y, z, w; };
template <typename R> struct alignas(2 * sizeof(R)) R2 { R x, y; };

template <typename R> struct Geometry {
  int nx, ny, pitch;
  long long plane;          // elements per plane (pitch * (ny + 2))
  int walls;                // y ghost rows are solid (never written)
  const uint16_t *nbmask;   // bit 4: cell solid; bit (dy+1)*3+(dx+1): neighbour (x+dx, y+dy) solid
  R beta[17][4];            // bilinear weights of corners (0,0), (s_x,0), (0,s_y), (s_x,s_y)
  float2 beta2[17][4];      // the same duplicated into pairs (packed two-cell arithmetic)
};

template <typename R> struct Physics {
  R omega0;        // dt T0 / (TAU_NUM eta/s): relaxation factor at eps = eps0
  R fpref;         // -6 dt / T0: force prefactor including dt
  R body_x, body_y;
  R vmax2;         // FP32 path: |v|^2 above which Landau runs in FP64
  int stochastic;  // 16-bit storage: stochastic rounding
  unsigned round_key;
  unsigned step;   // low 32 bits of the step index (rounding bits)
  int y_off;       // lattice row of row 0 (a strip of a larger lattice; else 0): rounding bits
};

// ---------------------------------------------------------------------------
// Stochastic rounding of the 16-bit stores: unbiased (E[round(v)] = v), so the rounding
// errors of successive steps do not add up coherently.  The random bits are a
// counter-based hash of (cell, step, key), advanced by a Weyl step (an odd constant near
// 2^32 / golden ratio added modulo 2^32) per value, so a run repeats exactly.  Every value's
// bits are uniform because the hash is; the 17 values of one cell take evenly spread
// offsets from it.  (An integer add, where a multiplicative generator would occupy the
// FMA pipe that the cell's arithmetic already saturates.)
// ---------------------------------------------------------------------------
__device__ __forceinline__ uint32_t cell_hash(uint32_t x, uint32_t y, uint32_t step, uint32_t key) {
  uint32_t h = (x * 0x9E3779B1u) ^ ((y + 0x7F4A7C15u) * 0x85EBCA77u) ^ ((step ^ key) * 0xC2B2AE3Du);
  h ^= h >> 16; h *= 0x7FEB352Du; h ^= h >> 15; h *= 0x846CA68Bu; h ^= h >> 16;
  return h;
}
__device__ __forceinline__ uint32_t next_bits(uint32_t r) { return r + 0x9E3779B9u; }

// v rounded to storage type S: to nearest, or stochastically with the random bits r.
// BF16: adding 16 random bits below the kept mantissa of the FP32 pattern and truncating
// (round toward zero) rounds the magnitude up with probability equal to the dropped
// fraction.  (FP16 pairs: round_pair_f16 below.)
template <typename S> __device__ __forceinline__ S store_round(float v, bool sr, uint32_t r) {
  return store_h<S, float>(v);
}
template <> __device__ __forceinline__ __nv_bfloat16 store_round<__nv_bfloat16>(float v, bool sr, uint32_t r) {
  if (!sr) return __float2bfloat16_rn(v);
  return __ushort_as_bfloat16((unsigned short)((__float_as_uint(v) + (r >> 16)) >> 16));
}

// The two cells of a pair, already multiplied by the storage scale, rounded stochastically
// to FP16 in one packed conversion with the random bits ra, rb (the low half of the result
// holds a, the high half b): 13 random bits are added below the kept FP16 mantissa of each
// FP32 value and the sums are truncated (round toward zero), which rounds the magnitude up
// with probability equal to the dropped fraction.  Below FP16's normal range (2^-14, i.e.
// |h| < 2^-22) the 13 bits do not reach every dropped bit and the rounding leans toward
// zero by less than one FP16 subnormal spacing, 2^-32 in h.
__device__ __forceinline__ uint32_t round_pair_f16_sr(float a, float b, uint32_t ra, uint32_t rb) {
  const float ua = __uint_as_float(__float_as_uint(a) + (ra >> 19));
  const float ub = __uint_as_float(__float_as_uint(b) + (rb >> 19));
  uint32_t d;
  asm("cvt.rz.f16x2.f32 %0, %1, %2;" : "=r"(d) : "f"(ub), "f"(ua));  // (high, low) = (b, a)
  return d;
}
// The same rounded to nearest.
__device__ __forceinline__ uint32_t round_pair_f16_rn(float a, float b) {
  const __half2 h = __floats2half2_rn(a, b);
  return *reinterpret_cast<const uint32_t *>(&h);
}

// The stirring modes of a lattice, grouped in rows of equal k_y (device pointers).
struct StirModes {
  const int *kx;          // [nmodes]
  const int *row_start;   // [nrows + 1] mode range of each row (modes sorted by k_y)
  const void *tw;         // [nx] R2: exp(i 2 pi j / nx)
  const double *scale;    // [nmodes] amplitude multipliers sigma_m; NULL = all 1
  unsigned long long seed;
  double amp;
};

template <typename R> struct Stir {
  int nrows;               // distinct k_y of the shell (0 = no stirring)
  const R4<R> *G_cur;      // [nrows][nx]: (Gx.re, -Gx.im, Gy.re, -Gy.im) of this step
  const R2<R> *EY;         // [nrows][eyp]: exp(i 2 pi k_y(row) y / ny), rows padded to eyp
  int eyp;
  R4<R> *G_next;           // the table of step step_next, built by the same launch (NULL: none)
  long long step_next;
  StirModes modes;
};

// ---------------------------------------------------------------------------
// Philox4x32-10 (Salmon, Moraes, Dror, Shaw, SC'11) and the stirring draws
// ---------------------------------------------------------------------------
__device__ __forceinline__ void philox4x32_10(uint32_t c[4], uint32_t k0, uint32_t k1) {
#pragma unroll
  for (int r = 0; r < 10; ++r) {
    if (r) { k0 += 0x9E3779B9u; k1 += 0xBB67AE85u; }
    const uint32_t lo0 = 0xD2511F53u * c[0], hi0 = __umulhi(0xD2511F53u, c[0]);
    const uint32_t lo1 = 0xCD9E8D57u * c[2], hi1 = __umulhi(0xCD9E8D57u, c[2]);
    const uint32_t n0 = hi1 ^ c[1] ^ k0, n2 = hi0 ^ c[3] ^ k1;
    c[0] = n0; c[1] = lo1; c[2] = n2; c[3] = lo0;
  }
}

// Mode m of step n: a = amp sqrt(-2 ln u0) cos(2 pi u1), phi = 2 pi u2, psi = 2 pi u3,
// coefficient pair (cx, cy) = a (cos psi, sin psi) exp(i phi).  FP64.
__device__ inline void stir_draw(unsigned long long seed, long long n, int m, double amp, double out[4]) {
  uint32_t c[4] = {(uint32_t)(n & 0xffffffffll), (uint32_t)m, (uint32_t)((unsigned long long)n >> 32), 0u};
  philox4x32_10(c, (uint32_t)(seed & 0xffffffffull), (uint32_t)(seed >> 32));
  double u[4];
#pragma unroll
  for (int j = 0; j < 4; ++j) u[j] = ((double)c[j] + 0.5) * 2.3283064365386962890625e-10;
  const double a = amp * sqrt(-2.0 * log(u[0])) * cospi(2.0 * u[1]);
  double sphi, cphi, spsi, cpsi;
  sincospi(2.0 * u[2], &sphi, &cphi);
  sincospi(2.0 * u[3], &spsi, &cpsi);
  out[0] = a * cpsi * cphi; out[1] = a * cpsi * sphi;
  out[2] = a * spsi * cphi; out[3] = a * spsi * sphi;
}

// Mode m of step n in FP32 (the draws of the FP32-compute paths; the uniform u_j and
// the Box-Muller transform in single precision, about 1e-7 relative).
__device__ inline void stir_draw_f32(unsigned long long seed, long long n, int m, float amp, float out[4]) {
  uint32_t c[4] = {(uint32_t)(n & 0xffffffffll), (uint32_t)m, (uint32_t)((unsigned long long)n >> 32), 0u};
  philox4x32_10(c, (uint32_t)(seed & 0xffffffffull), (uint32_t)(seed >> 32));
  float u[4];
#pragma unroll
  for (int j = 0; j < 4; ++j) u[j] = ((float)c[j] + 0.5f) * 2.3283064365386962890625e-10f;
  const float a = amp * sqrtf(-2.0f * logf(u[0])) * cospif(2.0f * u[1]);
  float sphi, cphi, spsi, cpsi;
  sincospif(2.0f * u[2], &sphi, &cphi);
  sincospif(2.0f * u[3], &spsi, &cpsi);
  out[0] = a * cpsi * cphi; out[1] = a * cpsi * sphi;
  out[2] = a * spsi * cphi; out[3] = a * spsi * sphi;
}

template <typename R>
__device__ __forceinline__ R4<R> stir_draw_r(unsigned long long seed, long long n, int m, double amp) {
  if constexpr (sizeof(R) == 8) {
    double c[4];
    stir_draw(seed, n, m, amp, c);
    return R4<R>{c[0], c[1], c[2], c[3]};
  } else {
    float c[4];
    stir_draw_f32(seed, n, m, (float)amp, c);
    return R4<R>{c[0], c[1], c[2], c[3]};
  }
}

// One row of a step's stirring table for the columns of one chunk, by one warp:
//   G_r(x) = sum_{m in row r} (cx_m, cy_m) exp(i 2 pi k_x,m x / nx),
// kept as (Re, -Im) of both components.  F = Re[G_r(x) exp(i 2 pi k_y y / ny)] is then a sum of
// products of parts that lie side by side, as packed multiply-adds take them.  Each lane draws
// modes of the row (Philox is counter-based: no state is kept between steps) and every lane
// adds all of them for its columns x0 + lane, + 32, ...; the phase is read from the table of
// the nx roots of unity at the exact residue k_x x mod nx.
// A chunk is one warp's serial chain over the row's modes, up to two dozen at a shell of 6 to 12,
// and a small lattice's step waits for it: two columns per lane in FP32 keep it short (128^2, 166
// modes: 5.1 us per step against 7.2 with eight; 512^2 10.0 against 12.2; 1024^2 and 4096^2 alike; one
// column: the draws are then made twice as often).  The loop over the modes is not unrolled: copies
// of its body take 1 us more off those two, but cost masked FP32 lattices, whose body force
// compiles the same kernel without running the loop, 6 % (1024 x 256: 9.1 us against 8.5).  In FP64
// the draws are most of it, so a chunk is wider.
template <typename R> constexpr int stir_chunk() { return 32 * (sizeof(R) == 8 ? 4 : 2); }

template <typename R>
__device__ __forceinline__ void stir_row_chunk(const StirModes &s, long long step, int r, int chunk, int nx, int lane,
                                               R4<R> *row) {
  constexpr int NCOL = stir_chunk<R>() / 32;
  const int x0 = chunk * stir_chunk<R>() + lane;
  const int m1 = s.row_start[r + 1];
  R4<R> g[NCOL];
#pragma unroll
  for (int i = 0; i < NCOL; ++i) g[i] = R4<R>{R(0), R(0), R(0), R(0)};
  for (int m0 = s.row_start[r]; m0 < m1; m0 += 32) {
    R4<R> c{R(0), R(0), R(0), R(0)};
    int kx = 0;
    if (m0 + lane < m1) {
      kx = s.kx[m0 + lane];
      c = stir_draw_r<R>(s.seed, step, m0 + lane, s.scale ? s.amp * s.scale[m0 + lane] : s.amp);
    }
    // residues of the lane's first column and of 32 columns (|k_x| < nx / 2, x < 2^15 + 2^8: no overflow)
    int d = (32 * kx) % nx;
    if (d < 0) d += nx;
    const int cnt = m1 - m0 < 32 ? m1 - m0 : 32;
#pragma unroll 1
    for (int k = 0; k < cnt; ++k) {
      const R4<R> a{__shfl_sync(0xffffffffu, c.x, k), __shfl_sync(0xffffffffu, c.y, k),
                    __shfl_sync(0xffffffffu, c.z, k), __shfl_sync(0xffffffffu, c.w, k)};
      const int kk = __shfl_sync(0xffffffffu, kx, k), dd = __shfl_sync(0xffffffffu, d, k);
      int j = (kk * x0) % nx;
      if (j < 0) j += nx;
#pragma unroll
      for (int i = 0; i < NCOL; ++i) {
        R2<R> e;
        if constexpr (sizeof(R) == 8) {
          const double2 v = __ldg(reinterpret_cast<const double2 *>(s.tw) + j);
          e = R2<R>{v.x, v.y};
        } else {
          const float2 v = __ldg(reinterpret_cast<const float2 *>(s.tw) + j);
          e = R2<R>{v.x, v.y};
        }
        g[i].x = fma(a.x, e.x, fma(-a.y, e.y, g[i].x));
        g[i].y = fma(-a.x, e.y, fma(-a.y, e.x, g[i].y));
        g[i].z = fma(a.z, e.x, fma(-a.w, e.y, g[i].z));
        g[i].w = fma(-a.z, e.y, fma(-a.w, e.x, g[i].w));
        j += dd;
        if (j >= nx) j -= nx;
      }
    }
  }
#pragma unroll
  for (int i = 0; i < NCOL; ++i)
    if (x0 + 32 * i < nx) row[x0 + 32 * i] = g[i];
}

// The phase table EY_r(y) = exp(i 2 pi k_y(r) y / ny): rows of eyp entries (re, im).
template <typename R> __device__ __forceinline__ R2<R> ey_at(const R *row, int y) {
  return R2<R>{row[2 * y], row[2 * y + 1]};
}

// ---------------------------------------------------------------------------
// Arithmetic helpers: correctly rounded or within an ulp or two in FP64, hardware approximations
// (<= 2 ulp) in FP32.
// ---------------------------------------------------------------------------
template <typename T> struct FM;
// FP64 roots by Newton's method from the FP32 approximation (1e-7), two steps (1e-14, rounding):
// 8 to 10 FP64 operations where the library functions take about 30, and on GB300 a warp's FP64
// instruction occupies its quarter of the SM for 64 cycles.  Arguments beyond FP32's range take
// the library functions.
template <> struct FM<double> {
  static __device__ __forceinline__ bool in_range(double x) { return x > 1e-30 && x < 1e30; }
  static __device__ __forceinline__ double rcp(double x) { return 1.0 / x; }
  static __device__ __forceinline__ double sqrt_(double x) { return sqrt(x); }
  static __device__ __forceinline__ double rsqrt(double x) {
    if (!in_range(x)) return 1.0 / sqrt(x);
    double y = (double)rsqrtf((float)x);
#pragma unroll
    for (int i = 0; i < 2; ++i) y = fma(0.5 * y, fma(-x * y, y, 1.0), y);
    return y;
  }
  static __device__ __forceinline__ double qroot(double x) {  // x^(1/4): q += (x - q^4) / (4 q^3)
    if (!in_range(x)) return sqrt(sqrt(x));
    const float f = rsqrtf(rsqrtf((float)x));
    const double c = (double)__fdividef(0.25f, f * f * f);
    double q = (double)f;
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      const double q2 = q * q;
      q = fma(c, fma(-q2, q2, x), q);
    }
    return q;
  }
  static __device__ __forceinline__ double croot(double x) {  // x^(1/3): q += (x - q^3) / (3 q^2)
    if (!in_range(x)) return cbrt(x);
    const float f = cbrtf((float)x);
    const double c = (double)__fdividef(1.0f, 3.0f * f * f);
    double q = (double)f;
#pragma unroll
    for (int i = 0; i < 2; ++i) q = fma(c, fma(-q * q, q, x), q);
    return q;
  }
};
// The .ftz forms are one instruction each; the others bring the scaling of subnormal arguments
// along (a compare, a select and two multiplications per call, a twentieth of the step
// kernel's instructions), and no argument here comes near those: T^00, determinants near
// -(1 + 1/D_p)^2 to -1, 1 - v^2, eps^ > 0 (an eps^ or 1 - v^2 so close to zero is reported as
// unstable or re-solved in FP64).
template <> struct FM<float> {
  static __device__ __forceinline__ float rcp(float x) {
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
  }
  static __device__ __forceinline__ float rsqrt(float x) {
    float r;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
  }
  static __device__ __forceinline__ float sqrt_(float x) {
    float r;
    asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
  }
  static __device__ __forceinline__ float qroot(float x) { return rsqrt(rsqrt(x)); }
  static __device__ __forceinline__ float croot(float x) { return cbrtf(x); }
};

// Two FP32 lanes (two lattice cells) in one register pair: Blackwell's packed FP32
// add/multiply/FMA (__fadd2_rn, __fmul2_rn, __ffma2_rn) do both in one instruction.
struct F2 {
  float2 v;
  F2() = default;  // (uninitialised)
  __device__ __forceinline__ explicit F2(float s) : v(make_float2(s, s)) {}
  __device__ __forceinline__ explicit F2(double s) : v(make_float2((float)s, (float)s)) {}
  __device__ __forceinline__ explicit F2(int s) : v(make_float2((float)s, (float)s)) {}
  __device__ __forceinline__ F2(float a, float b) : v(make_float2(a, b)) {}
  __device__ __forceinline__ explicit F2(float2 w) : v(w) {}
  __device__ __forceinline__ F2 &operator+=(F2 o) { v = __fadd2_rn(v, o.v); return *this; }
  __device__ __forceinline__ F2 &operator-=(F2 o) { v = __ffma2_rn(o.v, make_float2(-1.0f, -1.0f), v); return *this; }
};
__device__ __forceinline__ F2 operator+(F2 a, F2 b) { return F2(__fadd2_rn(a.v, b.v)); }
__device__ __forceinline__ F2 operator*(F2 a, F2 b) { return F2(__fmul2_rn(a.v, b.v)); }
__device__ __forceinline__ F2 operator-(F2 a) { return F2(make_float2(-a.v.x, -a.v.y)); }
__device__ __forceinline__ F2 operator-(F2 a, F2 b) { return F2(__ffma2_rn(b.v, make_float2(-1.0f, -1.0f), a.v)); }
__device__ __forceinline__ F2 fma(F2 a, F2 b, F2 c) { return F2(__ffma2_rn(a.v, b.v, c.v)); }
__device__ __forceinline__ F2 fmax(F2 a, F2 b) { return F2(fmaxf(a.v.x, b.v.x), fmaxf(a.v.y, b.v.y)); }
// a / b, correctly rounded per lane
template <typename T> __device__ __forceinline__ T divide(T a, T b) { return a / b; }
__device__ __forceinline__ F2 divide(F2 a, F2 b) { return F2(a.v.x / b.v.x, a.v.y / b.v.y); }

// Numbers as unevaluated sums h + l of two FP32 values (about 48 bits), two to a packed pair: sums
// and transforms of FP32 data that must not round at FP32, at FP32's rate (GB300's FP64 units run
// at 1/64 of it).  The sum is Knuth's exact two-sum of the high parts with the low parts added
// (Dekker 1971; error below 2^-46 (|a| + |b|)), the product an FMA-exact product of the high
// parts plus the cross terms.
struct DF2 {
  F2 h, l;
};
__device__ __forceinline__ DF2 df_norm(F2 h, F2 l) {  // |h| >= |l|
  const F2 s = h + l;
  return DF2{s, l - (s - h)};
}
__device__ __forceinline__ DF2 df_add(const DF2 &a, const DF2 &b) {
  const F2 s = a.h + b.h, bb = s - a.h;
  const F2 e = (a.h - (s - bb)) + (b.h - bb);
  return df_norm(s, e + (a.l + b.l));
}
__device__ __forceinline__ DF2 df_add(const DF2 &a, F2 b) {
  const F2 s = a.h + b, bb = s - a.h;
  const F2 e = (a.h - (s - bb)) + (b - bb);
  return df_norm(s, e + a.l);
}
__device__ __forceinline__ DF2 df_neg(const DF2 &a) { return DF2{-a.h, -a.l}; }
__device__ __forceinline__ DF2 df_mul(const DF2 &a, const DF2 &b) {
  const F2 p = a.h * b.h;
  return df_norm(p, fma(a.l, b.h, fma(a.h, b.l, fma(a.h, b.h, -p))));
}
__device__ __forceinline__ F2 shfl_xor(F2 a, int off) {
  return F2(__shfl_xor_sync(0xffffffffu, a.v.x, off), __shfl_xor_sync(0xffffffffu, a.v.y, off));
}
__device__ __forceinline__ DF2 df_shfl_xor(const DF2 &a, int off) { return DF2{shfl_xor(a.h, off), shfl_xor(a.l, off)}; }

template <> struct FM<F2> {
  static __device__ __forceinline__ F2 rcp(F2 x) { return F2(FM<float>::rcp(x.v.x), FM<float>::rcp(x.v.y)); }
  static __device__ __forceinline__ F2 rsqrt(F2 x) { return F2(FM<float>::rsqrt(x.v.x), FM<float>::rsqrt(x.v.y)); }
  static __device__ __forceinline__ F2 sqrt_(F2 x) { return F2(FM<float>::sqrt_(x.v.x), FM<float>::sqrt_(x.v.y)); }
  static __device__ __forceinline__ F2 qroot(F2 x) { return F2(FM<float>::qroot(x.v.x), FM<float>::qroot(x.v.y)); }
  static __device__ __forceinline__ F2 croot(F2 x) { return F2(cbrtf(x.v.x), cbrtf(x.v.y)); }
};

// ---------------------------------------------------------------------------
// Moments.  In units of eps0, with h the normalised deviations:
//   T^00 = 1 + e,  T^0a = m_a,  T^ab = delta_ab / D_p + t_ab  (a, b in {x, y})
//   e = sum w h, m = sum w h v, t = sum w h v v, and (for the force) the third
//   moments w_abc = sum w h v_a v_b v_c.  The rest-equilibrium parts are exact.
// ---------------------------------------------------------------------------
template <typename T> struct Mom { T e, mx, my, txx, txy, tyy, wxxx, wxxy, wxyy, wyyy; };

// Generic sum over classes with compile-time coefficients.  (The packed intrinsics are never
// contracted by the compiler, so the multiply-adds are written out.)
template <typename T, typename R, int VS, bool THIRD>
__device__ __forceinline__ Mom<T> moments_generic(const R h[VSet<VS>::Q]) {
  using V = VSet<VS>;
  const T z = T(0);
  Mom<T> M{z, z, z, z, z, z, z, z, z, z};
#pragma unroll
  for (int q = 0; q < V::Q; ++q) {
    const double w = V::w(q), vx = V::vx(q), vy = V::vy(q);
    const T hq = (T)h[q];
    M.e = fma(T(w), hq, M.e);
    if (vx != 0.0) { M.mx = fma(T(w * vx), hq, M.mx); M.txx = fma(T(w * vx * vx), hq, M.txx); }
    if (vy != 0.0) { M.my = fma(T(w * vy), hq, M.my); M.tyy = fma(T(w * vy * vy), hq, M.tyy); }
    if (vx != 0.0 && vy != 0.0) M.txy = fma(T(w * vx * vy), hq, M.txy);
    if (THIRD) {
      if (vx != 0.0) M.wxxx = fma(T(w * vx * vx * vx), hq, M.wxxx);
      if (vx != 0.0 && vy != 0.0) {
        M.wxxy = fma(T(w * vx * vx * vy), hq, M.wxxy);
        M.wxyy = fma(T(w * vx * vy * vy), hq, M.wxyy);
      }
      if (vy != 0.0) M.wyyy = fma(T(w * vy * vy * vy), hq, M.wyyy);
    }
  }
  return M;
}

// The 17 folded classes of the paper's set come in four sign-symmetric groups
// {(+a,+b), (-a,+b), (-a,-b), (+a,-b)} (diagonals) or {(+a,0), (0,+a), (-a,0), (0,-a)}
// (axes).  Sums and differences within a group (a butterfly) give each moment from one
// multiply-add per group instead of one per class.
template <typename T, bool THIRD>
__device__ __forceinline__ void moments_axis_group(Mom<T> &M, double w, double a, T h0, T h1, T h2, T h3) {
  // classes (+a,0), (0,+a), (-a,0), (0,-a)
  const T sx = h0 + h2, dx = h0 - h2, sy = h1 + h3, dy = h1 - h3;
  M.e = fma(T(w), sx + sy, M.e);
  M.mx = fma(T(w * a), dx, M.mx);
  M.my = fma(T(w * a), dy, M.my);
  M.txx = fma(T(w * a * a), sx, M.txx);
  M.tyy = fma(T(w * a * a), sy, M.tyy);
  if (THIRD) { M.wxxx = fma(T(w * a * a * a), dx, M.wxxx); M.wyyy = fma(T(w * a * a * a), dy, M.wyyy); }
}
// The diagonal groups (a, w) and (b, u) together: they alone reach t_xy, w_xxy and w_xyy.
template <typename T, bool THIRD>
__device__ __forceinline__ void moments_diag_groups(Mom<T> &M, double w, double a, T h0, T h1, T h2, T h3, double u,
                                                    double b, T g0, T g1, T g2, T g3) {
  // classes (+a,+a), (-a,+a), (-a,-a), (+a,-a)
  const T s02 = h0 + h2, d02 = h0 - h2, s13 = h1 + h3, d31 = h3 - h1;
  const T P0 = s02 + s13, Pxy = s02 - s13, Px = d02 + d31, Py = d02 - d31;
  const T r02 = g0 + g2, c02 = g0 - g2, r13 = g1 + g3, c31 = g3 - g1;
  const T Q0 = r02 + r13, Qxy = r02 - r13, Qx = c02 + c31, Qy = c02 - c31;
  M.e = fma(T(u), Q0, fma(T(w), P0, M.e));
  const T t2 = fma(T(u * b * b), Q0, T(w * a * a) * P0);
  M.txx += t2;
  M.tyy += t2;
  M.mx = fma(T(u * b), Qx, fma(T(w * a), Px, M.mx));
  M.my = fma(T(u * b), Qy, fma(T(w * a), Py, M.my));
  M.txy = fma(T(u * b * b), Qxy, T(w * a * a) * Pxy);
  if (THIRD) {
    M.wxyy = fma(T(u * b * b * b), Qx, T(w * a * a * a) * Px);
    M.wxxy = fma(T(u * b * b * b), Qy, T(w * a * a * a) * Py);
    M.wxxx += M.wxyy;
    M.wyyy += M.wxxy;
  }
}

template <typename T, typename R, int VS, bool THIRD>
__device__ __forceinline__ Mom<T> moments_of(const R h[VSet<VS>::Q]) {
  if constexpr (VS == 3) {
    using V = VSet<3>;
    Mom<T> M;
    {  // the unit axes start the sums
      const T sx = (T)h[1] + (T)h[3], dx = (T)h[1] - (T)h[3], sy = (T)h[2] + (T)h[4], dy = (T)h[2] - (T)h[4];
      constexpr double w = V::w(1);
      M.e = fma(T(w), sx + sy, T(V::w(0)) * (T)h[0]);
      M.mx = T(w) * dx;
      M.my = T(w) * dy;
      M.txx = T(w) * sx;
      M.tyy = T(w) * sy;
      M.wxxx = M.mx;
      M.wyyy = M.my;
    }
    moments_axis_group<T, THIRD>(M, V::w(9), RLBM_S2, (T)h[9], (T)h[10], (T)h[11], (T)h[12]);
    moments_diag_groups<T, THIRD>(M, V::w(5), RLBM_S2, (T)h[5], (T)h[6], (T)h[7], (T)h[8],
                                  V::w(13), RLBM_S3, (T)h[13], (T)h[14], (T)h[15], (T)h[16]);
    return M;
  } else {
    return moments_generic<T, R, VS, THIRD>(h);
  }
}

// ---------------------------------------------------------------------------
// Landau matching: the timelike eigenvector u = gamma (1, v) of T^mu_nu on the
// (t, x, y) block solves  R(v) = m - T^{ab} v_b - (T^00 - m.v) v = 0.  Starting point:
// the exact solution for an ideal fluid with the same T^00 and T^0a (for D_p = 3,
// |m| / T^00 = 4 v / (3 + v^2); for D_p = 2, 3 v / (2 + v^2)), then Newton steps.
// Returns false when the last Newton step is not small (|dv| > tol (|v| + 1e-6)) or
// the result is not a subluminal flow with positive energy density.
// ---------------------------------------------------------------------------
template <typename T, int VS>
__device__ __forceinline__ bool landau(const Mom<T> &M, int maxit, T tol, T &vx, T &vy) {
  constexpr T dinv = T(1.0 / VSet<VS>::DP);
  const T T00 = T(1) + M.e;
  const T i00 = FM<T>::rcp(T00);
  const T ax = M.mx * i00, ay = M.my * i00, m2 = ax * ax + ay * ay;
  T c;
  if (VS == 3) c = T(3) * FM<T>::rcp(T(2) + FM<T>::sqrt_(fmax(T(4) - T(3) * m2, T(0))));
  else c = T(4) * FM<T>::rcp(T(3) + FM<T>::sqrt_(fmax(T(9) - T(8) * m2, T(0))));
  vx = c * ax;
  vy = c * ay;
  const T Txx = dinv + M.txx, Txy = M.txy, Tyy = dinv + M.tyy;
  T d2 = T(0);
  for (int it = 0; it < maxit; ++it) {
    const T E = T00 - (M.mx * vx + M.my * vy);
    const T rx = M.mx - (Txx * vx + Txy * vy) - E * vx;
    const T ry = M.my - (Txy * vx + Tyy * vy) - E * vy;
    // J = dR/dv = -T^{ab} + v_a m_b - E delta_ab
    const T jxx = -Txx + vx * M.mx - E, jxy = -Txy + vx * M.my;
    const T jyx = -Txy + vy * M.mx, jyy = -Tyy + vy * M.my - E;
    const T idet = FM<T>::rcp(jxx * jyy - jxy * jyx);
    const T dx = (jxy * ry - jyy * rx) * idet;
    const T dy = (jyx * rx - jxx * ry) * idet;
    vx += dx;
    vy += dy;
    d2 = dx * dx + dy * dy;
    if constexpr (sizeof(T) == 8) {
      // Newton converges quadratically: after a step of |dv| = 1e-12 |v| the error is at rounding.
      // (A limit at the rounding itself, |dv| = 1e-16 |v|, is missed by the noise of the residual, and
      // whole warps run all 40 steps on the FP64 units, 1/64 of FP32's rate: 200 steps of a 64^2
      // lattice, all by this path, 5.4 ms against 26.5-31.4.  Cells that landau_refined solves
      // do not come here.)
      if (d2 <= 1e-24 * (vx * vx + vy * vy) + 1e-300) break;
    } else {
      if (d2 <= tol * tol * (T(1e-6) + vx * vx + vy * vy)) break;
    }
  }
  const T v2 = vx * vx + vy * vy;
  const T lim = tol * (T(1e-6) + v2);
  return (v2 < T(1)) && (T00 - (M.mx * vx + M.my * vy) > T(0)) && (d2 <= tol * lim);
}

// The FP64 solution from the FP32 one: the residual R(v) in FP64, the correction -J^{-1} R in FP32
// with the FP32 Jacobian, whose relative error (about 1e-6) is the factor by which a step reduces
// the error: two steps from FP32's 1e-7 to rounding, some 30 FP64 operations in place of four
// full Newton steps with an FP64 division each.  False when it has not converged (the full FP64
// iteration decides then).
template <int VS> __device__ __forceinline__ bool landau_refined(const Mom<double> &M, double &vx, double &vy) {
  Mom<float> f;
  f.e = (float)M.e; f.mx = (float)M.mx; f.my = (float)M.my;
  f.txx = (float)M.txx; f.txy = (float)M.txy; f.tyy = (float)M.tyy;
  float x, y;
  if (!landau<float, VS>(f, 4, 3e-4f, x, y)) return false;
  const float dinvf = 1.0f / VSet<VS>::DP;
  const float E = 1.0f + f.e - (f.mx * x + f.my * y);
  const float jxx = x * f.mx - (dinvf + f.txx) - E, jxy = x * f.my - f.txy;
  const float jyx = y * f.mx - f.txy, jyy = y * f.my - (dinvf + f.tyy) - E;
  const float idet = __fdividef(1.0f, jxx * jyy - jxy * jyx);
  constexpr double dinv = 1.0 / VSet<VS>::DP;
  const double nxx = -(dinv + M.txx), nyy = -(dinv + M.tyy), n00 = -(1.0 + M.e);
  vx = (double)x;
  vy = (double)y;
  for (int it = 0; it < 4; ++it) {
    const double nE = fma(M.mx, vx, fma(M.my, vy, n00));
    const float rx = (float)fma(nxx + nE, vx, fma(-M.txy, vy, M.mx));
    const float ry = (float)fma(nyy + nE, vy, fma(-M.txy, vx, M.my));
    const float dx = (jxy * ry - jyy * rx) * idet, dy = (jyx * rx - jxx * ry) * idet;
    vx += (double)dx;
    vy += (double)dy;
    // after a step of 1e-11 |v| the error is below rounding (the factor 1e-6 above)
    if (fabsf(dx) + fabsf(dy) <= 1e-11f * (fabsf(x) + fabsf(y))) return vx * vx + vy * vy < 1.0;
  }
  return false;
}

// Macroscopic result of one cell (eps^ = eps / eps0, u^mu = gamma (1, v)).
template <typename T> struct Macro { T eps_m1, u0, ux, uy, vx, vy; bool ok; };

// What a cell without a solution (ok false) is reported as: an energy density that is not positive
// and finite is an unstable run, else Landau matching found no timelike eigenvector.
template <typename T> __device__ __forceinline__ unsigned cell_error(const Macro<T> &m) {
  return T(1) + m.eps_m1 > T(0) && isfinite(m.eps_m1) ? ERR_UNPHYSICAL : ERR_UNSTABLE;
}
__device__ __forceinline__ unsigned cell_error(const Macro<F2> &m) {  // (of either cell)
  const float a = m.eps_m1.v.x, b = m.eps_m1.v.y;
  return 1.0f + a > 0.0f && isfinite(a) && 1.0f + b > 0.0f && isfinite(b) ? ERR_UNPHYSICAL : ERR_UNSTABLE;
}

template <typename T, int VS>
__device__ __forceinline__ Macro<T> macro_from(const Mom<T> &M, int maxit, T tol) {
  Macro<T> r;
  T vx, vy;
  bool ok;
  if constexpr (sizeof(T) == 8) {
    ok = landau_refined<VS>(M, vx, vy);
    if (!ok) ok = landau<T, VS>(M, maxit, tol, vx, vy);
  } else {
    ok = landau<T, VS>(M, maxit, tol, vx, vy);
  }
  const T v2 = vx * vx + vy * vy;
  const T gam = FM<T>::rsqrt(T(1) - v2);
  r.eps_m1 = M.e - (M.mx * vx + M.my * vy);
  r.u0 = gam; r.ux = gam * vx; r.uy = gam * vy; r.vx = vx; r.vy = vy;
  r.ok = ok && (T(1) + r.eps_m1 > T(0)) && isfinite(r.eps_m1) && isfinite(gam);
  return r;
}

// Landau matching of one cell in the compute type; the FP32 path re-solves in FP64
// (moments re-summed in FP64 from the same h) when its two Newton steps have not
// converged or |v|^2 exceeds vmax2.
template <typename R, int VS>
__device__ __forceinline__ Macro<R> cell_macro(const R h[VSet<VS>::Q], const Mom<R> &M, R vmax2) {
  if constexpr (sizeof(R) == 8) {
    return macro_from<double, VS>(M, 40, 1e-12);
  } else {
    Macro<float> m = macro_from<float, VS>(M, 4, 3e-4f);
    if (!m.ok || m.vx * m.vx + m.vy * m.vy > vmax2) {
      const Mom<double> Md = moments_of<double, R, VS, false>(h);
      const Macro<double> d = macro_from<double, VS>(Md, 40, 1e-12);
      m.eps_m1 = (float)d.eps_m1; m.u0 = (float)d.u0; m.ux = (float)d.ux; m.uy = (float)d.uy;
      m.vx = (float)d.vx; m.vy = (float)d.vy; m.ok = d.ok;
    }
    return m;
  }
}

// Landau matching of two cells at once: the Newton steps of `landau` on both lanes, each
// lane keeping its value from the step at which it converged (so a cell's result does not
// depend on the cell it is paired with); a lane that has not converged, or whose |v|^2
// exceeds vmax2, is re-solved in FP64 from the same populations.
template <int VS>
__device__ __forceinline__ Macro<F2> cell_macro_pair(const F2 h[VSet<VS>::Q], const Mom<F2> &M, float vmax2) {
  constexpr float dinv = 1.0f / VSet<VS>::DP;
  const float tol = 3e-4f;
  const F2 one(1.0f);
  const F2 T00 = one + M.e;
  const F2 i00 = FM<F2>::rcp(T00);
  const F2 ax = M.mx * i00, ay = M.my * i00, m2 = fma(ax, ax, ay * ay);
  F2 c;
  if (VS == 3) c = F2(3.0f) * FM<F2>::rcp(F2(2.0f) + FM<F2>::sqrt_(fmax(fma(F2(-3.0f), m2, F2(4.0f)), F2(0.0f))));
  else c = F2(4.0f) * FM<F2>::rcp(F2(3.0f) + FM<F2>::sqrt_(fmax(fma(F2(-8.0f), m2, F2(9.0f)), F2(0.0f))));
  F2 vx = c * ax, vy = c * ay;
  // -T^{ab} and -T^00: the residual and its Jacobian then take one multiply-add per term
  const F2 nxx = fma(M.txx, F2(-1.0f), F2(-dinv)), nxy = -M.txy, nyy = fma(M.tyy, F2(-1.0f), F2(-dinv));
  const F2 n00 = -T00;
  bool convA = false, convB = false;
  for (int it = 0; it < 4; ++it) {
    const F2 nE = fma(M.mx, vx, fma(M.my, vy, n00));  // -(T^00 - m.v)
    const F2 bx = nxx + nE, by = nyy + nE;
    const F2 rx = fma(bx, vx, fma(nxy, vy, M.mx)), ry = fma(by, vy, fma(nxy, vx, M.my));
    const F2 jxx = fma(vx, M.mx, bx), jxy = fma(vx, M.my, nxy);
    const F2 jyx = fma(vy, M.mx, nxy), jyy = fma(vy, M.my, by);
    const F2 idet = FM<F2>::rcp(jxx * jyy - jxy * jyx);
    const F2 dx = (jxy * ry - jyy * rx) * idet;
    const F2 dy = (jyx * rx - jxx * ry) * idet;
    vx += F2(convA ? 0.0f : dx.v.x, convB ? 0.0f : dx.v.y);
    vy += F2(convA ? 0.0f : dy.v.x, convB ? 0.0f : dy.v.y);
    const F2 d2 = fma(dx, dx, dy * dy), lim = fma(F2(tol * tol), fma(vx, vx, vy * vy), F2(tol * tol * 1e-6f));
    convA = convA || d2.v.x <= lim.v.x;
    convB = convB || d2.v.y <= lim.v.y;
    if (convA && convB) break;
  }
  const F2 v2 = fma(vx, vx, vy * vy), mv = fma(M.mx, vx, M.my * vy);
  const F2 E = T00 - mv;
  const bool okA = convA && v2.v.x < vmax2 && E.v.x > 0.0f, okB = convB && v2.v.y < vmax2 && E.v.y > 0.0f;
  Macro<F2> r;
  const F2 gam = FM<F2>::rsqrt(one - v2);
  r.eps_m1 = M.e - mv;
  r.u0 = gam; r.ux = gam * vx; r.uy = gam * vy; r.vx = vx; r.vy = vy;
  r.ok = true;
  if (!okA || !okB) {
    for (int lane = 0; lane < 2; ++lane) {
      if (lane == 0 ? okA : okB) continue;
      float hl[VSet<VS>::Q];
#pragma unroll
      for (int q = 0; q < VSet<VS>::Q; ++q) hl[q] = lane == 0 ? h[q].v.x : h[q].v.y;
      const Mom<double> Md = moments_of<double, float, VS, false>(hl);
      const Macro<double> d = macro_from<double, VS>(Md, 40, 1e-12);
      float *dst[6] = {lane ? &r.eps_m1.v.y : &r.eps_m1.v.x, lane ? &r.u0.v.y : &r.u0.v.x,
                       lane ? &r.ux.v.y : &r.ux.v.x, lane ? &r.uy.v.y : &r.uy.v.x,
                       lane ? &r.vx.v.y : &r.vx.v.x, lane ? &r.vy.v.y : &r.vy.v.x};
      *dst[0] = (float)d.eps_m1; *dst[1] = (float)d.u0; *dst[2] = (float)d.ux;
      *dst[3] = (float)d.uy; *dst[4] = (float)d.vx; *dst[5] = (float)d.vy;
      r.ok = r.ok && d.ok;
    }
  }
  r.ok = r.ok && isfinite(r.eps_m1.v.x) && isfinite(r.eps_m1.v.y) && (1.0f + r.eps_m1.v.x > 0.0f) &&
         (1.0f + r.eps_m1.v.y > 0.0f);
  return r;
}

// ---------------------------------------------------------------------------
// Collision and force of one cell, as per-class polynomials in v_i:
//   h*_i = h_i + omega (u^0 - u.v_i)(h_eq,i - h_i) + dt S_i / (w_i eps0)
//   h_eq,i = (eps^ - 1) + CA eps^ u^0 (u.v_i) + CB eps^ (u.v_i)^2 - CC eps^ |u|^2
// (the equilibrium of Eq. rel_pdf_exp_coef with T_eq = (eps + P) u u - P g), so with
// t = u.v_i:  h*_i = h_i (1 - omega u^0 + omega t) + p0 + p1 t + p2 t^2 + p3 t^3 + S_i.
// The force (Eq. forceTerm with App. B's coefficients, prefactor -6/T0 dt):
//   S_i = fpref [ F.M1 / 4 - (M0 / 2) F.v_i + 5/4 v_i.B.v_i - 5/2 (F.v_i)(v_i.M1) ]
//       = s0 + s1.v_i + v_i.S2.v_i + szz v_z,i^2
// with B_ab = sum f (F.v) v_a v_b and B_zz = F.M1 - B_xx - B_yy (|v| = 1).
// ---------------------------------------------------------------------------
template <typename R> struct Coll {
  R ux, uy, k0, om, p0, p1, p2, p3;
  R s0, s1x, s1y, sxx, sxy2, syy, szz;
};

// one: the scale of the collision's output (the stored form's HScale::up, with omega0 and
// fpref passed already multiplied by it; every coefficient below is then scaled by it too).
template <typename R, int VS, bool FORCE>
__device__ __forceinline__ Coll<R> coll_coeffs(const Mom<R> &M, const Macro<R> &m, R omega0, R fpref, R Fx, R Fy,
                                               R one = R(1)) {
  using V = VSet<VS>;
  Coll<R> c;
  const R epsh = R(1) + m.eps_m1;
  const R om = VS == 3 ? omega0 * FM<R>::qroot(epsh) : omega0 * FM<R>::croot(epsh);
  const R u2 = fma(m.ux, m.ux, m.uy * m.uy);
  const R ca = R(V::CA) * epsh * m.u0, cb = R(V::CB) * epsh, cc = fma(R(-V::CC) * epsh, u2, m.eps_m1);
  const R omu = om * m.u0;
  c.ux = m.ux; c.uy = m.uy; c.om = om;
  c.k0 = one - omu;
  c.p0 = omu * cc;
  c.p1 = om * fma(m.u0, ca, -cc);
  c.p2 = om * fma(m.u0, cb, -ca);
  c.p3 = R(-V::CB) * om * epsh;
  c.s0 = c.s1x = c.s1y = c.sxx = c.sxy2 = c.syy = c.szz = R(0);
  if (FORCE) {
    const R FM1 = fma(Fx, M.mx, Fy * M.my), M0 = R(1) + M.e;
    const R Bxx = fma(Fx, M.wxxx, Fy * M.wxxy);
    const R Bxy = fma(Fx, M.wxxy, Fy * M.wxyy);
    const R Byy = fma(Fx, M.wxyy, Fy * M.wyyy);
    const R Bzz = FM1 - Bxx - Byy;
    const R f54 = R(1.25) * fpref, h = R(-0.5) * fpref * M0;
    const R Fx2 = R(-2) * Fx, Fy2 = R(-2) * Fy;
    c.s0 = R(0.25) * fpref * FM1;
    c.s1x = h * Fx;
    c.s1y = h * Fy;
    c.sxx = f54 * fma(Fx2, M.mx, Bxx);
    c.sxy2 = f54 * fma(Fx2, M.my, fma(Fy2, M.mx, R(2) * Bxy));
    c.syy = f54 * fma(Fy2, M.my, Byy);
    c.szz = f54 * Bzz;
  }
  c.s0 += c.p0;
  return c;
}

template <typename R, int VS, bool FORCE>
__device__ __forceinline__ R collide_class(const Coll<R> &c, int q, R h) {
  using V = VSet<VS>;
  const double vx = V::vx(q), vy = V::vy(q), vz2 = V::vz2(q);
  R t = R(0);
  if (vx != 0.0) t = c.ux * R(vx);
  if (vy != 0.0) t = fma(c.uy, R(vy), t);
  R acc = c.s0;
  if (FORCE) {
    if (vx != 0.0) acc = fma(c.s1x, R(vx), acc);
    if (vy != 0.0) acc = fma(c.s1y, R(vy), acc);
    if (vx != 0.0) acc = fma(c.sxx, R(vx * vx), acc);
    if (vx != 0.0 && vy != 0.0) acc = fma(c.sxy2, R(vx * vy), acc);
    if (vy != 0.0) acc = fma(c.syy, R(vy * vy), acc);
    if (vz2 != 0.0) acc = fma(c.szz, R(vz2), acc);
  }
  if (vx != 0.0 || vy != 0.0) acc = fma(t, fma(t, fma(t, c.p3, c.p2), c.p1), acc);
  const R k = (vx != 0.0 || vy != 0.0) ? fma(c.om, t, c.k0) : c.k0;
  return fma(h, k, acc);
}

// Two opposite classes at once, t = u.v of the first: the polynomial's even part (with the
// force's even part e) and odd part (with the force's odd part x) are formed once.
template <typename R>
__device__ __forceinline__ void collide_opposite(const Coll<R> &c, R t, R e, R x, R hp, R hm, R &op, R &om) {
  const R t2 = t * t, ot = c.om * t;
  const R even = fma(t2, c.p2, e), odd = fma(t, fma(t2, c.p3, c.p1), x);
  op = fma(hp, c.k0 + ot, even + odd);
  om = fma(hm, c.k0 - ot, even - odd);
}

// The classes of a sign group {(+a,+b), (-a,+b), (-a,-b), (+a,-b)} share a u-projection pair
// (a u^x, b u^y) and the even part of the force polynomial; only signs differ between them.
template <typename R, bool FORCE>
__device__ __forceinline__ void collide_group(const Coll<R> &c, double a, double b, double vz2, R h0, R h1, R h2,
                                              R h3, R &o0, R &o1, R &o2, R &o3) {
  if (b != 0.0) {  // diagonal group: (+a,+b), (-a,+b), (-a,-b), (+a,-b)
    const R A = c.ux * R(a), B = c.uy * R(b);
    R even = c.s0, X = R(0), Y = R(0), e0 = c.s0, e1 = c.s0;
    if (FORCE) {
      even = fma(c.syy, R(b * b), fma(c.sxx, R(a * a), even));
      if (vz2 != 0.0) even = fma(c.szz, R(vz2), even);
      X = c.s1x * R(a);
      Y = c.s1y * R(b);
      e0 = fma(c.sxy2, R(a * b), even);
      e1 = fma(c.sxy2, R(-a * b), even);
    }
    collide_opposite<R>(c, A + B, e0, X + Y, h0, h2, o0, o2);
    collide_opposite<R>(c, B - A, e1, Y - X, h1, h3, o1, o3);
  } else {  // axis group: (+a,0), (0,+a), (-a,0), (0,-a)
    R ex = c.s0, ey = c.s0, X = R(0), Y = R(0);
    if (FORCE) {
      const R ez = vz2 != 0.0 ? fma(c.szz, R(vz2), c.s0) : c.s0;
      ex = fma(c.sxx, R(a * a), ez);
      ey = fma(c.syy, R(a * a), ez);
      X = c.s1x * R(a);
      Y = c.s1y * R(a);
    }
    collide_opposite<R>(c, c.ux * R(a), ex, X, h0, h2, o0, o2);
    collide_opposite<R>(c, c.uy * R(a), ey, Y, h1, h3, o1, o3);
  }
}

template <typename R, int VS, bool FORCE>
__device__ __forceinline__ void collide_all(const Coll<R> &c, const R h[VSet<VS>::Q], R hn[VSet<VS>::Q]) {
  if constexpr (VS == 3) {
    // class 0: v = (0, 0), v_z^2 = 1
    hn[0] = fma(h[0], c.k0, FORCE ? fma(c.szz, R(1), c.s0) : c.s0);
    collide_group<R, FORCE>(c, 1.0, 0.0, 0.0, h[1], h[2], h[3], h[4], hn[1], hn[2], hn[3], hn[4]);
    collide_group<R, FORCE>(c, RLBM_S2, RLBM_S2, 0.0, h[5], h[6], h[7], h[8], hn[5], hn[6], hn[7], hn[8]);
    collide_group<R, FORCE>(c, RLBM_S2, 0.0, 0.5, h[9], h[10], h[11], h[12], hn[9], hn[10], hn[11], hn[12]);
    collide_group<R, FORCE>(c, RLBM_S3, RLBM_S3, 1.0 / 3.0, h[13], h[14], h[15], h[16], hn[13], hn[14], hn[15], hn[16]);
  } else {
#pragma unroll
    for (int q = 0; q < VSet<VS>::Q; ++q) hn[q] = collide_class<R, VS, FORCE>(c, q, h[q]);
  }
}

}  // namespace rlbm
