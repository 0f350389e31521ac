// Reductions and the energy spectrum of the velocity field.
//
// Spectrum (Sec. "Turbulence": E(k) is the shell density of 1/2 |v(k)|^2): with
// z = v_x + i v_y, |V_x(k)|^2 + |V_y(k)|^2 = (|Z(k)|^2 + |Z(-k)|^2) / 2, and every shell
// round(|k|) = n is closed under k -> -k, so the shell sum of |V_x|^2 + |V_y|^2 equals the
// shell sum of |Z|^2: one complex 2-D transform serves both components.  The
// transform is a mixed-radix Stockham FFT (radices 2-8 in registers, any larger prime
// factor as a direct DFT stage): rows in shared memory, then strips of columns in shared
// memory with the binning in the same kernel; lengths whose buffers do not fit there run in
// global memory with a transpose between.  It runs in FP64 on FP64 velocities and in pairs
// of FP32 numbers (48 bits) on those of FP32 states: GB300's FP64 units, at 1/64 of FP32's
// rate, took 78 us for the rows and 138 us for the columns of a 1024^2 field.
#include "rlbm_device.cuh"
#include "rlbm_launch.h"
#include "rlbm_tma.cuh"

namespace rlbm {

// ---------------------------------------------------------------------------
// Deterministic sum of per-block partials: thread t takes term t mod 4 of the blocks t / 4,
// t / 4 + 256, ... in order; a tree of fixed shape adds the threads.  (Thread 0 adding 256
// thread sums one after the other took 12 us of a launch that now takes 3.)
// ---------------------------------------------------------------------------
__global__ void reduce_partials_kernel(const double *__restrict__ partials, long long nblocks,
                                       double *__restrict__ totals) {
  __shared__ double s[32][4];
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  double v = 0.0;
#pragma unroll 4
  for (long long i = t >> 2; i < nblocks; i += 256) v += partials[i * 4 + (t & 3)];
  for (int off = 16; off >= 4; off >>= 1) v += __shfl_down_sync(0xffffffffu, v, off);
  if (lane < 4) s[warp][lane] = v;
  __syncthreads();
  if (warp != 0) return;
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    double w = s[lane][k];
    for (int off = 16; off > 0; off >>= 1) w += __shfl_down_sync(0xffffffffu, w, off);
    if (lane == 0) totals[k] = w;
  }
}

__global__ void counter_inc_kernel(long long *c, int *tile_ctr) {
  *c += 1;
  *tile_ctr = 0;
}

// Advances the batch step counter between two batched step launches (stream order) and
// clears the tile counter for the next launch.
cudaError_t launch_counter_inc(long long *counter, int *tile_ctr, cudaStream_t st) {
  counter_inc_kernel<<<1, 1, 0, st>>>(counter, tile_ctr);
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Self-test of the failure path of the bounded waits: one thread waits on an mbarrier that
// nothing arrives on, with the bounded wait the step kernels use on their TMA copies; when
// it runs out after max_cycles SM clocks the timeout is latched in the error word, as a
// step kernel does.  No copy is in flight, so the thread returns at once.
// ---------------------------------------------------------------------------
__global__ void wait_selftest_kernel(unsigned *err, long long max_cycles) {
  __shared__ alignas(8) uint64_t bar;
  if (threadIdx.x != 0) return;
  mbar_init(&bar, 1);
  fence_mbar_init();
  if (!mbar_wait_bounded(&bar, 0, max_cycles)) atomicOr(err, ERR_TIMEOUT);
}

cudaError_t launch_wait_selftest(unsigned *err, long long max_cycles, cudaStream_t st) {
  wait_selftest_kernel<<<1, 32, 0, st>>>(err, max_cycles);
  return cudaGetLastError();
}

// Halo rows of a strip: block p copies the padded row of plane p between the population
// buffer and the message buffer, 16 bytes per thread and step (rows start on 128-byte lines
// of the buffer; the message buffer is 16-byte aligned).
__global__ void halo_copy_kernel(char *__restrict__ pop, const HaloRows rows, long long row_bytes,
                                 char *__restrict__ buf, bool pack) {
  const int p = blockIdx.x;
  uint4 *a = reinterpret_cast<uint4 *>(pop + rows.off[p]);
  uint4 *b = reinterpret_cast<uint4 *>(buf + p * row_bytes);
  const long long n = row_bytes / 16;
  for (long long i = threadIdx.x; i < n; i += blockDim.x) {
    if (pack) b[i] = a[i];
    else a[i] = b[i];
  }
}

cudaError_t launch_halo_copy(char *pop, const HaloRows &rows, long long row_bytes, char *buf, bool pack,
                             cudaStream_t st) {
  if (rows.nplanes < 1) return cudaSuccess;
  halo_copy_kernel<<<rows.nplanes, 256, 0, st>>>(pop, rows, row_bytes, buf, pack);
  return cudaGetLastError();
}

cudaError_t launch_reduce_partials(const double *partials, long long nblocks, double *totals, cudaStream_t st) {
  reduce_partials_kernel<<<1, 1024, 0, st>>>(partials, nblocks, totals);
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// FFT
// ---------------------------------------------------------------------------
struct FftPlan {
  int n, nstages;
  int radix[40];
};

static FftPlan make_plan(int n) {
  FftPlan p;
  p.n = n;
  p.nstages = 0;
  int m = n;
  const int pref[] = {8, 4, 2, 3, 5, 7};
  for (int r : pref)
    while (m % r == 0 && (r != 8 || m % 8 == 0)) { p.radix[p.nstages++] = r; m /= r; }
  for (int f = 11; m > 1; f += 2)
    while (m % f == 0) { p.radix[p.nstages++] = f; m /= f; }
  return p;
}

// A complex number in FP64 (Cd) or in pairs of FP32 numbers (Cf: real part in the first lane);
// 16 bytes either way.
struct alignas(16) Cd {
  double x, y;
};
struct alignas(16) Cf {
  float4 v;  // high re, im, low re, im
};
__device__ __forceinline__ DF2 df_of(const Cf &a) { return DF2{F2(a.v.x, a.v.y), F2(a.v.z, a.v.w)}; }
__device__ __forceinline__ Cf cf_of(const DF2 &d) { return Cf{make_float4(d.h.v.x, d.h.v.y, d.l.v.x, d.l.v.y)}; }

__device__ __forceinline__ Cd ldg(const Cd *p) {
  const double2 v = __ldg(reinterpret_cast<const double2 *>(p));
  return Cd{v.x, v.y};
}
__device__ __forceinline__ Cf ldg(const Cf *p) { return Cf{__ldg(reinterpret_cast<const float4 *>(p))}; }
__device__ __forceinline__ Cd cadd(Cd a, Cd b) { return Cd{a.x + b.x, a.y + b.y}; }
__device__ __forceinline__ Cd csub(Cd a, Cd b) { return Cd{a.x - b.x, a.y - b.y}; }
__device__ __forceinline__ Cd cmul(Cd a, Cd b) { return Cd{a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x}; }
__device__ __forceinline__ Cd cmul_mi(Cd a) { return Cd{a.y, -a.x}; }  // times -i
__device__ __forceinline__ Cd cscale_s2(Cd a) { return Cd{RLBM_S2 * a.x, RLBM_S2 * a.y}; }
__device__ __forceinline__ Cf cadd(Cf a, Cf b) { return cf_of(df_add(df_of(a), df_of(b))); }
__device__ __forceinline__ Cf csub(Cf a, Cf b) { return cf_of(df_add(df_of(a), df_neg(df_of(b)))); }
__device__ __forceinline__ Cf cmul(Cf a, Cf b) {
  const DF2 A = df_of(a);
  const DF2 S{F2(-a.v.y, a.v.x), F2(-a.v.w, a.v.z)};  // i a
  return cf_of(df_add(df_mul(A, DF2{F2(b.v.x), F2(b.v.z)}), df_mul(S, DF2{F2(b.v.y), F2(b.v.w)})));
}
__device__ __forceinline__ Cf cmul_mi(Cf a) { return Cf{make_float4(a.v.y, -a.v.x, a.v.w, -a.v.z)}; }
__device__ __forceinline__ Cf cscale_s2(Cf a) {
  constexpr float hi = (float)RLBM_S2, lo = (float)(RLBM_S2 - (double)hi);
  return cf_of(df_mul(df_of(a), DF2{F2(hi), F2(lo)}));
}
template <class C> __device__ __forceinline__ C czero();
template <> __device__ __forceinline__ Cd czero<Cd>() { return Cd{0.0, 0.0}; }
template <> __device__ __forceinline__ Cf czero<Cf>() { return Cf{make_float4(0.0f, 0.0f, 0.0f, 0.0f)}; }
// Sums of squared moduli: FP64, or the real and imaginary squares in the lanes of a pair.
struct SumD {
  double v = 0.0;
  __device__ __forceinline__ void add(Cd z) { v += z.x * z.x + z.y * z.y; }
  __device__ __forceinline__ double value() const { return v; }
};
// (The square of a pair has its 48 bits in FP32's range from |z| = 2^-50 on, while FP32 velocities reach
// down to 1e-38: pairs are transformed scaled by spectrum_scale.)
struct SumF {
  DF2 v{F2(0.0f), F2(0.0f)};
  __device__ __forceinline__ void add(Cf z) { const DF2 d = df_of(z); v = df_add(v, df_mul(d, d)); }
  __device__ __forceinline__ double value() const {
    return ((double)v.h.v.x + (double)v.h.v.y) + ((double)v.l.v.x + (double)v.l.v.y);
  }
};
template <class C> struct SumOf;
template <> struct SumOf<Cd> { using type = SumD; };
template <> struct SumOf<Cf> { using type = SumF; };

// Forward DFTs of length 4 and 8 in place: two levels of sums and differences (W_4 = -i is an
// exchange of the parts), and 8 = two length-4 transforms of the even and odd inputs joined
// by W_8^k = ((1 - i) / sqrt 2)^k.
template <class C> __device__ __forceinline__ void dft4(C &v0, C &v1, C &v2, C &v3) {
  const C a0 = cadd(v0, v2), a1 = csub(v0, v2), a2 = cadd(v1, v3), a3 = cmul_mi(csub(v1, v3));
  v0 = cadd(a0, a2);
  v1 = cadd(a1, a3);
  v2 = csub(a0, a2);
  v3 = csub(a1, a3);
}
template <class C> __device__ __forceinline__ void dft8(C v[8]) {
  dft4(v[0], v[2], v[4], v[6]);  // even part X_0..X_3 in v[0], v[2], v[4], v[6]
  dft4(v[1], v[3], v[5], v[7]);
  const C o1 = cscale_s2(cadd(v[3], cmul_mi(v[3])));            // (1 - i) / sqrt 2
  const C o2 = cmul_mi(v[5]);
  const C o3 = cscale_s2(csub(cmul_mi(v[7]), v[7]));            // (-1 - i) / sqrt 2
  const C e0 = v[0], e1 = v[2], e2 = v[4], e3 = v[6], o0 = v[1];
  v[0] = cadd(e0, o0); v[4] = csub(e0, o0);
  v[1] = cadd(e1, o1); v[5] = csub(e1, o1);
  v[2] = cadd(e2, o2); v[6] = csub(e2, o2);
  v[3] = cadd(e3, o3); v[7] = csub(e3, o3);
}

// w / n and w mod n; a shift and a mask for powers of two (n is the same for all threads, and
// the integer division was a fifth of a stage's instructions).
__device__ __forceinline__ int2 div_mod(int w, int n) {
  if ((n & (n - 1)) == 0) return make_int2(w >> (__ffs(n) - 1), w & (n - 1));
  const int q = w / n;
  return make_int2(q, w - q * n);
}

// One Stockham stage of `count` transforms of length n, by all threads of a block: transform c
// from src + c * stride to dst + c * stride, element i at place P(i).  tw[t] = exp(-2 pi i t / n).
// Stage with radix R after radices of product Ns:
//   v_r = x[j + r n/R] * w^(r (j mod Ns) n/(Ns R)),  y[(j div Ns) Ns R + (j mod Ns) + k Ns] = DFT_R(v)_k.
// Radices 2, 4 and 8 use their butterflies; the others evaluate the length-R sums directly
// (O(n R) work for the stage; a prime factor above 8 shares its outputs over the threads).
template <class C, class P>
__device__ __forceinline__ void fft_stage(const C *src, C *dst, int count, int stride, int n, int R, int Ns,
                                          const C *__restrict__ tw, P place) {
  const int nR = n / R;
  const int ts = n / (Ns * R);
  if (R > 8) {
    for (int w = threadIdx.x; w < count * n; w += blockDim.x) {
      const int c = w / n, t = w - c * n;
      const C *s = src + c * stride;
      const int j = t / R, k = t - j * R;
      const int jm = j % Ns;
      const int base = (j / Ns) * Ns * R + jm;
      C acc = czero<C>();
      for (int r = 0; r < R; ++r) {
        const C v = cmul(s[place(j + r * nR)], ldg(&tw[r * jm * ts]));
        acc = cadd(acc, cmul(v, ldg(&tw[((r * k) % R) * nR])));
      }
      dst[c * stride + place(base + k * Ns)] = acc;
    }
    return;
  }
  for (int w = threadIdx.x; w < count * nR; w += blockDim.x) {
    const int2 cj = div_mod(w, nR);
    const int c = cj.x, j = cj.y;
    const C *s = src + c * stride;
    C *d = dst + c * stride;
    const int2 js = div_mod(j, Ns);
    const int jm = js.y;
    const int base = js.x * Ns * R + jm;
    C v[8];
    auto load = [&](int r) {
      const C a = s[place(j + r * nR)];
      return (r == 0 || Ns == 1) ? a : cmul(a, ldg(&tw[r * jm * ts]));  // r jm ts < n
    };
    if (R == 8) {
#pragma unroll
      for (int r = 0; r < 8; ++r) v[r] = load(r);
      dft8(v);
#pragma unroll
      for (int k = 0; k < 8; ++k) d[place(base + k * Ns)] = v[k];
    } else if (R == 4) {
#pragma unroll
      for (int r = 0; r < 4; ++r) v[r] = load(r);
      dft4(v[0], v[1], v[2], v[3]);
#pragma unroll
      for (int k = 0; k < 4; ++k) d[place(base + k * Ns)] = v[k];
    } else if (R == 2) {
      const C a = load(0), b = load(1);
      d[place(base)] = cadd(a, b);
      d[place(base + Ns)] = csub(a, b);
    } else {  // radix 3, 5 or 7: the length-R sums
#pragma unroll
      for (int r = 0; r < 7; ++r)
        if (r < R) v[r] = load(r);
      for (int k = 0; k < R; ++k) {
        C acc = v[0];
#pragma unroll
        for (int r = 1; r < 7; ++r)
          if (r < R) acc = cadd(acc, cmul(v[r], ldg(&tw[((r * k) % R) * nR])));
        d[place(base + k * Ns)] = acc;
      }
    }
  }
}

// Rows too long for shared memory: one block transforms one row in global memory (ping-pong
// between a and b).
template <class C> __global__ void fft_rows_kernel(C *a, C *b, const C *__restrict__ tw, FftPlan plan) {
  C *src = a + (long long)blockIdx.x * plan.n, *dst = b + (long long)blockIdx.x * plan.n;
  int Ns = 1;
  for (int s = 0; s < plan.nstages; ++s) {
    fft_stage(src, dst, 1, plan.n, plan.n, plan.radix[s], Ns, tw, [](int i) { return i; });
    __syncthreads();
    C *tmp = src; src = dst; dst = tmp;
    Ns *= plan.radix[s];
  }
}

// Transforms in shared memory.  Element i of a row lies at i + i / 8: the stages write at
// strides of the product of the radices so far, a power of two as a rule, and the gap of one
// element in eight spreads those over the banks.
__device__ __forceinline__ int fft_place(int i) { return i + (i >> 3); }
static int fft_padded(int n) { return n + (n >> 3) + 1; }
constexpr int FFT_SMEM = 226 * 1024;  // (1 KB left for static shared memory)

template <typename K> static cudaError_t fft_allow_smem(K kern, int bytes) {
  if (bytes <= 48 * 1024) return cudaSuccess;
  return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, FFT_SMEM);
}

// The row transforms: one block per row, in place in global memory, all stages in shared
// memory.  Through global memory the stages of a 512-point row took 26 us for 512 rows, by
// the latency of the write and read between two stages; here the reads and writes of a row
// are one pass each, and FP64 arithmetic (1/64 of FP32's rate) bounds long rows.
template <class C>
__global__ void __launch_bounds__(512) fft_rows_smem_kernel(C *z, const C *__restrict__ tw, FftPlan plan, int padded) {
  extern __shared__ __align__(16) unsigned char fft_sm[];
  C *src = reinterpret_cast<C *>(fft_sm), *dst = src + padded;
  C *row = z + (long long)blockIdx.x * plan.n;
  for (int i = threadIdx.x; i < plan.n; i += blockDim.x) src[fft_place(i)] = row[i];
  __syncthreads();
  int Ns = 1;
  for (int s = 0; s < plan.nstages; ++s) {
    fft_stage(src, dst, 1, padded, plan.n, plan.radix[s], Ns, tw, fft_place);
    __syncthreads();
    C *tmp = src; src = dst; dst = tmp;
    Ns *= plan.radix[s];
  }
  for (int i = threadIdx.x; i < plan.n; i += blockDim.x) row[i] = src[fft_place(i)];
}

// The shell of an integer squared wave number: round(sqrt(k2)), from the single-precision
// root corrected with integers ((n - 1/2)^2 < k2 < (n + 1/2)^2 reads n^2 - n < k2 <= n^2 + n).
__device__ __forceinline__ int shell_of(int k2) {
  int n = __float2int_rn(sqrtf((float)k2));
  while (k2 > n * n + n) ++n;
  while (n > 0 && k2 <= n * n - n) --n;
  return n;
}
// The largest integer whose square does not exceed v >= 0.
__device__ __forceinline__ int isqrt(int v) {
  int r = (int)sqrtf((float)v);
  while (r * r > v) --r;
  while ((r + 1) * (r + 1) <= v) ++r;
  return r;
}

// The column transforms of `ncol` adjacent columns (k_x indices) per block, and what is
// summed of them: the spectrum's shells (BINS) or a band's energy.  Z is [y][x] after the row
// transforms; a strip is read in pieces of ncol * 16 bytes.  A thread takes shells of the
// strip, not elements: the k_y of one shell and column are a run of neighbours, so the strip
// adds one value per shell to the global bins (one FP64 atomic per element cost 16 us at
// 512^2).  The transposes and the write and read of the transformed field are gone too.
template <class C, bool BINS>
__global__ void __launch_bounds__(512)
fft_cols_kernel(const C *__restrict__ Z, int nx, int ny, const C *__restrict__ tw, FftPlan plan, int padded, int ncol,
                double scale, double *__restrict__ bins, int nbins, long long k2lo, long long k2hi,
                double *__restrict__ partials, double *__restrict__ out4, unsigned *__restrict__ sync) {
  using Sum = typename SumOf<C>::type;
  extern __shared__ __align__(16) unsigned char fft_sm[];
  C *src = reinterpret_cast<C *>(fft_sm), *dst = src + ncol * padded;
  const int x0 = blockIdx.x * ncol, nc = min(ncol, nx - x0);
  for (int i = threadIdx.x; i < ncol * ny; i += blockDim.x) {
    const int y = i / ncol, c = i - y * ncol;
    if (c < nc) src[c * padded + fft_place(y)] = Z[(long long)y * nx + x0 + c];
  }
  __syncthreads();
  int Ns = 1;
  for (int s = 0; s < plan.nstages; ++s) {
    fft_stage(src, dst, nc, padded, ny, plan.radix[s], Ns, tw, fft_place);
    __syncthreads();
    C *tmp = src; src = dst; dst = tmp;
    Ns *= plan.radix[s];
  }
  const int top = (ny + 1) / 2;  // k_y = 0 .. top - 1, then the negative ones
  auto energy = [&](Sum &acc, int c, int ky) {  // |Z|^2 at k_y and, where the lattice has it, -k_y
    if (ky < top) acc.add(src[c * padded + fft_place(ky)]);
    if (ky > 0 && ky <= ny - top) acc.add(src[c * padded + fft_place(ny - ky)]);
  };
  if (BINS) {
    for (int n = threadIdx.x; n < nbins; n += blockDim.x) {
      Sum acc;
      for (int c = 0; c < nc; ++c) {
        const int qx = x0 + c, kx = qx < (nx + 1) / 2 ? qx : nx - qx;  // |k_x|
        const int hi2 = n * n + n - kx * kx, lo2 = n * n - n - kx * kx;  // lo2 < k_y^2 <= hi2
        if (hi2 < 0) continue;
        const int hi = min(isqrt(hi2), ny / 2);
        for (int ky = lo2 < 0 || n == 0 ? 0 : isqrt(lo2) + 1; ky <= hi; ++ky) energy(acc, c, ky);
      }
      const double v = acc.value();
      if (v != 0.0) atomicAdd(&bins[n], scale * v);
    }
  } else {
    Sum sum_t;
    for (int i = threadIdx.x; i < nc * (ny / 2 + 1); i += blockDim.x) {
      const int c = i / (ny / 2 + 1), ky = i - c * (ny / 2 + 1);
      const long long qx = x0 + c, kx = qx < (nx + 1) / 2 ? qx : nx - qx;
      const long long k2 = kx * kx + (long long)ky * ky;
      if (k2 < k2lo || (k2hi > 0 && k2 >= k2hi)) continue;
      energy(sum_t, c, ky);
    }
    double acc = sum_t.value();
    __shared__ double red[32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int off = 16; off > 0; off >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, off);
    if (lane == 0) red[warp] = acc;
    __syncthreads();
    // the last block adds the strips' sums in order
    __shared__ bool last;
    if (threadIdx.x == 0) {
      double sum = 0.0;
      for (int w = 0; w < (int)(blockDim.x >> 5); ++w) sum += red[w];
      partials[blockIdx.x] = scale * sum;
      __threadfence();
      last = atomicInc(sync, gridDim.x - 1) == gridDim.x - 1;
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    double v = 0.0;
    for (int i = threadIdx.x; i < (int)gridDim.x; i += blockDim.x) v += __ldcg(&partials[i]);
    for (int off = 16; off > 0; off >>= 1) v += __shfl_down_sync(0xffffffffu, v, off);
    if (lane == 0) red[warp] = v;
    __syncthreads();
    if (threadIdx.x == 0) {
      double sum = 0.0;
      for (int w = 0; w < (int)(blockDim.x >> 5); ++w) sum += red[w];
      out4[0] = sum;
    }
  }
}

__global__ void make_z_kernel(const double *__restrict__ ux, const double *__restrict__ uy, double2 *__restrict__ z,
                              long long ncell) {
  const long long c = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= ncell) return;
  const double a = ux[c], b = uy[c];
  const double u0 = sqrt(1.0 + a * a + b * b);
  z[c] = make_double2(a / u0, b / u0);
}

// out[x * ny + y] = in[y * nx + x]
template <class C> __global__ void transpose_kernel(const C *__restrict__ in, C *__restrict__ out, int nx, int ny) {
  __shared__ C tile[32][33];
  const int x0 = blockIdx.x * 32, y0 = blockIdx.y * 32;
  for (int k = threadIdx.y; k < 32; k += blockDim.y) {
    const int x = x0 + threadIdx.x, y = y0 + k;
    if (x < nx && y < ny) tile[k][threadIdx.x] = in[(long long)y * nx + x];
  }
  __syncthreads();
  for (int k = threadIdx.y; k < 32; k += blockDim.y) {
    const int y = y0 + threadIdx.x, x = x0 + k;
    if (x < nx && y < ny) out[(long long)x * ny + y] = tile[threadIdx.x][k];
  }
}

// Z is transposed: row = k_x index, column = k_y index.  E[round|k|] += 1/2 |Z|^2 / (nx ny)^2.
template <class C>
__global__ void bin_kernel(const C *__restrict__ Z, int nx, int ny, double *__restrict__ bins, int nbins,
                           double scale) {
  extern __shared__ double sb[];
  const bool use_smem = nbins <= 6144;
  if (use_smem)
    for (int i = threadIdx.x; i < nbins; i += blockDim.x) sb[i] = 0.0;
  __syncthreads();
  const int qx = blockIdx.x;
  const int kx = qx < (nx + 1) / 2 ? qx : qx - nx;
  for (int qy = threadIdx.x; qy < ny; qy += blockDim.x) {
    const int ky = qy < (ny + 1) / 2 ? qy : qy - ny;
    const int n = shell_of(kx * kx + ky * ky);
    if (n >= nbins) continue;
    typename SumOf<C>::type a;
    a.add(Z[(long long)qx * ny + qy]);
    const double e = scale * a.value();
    if (use_smem) atomicAdd(&sb[n], e);
    else atomicAdd(&bins[n], e);
  }
  __syncthreads();
  if (use_smem)
    for (int i = threadIdx.x; i < nbins; i += blockDim.x)
      if (sb[i] != 0.0) atomicAdd(&bins[i], sb[i]);
}

cudaError_t launch_make_z(const double *ux, const double *uy, double2 *z, long long ncell, cudaStream_t st) {
  make_z_kernel<<<(unsigned)((ncell + 255) / 256), 256, 0, st>>>(ux, uy, z, ncell);
  return cudaGetLastError();
}

// Whether a prime factor above 8 (the last radix) takes direct sums.
static bool direct_sums(const FftPlan &p) { return p.nstages && p.radix[p.nstages - 1] > 8; }

// Threads of a block that transforms `count` rows: one per radix-8 butterfly, or one per
// output of direct sums.
static int fft_threads(const FftPlan &p, int count) {
  const int work = direct_sums(p) ? p.n : p.n / 8;
  const int t = (work * count + 31) / 32 * 32;
  return t < 32 ? 32 : t > 512 ? 512 : t;
}

// (at least four warps for the loads and the sums over shells)
static int cols_threads(const FftPlan &p, int ncol) { return fft_threads(p, ncol) < 128 ? 128 : fft_threads(p, ncol); }

// Row transforms of z0 (z1: a second buffer for rows too long for shared memory); returns
// the buffer that holds them.
template <class C>
static C *row_transforms(const FftPlan &p, int rows, const C *tw, C *z0, C *z1, cudaStream_t st, cudaError_t &e) {
  const int smem = 2 * fft_padded(p.n) * (int)sizeof(C);
  if (smem <= FFT_SMEM) {
    e = fft_allow_smem(fft_rows_smem_kernel<C>, smem);
    if (e != cudaSuccess) return z0;
    fft_rows_smem_kernel<C><<<rows, fft_threads(p, 1), smem, st>>>(z0, tw, p, fft_padded(p.n));
    return z0;
  }
  fft_rows_kernel<C><<<rows, 256, 0, st>>>(z0, z1, tw, p);
  return (p.nstages % 2) ? z1 : z0;
}

// Columns of a strip: as wide as shared memory and the number of SMs allow, down to two
// columns (32 bytes, a whole sector of each row); 0 = the columns go through a transpose.
// Strips of 4 columns fill the chip from 608 columns on and read 64-byte pieces.  Lengths with a
// prime factor above 8 are bound by the direct sums of that factor, not by the reads: there one
// column to a strip shares the work over the most SMs (FP64, 64 columns of 2039: 22.7 ms in
// strips of two, on 32 SMs).
static int strip_columns(int nx, const FftPlan &py) {
  const int fit = FFT_SMEM / (2 * fft_padded(py.n) * (int)sizeof(Cd));
  if (fit < 2) return 0;
  if (direct_sums(py)) return 1;
  return fit >= 4 && nx >= 4 * 152 ? 4 : 2;
}

// Z = 2-D transform of z0, laid out [k_x][k_y]; returns which of the two work buffers holds it.
template <class C>
static C *velocity_transform(int nx, int ny, const C *twx, const C *twy, C *z0, C *z1, cudaStream_t st, cudaError_t &e) {
  C *r = row_transforms(make_plan(nx), ny, twx, z0, z1, st, e);
  C *o = r == z0 ? z1 : z0;
  transpose_kernel<C><<<dim3((nx + 31) / 32, (ny + 31) / 32), dim3(32, 8), 0, st>>>(r, o, nx, ny);
  return row_transforms(make_plan(ny), nx, twy, o, r, st, e);
}

// Energy of a band of wave vectors, k2lo <= k_x^2 + k_y^2 < k2hi (k2hi <= 0: no upper
// bound): (1/2) sum |V_x|^2 + |V_y|^2 / (nx ny)^2, as the spectrum's bins but with an exact
// integer band edge (the velocity filter that removes the driven range).  One FP64 partial
// per block (k_x column), summed in order afterwards.
template <class C>
__global__ void band_kernel(const C *__restrict__ Z, int nx, int ny, long long k2lo, long long k2hi,
                            double scale, double *__restrict__ partials) {
  const int qx = blockIdx.x;
  const long long kx = qx < (nx + 1) / 2 ? qx : qx - nx;
  double acc = 0.0;
  for (int qy = threadIdx.x; qy < ny; qy += blockDim.x) {
    const long long ky = qy < (ny + 1) / 2 ? qy : qy - ny;
    const long long k2 = kx * kx + ky * ky;
    if (k2 < k2lo || (k2hi > 0 && k2 >= k2hi)) continue;
    typename SumOf<C>::type a;
    a.add(Z[(long long)qx * ny + qy]);
    acc += scale * a.value();
  }
  __shared__ double red[8];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int off = 16; off > 0; off >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, off);
  if (lane == 0) red[warp] = acc;
  __syncthreads();
  if (threadIdx.x == 0) {
    double s = 0.0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) s += red[w];
    partials[(long long)qx * 4] = s;
    partials[(long long)qx * 4 + 1] = partials[(long long)qx * 4 + 2] = partials[(long long)qx * 4 + 3] = 0.0;
  }
}

// 1/2 / (nx ny)^2 of the energies, with the scale of the velocities undone.
template <class C> static double energy_scale(int nx, int ny) {
  const double s = std::is_same<C, Cd>::value ? 1.0 : (double)spectrum_scale((long long)nx * ny);
  return 0.5 / ((double)nx * ny * (double)nx * ny) / (s * s);
}

template <class C>
static cudaError_t band_energy_t(int nx, int ny, const C *twx, const C *twy, C *z0, C *z1, long long k2lo, long long k2hi,
                                 double *partials, double *out4, unsigned *sync, cudaStream_t st) {
  const double scale = energy_scale<C>(nx, ny);
  cudaError_t e = cudaSuccess;
  const FftPlan py = make_plan(ny);
  if (const int nc = strip_columns(nx, py)) {
    const int smem = 2 * nc * fft_padded(ny) * (int)sizeof(C);
    if ((e = fft_allow_smem(fft_cols_kernel<C, false>, smem)) != cudaSuccess) return e;
    C *Z = row_transforms(make_plan(nx), ny, twx, z0, z1, st, e);
    fft_cols_kernel<C, false><<<(nx + nc - 1) / nc, cols_threads(py, nc), smem, st>>>(
        Z, nx, ny, twy, py, fft_padded(ny), nc, scale, nullptr, 0, k2lo, k2hi, partials, out4, sync);
    return e == cudaSuccess ? cudaGetLastError() : e;
  } else {
    C *Z = velocity_transform(nx, ny, twx, twy, z0, z1, st, e);
    band_kernel<C><<<nx, 256, 0, st>>>(Z, nx, ny, k2lo, k2hi, scale, partials);
  }
  if (e == cudaSuccess) e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  return launch_reduce_partials(partials, nx, out4, st);
}

template <class C>
static cudaError_t spectrum_t(int nx, int ny, const C *twx, const C *twy, C *z0, C *z1, double *bins, int nbins,
                              cudaStream_t st) {
  const double scale = energy_scale<C>(nx, ny);
  cudaError_t e = cudaSuccess;
  const FftPlan py = make_plan(ny);
  if (const int nc = strip_columns(nx, py)) {
    const int smem = 2 * nc * fft_padded(ny) * (int)sizeof(C);
    if ((e = fft_allow_smem(fft_cols_kernel<C, true>, smem)) != cudaSuccess) return e;
    C *Z = row_transforms(make_plan(nx), ny, twx, z0, z1, st, e);
    fft_cols_kernel<C, true><<<(nx + nc - 1) / nc, cols_threads(py, nc), smem, st>>>(
        Z, nx, ny, twy, py, fft_padded(ny), nc, scale, bins, nbins, 0, 0, nullptr, nullptr, nullptr);
  } else {
    C *Z = velocity_transform(nx, ny, twx, twy, z0, z1, st, e);
    const size_t smem = nbins <= 6144 ? sizeof(double) * nbins : 0;
    bin_kernel<C><<<nx, 256, smem, st>>>(Z, nx, ny, bins, nbins, scale);
  }
  return e != cudaSuccess ? e : cudaGetLastError();
}

cudaError_t launch_band_energy(bool f64, int nx, int ny, const void *twx, const void *twy, void *z0, void *z1, long long k2lo,
                               long long k2hi, double *partials, double *out4, unsigned *sync, cudaStream_t st) {
  if (f64) return band_energy_t<Cd>(nx, ny, (const Cd *)twx, (const Cd *)twy, (Cd *)z0, (Cd *)z1, k2lo, k2hi, partials, out4, sync, st);
  return band_energy_t<Cf>(nx, ny, (const Cf *)twx, (const Cf *)twy, (Cf *)z0, (Cf *)z1, k2lo, k2hi, partials, out4, sync, st);
}

cudaError_t launch_spectrum(bool f64, int nx, int ny, const void *twx, const void *twy, void *z0, void *z1, double *bins,
                            int nbins, cudaStream_t st) {
  if (f64) return spectrum_t<Cd>(nx, ny, (const Cd *)twx, (const Cd *)twy, (Cd *)z0, (Cd *)z1, bins, nbins, st);
  return spectrum_t<Cf>(nx, ny, (const Cf *)twx, (const Cf *)twy, (Cf *)z0, (Cf *)z1, bins, nbins, st);
}

}  // namespace rlbm
