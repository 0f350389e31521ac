// Host-side launch interface between the C ABI (rlbm_capi.cu) and the kernels of
// each storage type (rlbm_kernels_*.cu).  Plain structs, no templates.
#pragma once

#include <cuda.h>
#include <cuda_runtime.h>
#include <stdint.h>

namespace rlbm {

// Boundary flags of a lattice (Geometry::walls): bit 0 = bounce-back walls in y (the ghost
// rows stay zero), bit 1 = open channel in x (inflow column left of x = 0, written once;
// zero-gradient outflow right of x = nx - 1), bit 2 = a strip of a larger lattice (the
// ghost rows are written by the halo exchange, never by the kernels; which ghost-row cells
// are solid is in the neighbour mask).
constexpr int WALLS_Y = 1, OPEN_X = 2, STRIP_Y = 4;

struct HostGeom {
  int nx, ny, pitch;
  long long plane;         // elements per ghost-padded plane: pitch * (ny + 2)
  int walls;
  const uint16_t *nbmask;  // device; NULL when the lattice has no solid cells or walls
  double beta[17][4];
};

struct HostPhys {
  double omega0, fpref, body_x, body_y, vmax2;
  int has_force;
  int stochastic;          // 16-bit storage: stochastic rounding
  unsigned round_key;      // key of the rounding bits
  long long step;          // index n of the step being launched
  int y_off;               // lattice row of the context's row 0 (a strip of a larger lattice; else 0)
};

// A lattice's stirring: modes and phase tables (device pointers) and the tables of a step.
struct HostStir {
  int nrows;
  const void *G_cur, *EY;
  int eyp;
  void *G_next;              // the table of step_next, built by the launch (NULL: none)
  long long step_next;
  const int *mode_kx, *row_start;
  const void *tw;            // [nx] exp(i 2 pi j / nx), (re, im) in the compute type
  unsigned long long seed;
  double amp;
  const double *mode_scale;  // device [nmodes]; NULL = all 1
};

// What an observation of a lattice writes (device memory; rlbm_kernels.cuh): fields and
// totals (mode 0), velocities for the transform (mode 1) or column means (mode 2).
struct HostObs {
  double *eps, *ux, *uy;
  double2 *z;
  double *partials, *totals;
  unsigned *sync;
  double *bins;  // mode 1: nbins values cleared for the spectrum
  int nbins;
  float zscale;  // mode 1, FP32 states: the factor of z (spectrum_scale)
};

// The power of two that FP32 velocities are scaled by for their transform (an exact product): the
// largest for which sum |Z|^2 <= (nx ny)^2 max |v|^2 stays below 2^126, so that the squares of all
// velocities of FP32's normal range count.
inline float spectrum_scale(long long ncell) {
  float s = 0x1p63f;
  for (long long n = 1; n < ncell; n *= 2) s *= 0.5f;
  return s;
}

// One lattice of a batch, as the batched step kernel sees it (device memory, written by
// the host before the launches; 128-byte aligned so its tensor maps are 64-byte aligned).
struct alignas(128) MemberDesc {
  CUtensorMap tin[2];      // loads of population buffer 0 / 1
  CUtensorMap tG[2];       // stirring rows of step parity 0 / 1
  CUtensorMap tEY;
  void *f[2];              // population buffers
  const uint16_t *nbmask;  // NULL = no solid cells and no walls
  int nx, ny, pitch, walls;
  long long plane;
  int cur0;                // buffer holding f*_n at batch step 0
  int nrows, eyp;
  long long step0;         // the member's step index at batch step 0
  void *G[2];              // stirring tables of even and odd steps
  const void *EY, *tw;
  const int *mode_kx, *row_start;
  const double *mode_scale;
  unsigned long long seed;
  unsigned round_key;
  unsigned *err;
  int ntx;                 // tiles per row
  float rcp_ntx;           // 1 / ntx (tile index -> row and column with one correction)
};

// Prefix tables of a batch (device): tiles and chunks of stirring tables per member.
struct BatchTables {
  const MemberDesc *mem;
  const int *tile0;        // [n + 1]
  const int *prep0;        // [n + 1]
  int *tile_ctr;           // tiles handed out so far in this launch (0 before each launch)
  int n;
};

#define RLBM_DECLARE_LAUNCHERS(SUF)                                                                      \
  cudaError_t launch_step_##SUF(int vset, const void *tin, const void *tg, const void *tey, void *fout,     \
                                const HostGeom &g, const HostPhys &p, const HostStir &s, unsigned *err, \
                                int grid_limit, int stages, int stir_rows, int *ctr, unsigned seq,      \
                                bool chained, void *macro_out, cudaStream_t st);                         \
  cudaError_t launch_ghosts_##SUF(int vset, void *f, const HostGeom &g, cudaStream_t st);               \
  cudaError_t launch_batch_step_##SUF(int vset, const BatchTables &bt, const HostGeom &w, const HostPhys &p, \
                                      int srows, double amp, const long long *bstep, bool mask, int stages, \
                                      int grid_limit, int ntiles, cudaStream_t st);                       \
  cudaError_t launch_observe_##SUF(int vset, int mode, const void *fin, const HostGeom &g, double eps0,   \
                                   double vmax2, const HostObs &o, unsigned *err, int sms, cudaStream_t st); \
  cudaError_t launch_init_##SUF(int vset, void *fout, const HostGeom &g, double eps0, const double *e,  \
                                const double *ux, const double *uy, cudaStream_t st);                   \
  cudaError_t launch_open_ghosts_##SUF(int vset, void *f, const HostGeom &g, double ux_in, cudaStream_t st); \
  cudaError_t launch_stir_tables_##SUF(const HostStir &s, void *G, long long table, int nx, long long n,  \
                                       int count, cudaStream_t st);

RLBM_DECLARE_LAUNCHERS(f64)
RLBM_DECLARE_LAUNCHERS(f32)
RLBM_DECLARE_LAUNCHERS(f16)
RLBM_DECLARE_LAUNCHERS(bf16)

// One adjoint step (rlbm_adjoint.cu): buffers and tables of the launch.
struct AdjointArgs {
  const void *kin;         // kappa_{n+1} (compute type), NULL for the last state
  const void *tB, *tK;     // host CUtensorMap load maps of the post-collision buffer B_{n-1} and of kin
  bool chained;            // the launch directly follows the reverse step of step n + 1 on the
                           // stream, and B_{n-1} was written before that step (programmatic launch)
  const void *macro;       // the step's eps/eps0 - 1, v_x, v_y, F_x, F_y and streamed h_0 .. h_{Q-1}
                           // per cell from the forward recomputation (5 + Q planes of nx * ny), or
                           // NULL (then B_{n-1} is pulled and matched: the objective of the last state)
  void *kout;              // kappa_n
  double cj;               // objective weight of the state S_n
  double *acc;             // [blocks][4] FP64 accumulators
  void *zpart;             // [block rows][nrows][nx] R4 of the compute type (this step's slot)
  const void *EY;          // phase rows of the stirring tables
  int nrows, eyp;
  unsigned *err;
};
// The mode gradients of nj consecutive steps from their adjoint launches' row projections.
struct ModeGradArgs {
  const void *zpart;       // [nj][block rows][nrows][nx] R4 of the compute type
  void *zsum;              // [nj][nrows][nx] R4 of the compute type
  const void *tw;          // [nx] double2 exp(+2 pi i t / nx)
  const void *twf;         // [nx] float2, the same rounded to FP32
  int nj, nby, nrows, nx, nmodes;
  const int *mode_kx, *row_start;
  unsigned long long seed;
  long long n0;            // step index of j = 0
  double amp;
  double *gstep;           // [nj][nmodes] per-step d J / d sigma_m (this segment's rows)
};
cudaError_t launch_adjoint_f64(int vset, const AdjointArgs &a, const HostGeom &g, const HostPhys &p, cudaStream_t st);
cudaError_t launch_adjoint_f32(int vset, const AdjointArgs &a, const HostGeom &g, const HostPhys &p, cudaStream_t st);
cudaError_t launch_mode_grads_f64(const ModeGradArgs &a, cudaStream_t st);
cudaError_t launch_mode_grads_f32(const ModeGradArgs &a, cudaStream_t st);
cudaError_t launch_mode_sum(const double *gstep, long long nsteps, int nmodes, double *gsig, cudaStream_t st);
cudaError_t launch_adj_twiddles(double2 *tw, float2 *twf, int n, cudaStream_t st);

// Halo rows of a strip (rlbm_aux.cu): nplanes rows of row_bytes each, the plane p's row at
// byte offset off[p] of the population buffer, to (pack) or from (unpack) buf[p * row_bytes].
struct HaloRows {
  int nplanes;
  long long off[8];
};
cudaError_t launch_halo_copy(char *pop, const HaloRows &rows, long long row_bytes, char *buf, bool pack,
                             cudaStream_t st);

// Reductions and spectrum (rlbm_aux.cu)
cudaError_t launch_counter_inc(long long *counter, int *tile_ctr, cudaStream_t st);
cudaError_t launch_reduce_partials(const double *partials, long long nblocks, double *totals, cudaStream_t st);

// The velocity field z = v_x + i v_y (interleaved, [y][x]) of caller-provided u^x, u^y.
cudaError_t launch_make_z(const double *ux, const double *uy, double2 *z, long long ncell, cudaStream_t st);
// Spectrum and band energy of z0; both buffers hold nx * ny complex numbers of 16 bytes and are
// overwritten.  f64: (re, im) in FP64; else high and low FP32 parts (re_h, im_h, re_l, im_l) of the
// velocities times spectrum_scale(nx * ny).
// twx, twy: exp(-2 pi i t / n) in the same form.
cudaError_t launch_band_energy(bool f64, int nx, int ny, const void *twx, const void *twy, void *z0, void *z1, long long k2lo,
                               long long k2hi, double *partials, double *out4, unsigned *sync, cudaStream_t st);
// (launch_spectrum adds to bins, which the caller has cleared; launch_band_energy uses the zeroed
// counter `sync` and leaves it zero)
cudaError_t launch_spectrum(bool f64, int nx, int ny, const void *twx, const void *twy, void *z0, void *z1, double *bins,
                            int nbins, cudaStream_t st);

}  // namespace rlbm
