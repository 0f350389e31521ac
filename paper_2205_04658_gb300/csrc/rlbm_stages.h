// Rotation of shared-memory stages, in plain C++ so that it can be checked without a GPU.
// Fill j (j = 0, 1, ...) of a CTA goes into stage j % nst; its completion ends phase j / nst of
// that stage's mbarrier, and a wait for it names the parity (j / nst) & 1.
#pragma once

#ifdef __CUDACC__
#define RLBM_HD __host__ __device__ __forceinline__
#else
#define RLBM_HD inline
#endif

namespace rlbm {

// The parity that a wait for the last of `fills` fills that went into stage s names (fills > s).
RLBM_HD int last_fill_parity(int fills, int s, int nst) { return ((fills - 1 - s) / nst) & 1; }

// Before a CTA leaves early: wait(s, parity) once for the last fill of every stage, the only
// one that can still be in flight (a stage is refilled only after its fill before has landed).
// A wait for any other phase would return at once, or for nothing, and leave that copy to land in
// shared memory that may belong to another CTA by then.
template <class Wait> RLBM_HD void wind_down(int fills, int nst, Wait wait) {
  for (int s = 0; s < nst && s < fills; ++s) wait(s, last_fill_parity(fills, s, nst));
}

}  // namespace rlbm
