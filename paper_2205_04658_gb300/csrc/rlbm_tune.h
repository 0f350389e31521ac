// The search for a step kernel's launch shape, in plain C++ so that it can be checked without a GPU.
#pragma once

namespace rlbm {

struct LaunchShape {
  int grid;    // CTAs (0: as many as are resident)
  int stages;  // tiles of shared memory in the pipeline
  int rows;    // where the stirring rows of a tile come from (rlbm_set_launch)
};

// Times the candidates and keeps the fastest in `best` (its time per step in `ms`).  Trial steps are
// chained as in a run, and alternate between even and odd as there: on large lattices odd steps walk
// the tiles backwards, and a trial of one parity alone would miss L2 where a run hits.
// Gpu: step(shape, odd, chained) queues a trial step, start() and stop(ms) time what is queued
// between; false from any ends the search.
template <class Gpu>
bool tune_shape(Gpu &gpu, const int *grids, int ngrids, int nrows_opts, int reps, LaunchShape &best, float &ms) {
  LaunchShape found = best;
  ms = 1e30f;
  for (int rows = 1; rows <= nrows_opts; ++rows)
    for (int stages = 2; stages >= 1; --stages)
      for (int gi = 0; gi < ngrids; ++gi) {
        const LaunchShape s{grids[gi], stages, rows};
        float t = 0.0f;
        if (!gpu.step(s, true, false) || !gpu.start()) return false;  // (warm-up first)
        for (int r = 0; r < reps; ++r)
          if (!gpu.step(s, r & 1, r > 0)) return false;
        if (!gpu.stop(t)) return false;
        t /= (float)reps;
        if (t < ms) { ms = t; found = s; }
      }
  best = found;
  return true;
}

}  // namespace rlbm
