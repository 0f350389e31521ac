// The search for a step kernel's launch shape, in plain C++ so that it can be checked without a GPU.
#pragma once

namespace rlbm {

struct LaunchShape {
  int grid;            // CTAs (0: as many as are resident)
  int chained_stages;  // stages of a step that follows another in the same call
  int stages;          // stages of a step launched by itself
  int rows;            // where the stirring rows of a tile come from (rlbm_set_launch)
};

// Times the candidates and keeps the fastest in `best` (its time per step in `ms`): the pipeline depth
// of chained steps with the CTA count and the source of the stirring rows, then, with those, the
// depth of steps launched by themselves.  Trial steps alternate between even and odd, as steps do
// in a run: on large lattices odd ones walk the tiles backwards, and a trial of one parity alone
// would miss L2 where a run hits.  Gpu: step(shape, odd, chained) queues a trial step, start() and
// stop(ms) time what is queued between; false from any ends the search.
template <class Gpu>
bool tune_shape(Gpu &gpu, const int *grids, int ngrids, int nrows_opts, int reps, LaunchShape &best, float &ms) {
  auto trial = [&](const LaunchShape &s, bool chain, float &t) {
    // (warm-up first, of each depth that the trial uses)
    if (!gpu.step(s, false, false) || !gpu.step(s, true, chain) || !gpu.start()) return false;
    for (int r = 0; r < reps; ++r)
      if (!gpu.step(s, r & 1, chain && r > 0)) return false;
    if (!gpu.stop(t)) return false;
    t /= (float)reps;
    return true;
  };
  LaunchShape found = best;
  float t = 0.0f;
  ms = 1e30f;
  for (int rows = 1; rows <= nrows_opts; ++rows)
    for (int stages = 2; stages >= 1; --stages)
      for (int gi = 0; gi < ngrids; ++gi) {
        const LaunchShape s{grids[gi], stages, best.stages, rows};  // (the first step of a trial is not chained)
        if (!trial(s, true, t)) return false;
        if (t < ms) { ms = t; found = s; }
      }
  float alone = 1e30f;
  int best_alone = found.stages;
  for (int stages = 2; stages >= 1; --stages) {
    LaunchShape s = found;
    s.stages = stages;
    if (!trial(s, false, t)) return false;
    if (t < alone) { alone = t; best_alone = stages; }
  }
  best = found;
  best.stages = best_alone;
  return true;
}

}  // namespace rlbm
