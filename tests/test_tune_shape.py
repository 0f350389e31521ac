"""The search for a launch shape on a model of the GPU: it times steps as a run makes them (parities
alternating, all but the first of a call chained) and leaves the shape alone when a launch fails."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2205_04658_gb300", "csrc")

PROGRAM = r"""
#include <cstdio>
#include <vector>
#include "rlbm_tune.h"
using rlbm::LaunchShape;

// A lattice of two large buffers: two stages, 304 CTAs and staged rows are fastest, and a step is slow
// when the one before it walked the same way.
struct Gpu {
  int calls = 0, fail_at = -1, queued = 0;
  bool warm = false, last_odd = false, timing = false, right = true;
  LaunchShape last{-1, 0, 0};
  float ms = 0.0f;
  bool step(const LaunchShape &s, bool odd, bool chained) {
    if (calls++ == fail_at) return false;
    if (!timing) warm = true;
    if (timing && (s.grid != last.grid || s.stages != last.stages || s.rows != last.rows)) right = false;  // not warmed up
    if (chained != (timing && queued > 0)) right = false;  // the first step of a call is not chained
    if (timing) {
      ms += 10.0f + (s.stages == 2 ? 0.0f : 1.0f) + (s.grid == 304 ? 0.0f : 0.5f) + (s.rows == 1 ? 0.0f : 0.25f);
      if (odd == last_odd) ms += 20.0f;
      ++queued;
    }
    last = s;
    last_odd = odd;
    return true;
  }
  bool start() { timing = true; queued = 0; ms = 0.0f; return true; }
  bool stop(float &t) { timing = false; t = ms; return true; }
};

int main() {
  const int grids[4] = {0, 304, 456, 608};
  for (int reps : {1, 2, 3, 10}) {
    Gpu gpu;
    LaunchShape best{0, 1, 1};
    float ms = 0.0f;
    if (!rlbm::tune_shape(gpu, grids, 4, 2, reps, best, ms) || !gpu.right || !gpu.warm) return std::printf("order of the trials\n"), 1;
    if (best.grid != 304 || best.rows != 1 || best.stages != 2)
      return std::printf("grid %d rows %d stages %d\n", best.grid, best.rows, best.stages), 1;
    if (!(ms > 9.9f && ms < 10.1f)) return std::printf("ms %f: a parity was repeated\n", ms), 1;
  }
  for (int f = 0; f < 60; ++f) {
    Gpu gpu;
    gpu.fail_at = f;
    LaunchShape best{456, 1, 2};
    float ms = 0.0f;
    if (rlbm::tune_shape(gpu, grids, 4, 2, 3, best, ms) || best.grid != 456 || best.stages != 1 || best.rows != 2)
      return std::printf("failure at call %d\n", f), 1;
  }
  return 0;
}
"""


def test_search_times_what_a_run_does(tmp_path):
    src, exe = tmp_path / "tune.cpp", tmp_path / "tune"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-O1", "-Wall", "-Werror", "-I", CSRC, "-o", str(exe), str(src)], check=True)
    out = subprocess.run([str(exe)], capture_output=True, text=True)
    assert out.returncode == 0, out.stdout


def test_autotune_uses_the_search():
    src = open(os.path.join(CSRC, "rlbm_capi.cu")).read()
    body = src[src.index("rlbm_status rlbm_autotune("):src.index("rlbm_status rlbm_wait_selftest(")]
    assert "tune_shape(" in body
