"""The search for a launch shape on a model of the GPU: it times steps as a run makes them (parities
alternating, chained steps chained), picks the depth of chained steps and of steps launched by
themselves apart, and leaves the shape alone when a launch fails."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2205_04658_gb300", "csrc")

PROGRAM = r"""
#include <cstdio>
#include <vector>
#include "rlbm_tune.h"
using rlbm::LaunchShape;

// A masked FP32 lattice of two large buffers: chained steps are fastest with two stages, steps by
// themselves with one, and a step is slow when the one before it walked the same way.
struct Gpu {
  int calls = 0, fail_at = -1, queued = 0;
  bool warm[3] = {false, false, false};
  bool last_odd = false, timing = false, right = true;
  float ms = 0.0f;
  bool step(const LaunchShape &s, bool odd, bool chained) {
    if (calls++ == fail_at) return false;
    if (!timing) warm[chained ? s.chained_stages : s.stages] = true;
    if (timing && !warm[chained ? s.chained_stages : s.stages]) right = false;  // each depth ran before it is timed
    if (timing && queued == 0 && chained) right = false;  // as is the first of a call
    const int stages = chained ? s.chained_stages : s.stages;
    if (timing) {
      float t = 10.0f + (chained ? (stages == 2 ? 0.0f : 1.0f) : 3.0f + (stages == 1 ? 0.0f : 2.0f));
      t += s.grid == 304 ? 0.0f : 0.5f;
      t += s.rows == 1 ? 0.0f : 0.25f;
      if (odd == last_odd) t += 20.0f;
      ms += t;
      ++queued;
    }
    last_odd = odd;
    return true;
  }
  bool start() { timing = true; queued = 0; ms = 0.0f; return calls != fail_at; }
  bool stop(float &t) { timing = false; t = ms; return true; }
};

int main() {
  const int grids[4] = {0, 304, 456, 608};
  for (int reps : {2, 3, 10}) {
    Gpu gpu;
    LaunchShape best{0, 1, 1, 1};
    float ms = 0.0f;
    if (!rlbm::tune_shape(gpu, grids, 4, 2, reps, best, ms) || !gpu.right) return std::printf("order of the trials\n"), 1;
    if (best.grid != 304 || best.rows != 1 || best.chained_stages != 2 || best.stages != 1)
      return std::printf("grid %d rows %d chained %d alone %d\n", best.grid, best.rows, best.chained_stages, best.stages), 1;
    if (!(ms > 9.9f && ms < 12.6f)) return std::printf("ms %f: a parity was repeated\n", ms), 1;
  }
  for (int f = 0; f < 60; ++f) {
    Gpu gpu;
    gpu.fail_at = f;
    LaunchShape best{456, 1, 2, 2};
    float ms = 0.0f;
    if (rlbm::tune_shape(gpu, grids, 4, 2, 3, best, ms) || best.grid != 456 || best.chained_stages != 1 || best.stages != 2 || best.rows != 2)
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
    assert "tune_shape(" in body and "stages = c->chained_stages" not in body
