"""The wind-down of a CTA whose staged copy does not land in time, on a model of its mbarriers: it
waits for every copy still in flight, whichever fill of the rotation that is.  (A barrier's phase c
is the one after c completed ones; a wait for parity p returns at once unless p is phase c's own.)"""
import os
import re
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2205_04658_gb300", "csrc")

PROGRAM = r"""
#include <cstdio>
#include <set>
#include <vector>
#include "rlbm_stages.h"

// A rotation of nst stages in which the copy of fill `late` does not land; `total` fills at most.
// The loop waits for fill k at the head of item k (nst = 1, refilled behind that wait), or for
// fill k + 1 at the end of item k, before stage k % nst is refilled (nst >= 2).
struct Run {
  int nst, late, started = 0, k = 0;
  std::vector<int> completed;
  Run(int nst_, int late_, int total) : nst(nst_), late(late_), completed(nst_, 0) {
    auto start = [&] { if (started < total) ++started; };
    for (int s = 0; s < nst; ++s) start();
    for (int j = 0; j < late; ++j) completed[j % nst]++;  // fills before the late one have landed
    if (nst == 1) {
      for (k = 0; k < late; ++k) start();
    } else if (late > 0) {
      for (k = 0; k + 1 < late; ++k) start();
    }
  }
  bool returns_at_once(int s, int parity) const { return (completed[s] & 1) != parity; }
};

int main() {
  int fixed_parity_misses = 0;
  for (int nst = 1; nst <= 3; ++nst)
    for (int total = 1; total <= 9; ++total)
      for (int late = 0; late < total; ++late) {
        const Run r(nst, late, total);
        const int fills = nst + r.k < total ? nst + r.k : total;  // as the kernels count them
        if (fills != r.started) return std::printf("fills %d, started %d (nst %d late %d)\n", fills, r.started, nst, late), 1;
        std::set<int> in_flight;  // stages with a fill that has not landed
        for (int j = late; j < r.started; ++j) in_flight.insert(j % nst);
        std::set<int> waited;
        bool right = true;
        rlbm::wind_down(fills, nst, [&](int s, int parity) {
          waited.insert(s);
          // it blocks exactly when the stage's copy is still in flight
          if (r.returns_at_once(s, parity) == (in_flight.count(s) != 0)) right = false;
        });
        for (int s : in_flight) {
          if (!waited.count(s)) right = false;
          if (r.returns_at_once(s, 0)) ++fixed_parity_misses;
        }
        if (!right) return std::printf("nst %d total %d late %d\n", nst, total, late), 1;
      }
  std::printf("%d\n", fixed_parity_misses);
  return 0;
}
"""


def test_wind_down_waits_for_the_copies_in_flight(tmp_path):
    src, exe = tmp_path / "stages.cpp", tmp_path / "stages"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-O1", "-Wall", "-Werror", "-I", CSRC, "-o", str(exe), str(src)], check=True)
    out = subprocess.run([str(exe)], capture_output=True, text=True)
    assert out.returncode == 0, out.stdout
    # a wait for parity 0 whatever the fill, as each kernel had it, passes by copies of odd phases
    assert int(out.stdout) > 0


@pytest.mark.parametrize("name,kernels", [("rlbm_kernels.cuh", 2), ("rlbm_adjoint.cu", 2)])
def test_every_tiled_kernel_winds_down(name, kernels):
    src = open(os.path.join(CSRC, name)).read()
    latched = [m.end() for m in re.finditer(r"atomicOr\([^;]*ERR_TIMEOUT\);", src)]
    assert len(latched) == kernels
    for at in latched:
        assert re.match(r"\s*(//[^\n]*\n\s*)*wind_down\((NST == 1 \? k : NST \+ k, NST|min\(NST \+ k, my_tiles\), NST|1 \+ k, 1),", src[at:]), src[at:at + 200]
