"""Host logic of the launches of the deterministic schedules, on the CPU: `rounds_shape` (csrc/prrtc_launch.h)
keeps the rows that a batch's virtual workers hold back within the limit it is given, down to one round of the
caller's workers, and otherwise gives every block its sixteen warps.  A small host program built with nvcc
prints the shapes (device code is cross-compiled, nothing runs on a GPU)."""
import os
import subprocess

import pytest

from paper_2503_06757_gb300 import build as B

PROGRAM = r'''
#include <cstdio>
#include "prrtc_launch.h"
using namespace prrtc;

int main() {
  const size_t limit = (size_t)1 << 28;
  const int modes[2] = {PRRTC_MODE_SERIAL, PRRTC_MODE_LOCKSTEP};
  for (int mode : modes)
    for (int workers : {1, 2, 3, 5, 8, 15, 16, 17, 40, 300, 1024})
      for (int n : {1, 5, 70, 152, 400})
        for (int given : {0, 3})       // the caller's warps per block
          for (size_t part : {1, 3, 16, 64, 1 << 20}) {
            const size_t held = limit / part / (mode == PRRTC_MODE_SERIAL ? 16 : workers);
            if (!held) continue;
            PlanLaunch base{};
            base.warps = mode == PRRTC_MODE_SERIAL ? 1 : std::min(given ? given : 8, workers);
            base.robot_bytes = 9000;
            base.env_bytes = 1600;
            base.stage_bytes = 11000;
            const RoundsLaunch c = rounds_shape(base, n, mode, 0, given, workers, held, limit, false, 152,
                                                [](int, int) { return 1; }, [](int, int) { return 16; });
            printf("%d %d %d %d %d %zu %d %d %d %d\n", mode, workers, n, given, (int)part, held, c.ph[c.n_phases - 1].warps, c.workers,
                   c.n_phases, c.ph[c.n_phases - 1].blocks);
          }
  return 0;
}
'''
LIMIT = 1 << 28
SERIAL = 1


@pytest.fixture(scope="module")
def shapes(tmp_path_factory):
    d = tmp_path_factory.mktemp("rounds")
    src, exe = os.path.join(d, "rounds.cu"), os.path.join(d, "rounds")
    with open(src, "w") as f:
        f.write(PROGRAM)
    cmd = [B.nvcc()] + B.ARCH + ["-std=c++17", "--expt-relaxed-constexpr", "-I", B.CSRC, "-I", B.INCLUDE, src, "-o", exe]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-2000:]
    out = subprocess.run([exe], capture_output=True, text=True, check=True).stdout
    names = ("mode", "workers", "n", "given", "part", "held", "warps", "virtual", "phases", "blocks")
    return [dict(zip(names, map(int, line.split()))) for line in out.splitlines()]


def test_held_rows_stay_within_the_limit(shapes):
    assert len(shapes) > 300
    for s in shapes:
        assert s["held"] * s["virtual"] <= LIMIT, s
        round_of = 1 if s["mode"] == SERIAL else s["workers"]
        assert s["virtual"] >= round_of and s["virtual"] % round_of == 0, s


def test_shapes_with_room_are_full(shapes):
    for s in shapes:
        if s["given"] and s["mode"] != SERIAL:
            assert (s["phases"], s["blocks"], s["warps"]) == (1, 1, min(s["given"], s["workers"])), s
        elif s["part"] == 1 << 20:
            assert (s["warps"], s["blocks"]) == (16, 16), s
