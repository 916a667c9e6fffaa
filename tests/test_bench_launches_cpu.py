"""bench.py counts the launches, and the steps that a pass takes, as the
library plans them (csrc/step_plan.h)."""
import os
import subprocess

import bench

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2103_01444_gb300", "csrc")

PROGRAM = r"""
#include <cstdio>
#include "step_plan.h"
int main() {
  for (int most : {1, 2, 4})
    for (int open = 0; open < 2; ++open)
      for (int n = 0; n <= 300; ++n)
        std::printf("plan %d %d %d %ld\n", most, open, n,
                    (long)pemlbm::plan_steps(most == 4, most >= 2, n, open, false).launches());
  for (int nx : {4, 26, 64, 65, 179, 180, 200, 640, 720, 1023, 1024, 1300, 2000, 4096, 8192, 100000})
    for (int ny : {3, 10, 12, 40, 160, 163, 256, 488, 489, 500, 1024, 2048, 30000})
      for (int cl : {0, 1, ny / 4, ny / 4 + 1, ny - 1})
        for (int esize : {2, 4})
          std::printf("most %d %d %d %d %d\n", nx, ny, cl, esize,
                      pemlbm::steps_at_once(nx, ny, (nx + 63) / 64 * 64, cl, esize));
}
"""


def test_launches_and_steps_at_once_follow_the_library(tmp_path):
    (tmp_path / "plan.cc").write_text(PROGRAM)
    subprocess.check_call(["g++", "-std=c++17", "-I", CSRC, str(tmp_path / "plan.cc"), "-o",
                           str(tmp_path / "plan")])
    out = subprocess.check_output([str(tmp_path / "plan")], text=True).splitlines()
    assert len(out) == 3 * 2 * 301 + 16 * 13 * 5 * 2
    seen = set()
    for line in out:
        v = [int(w) for w in line.split()[1:]]
        if line.startswith("plan"):
            assert bench.run_launches(v[2], v[0], bool(v[1])) == v[3], line
        else:
            case = {"nx": v[0], "ny": v[1], "ny_cl": v[2]}
            precision = "fp32" if v[3] == 4 else "bf16"
            assert bench.steps_at_once(case, precision) == v[4], line
            seen.add((v[3], v[4]))
    assert seen == {(e, k) for e in (2, 4) for k in (1, 2, 4)}


def test_launches_of_calls():
    assert bench.step_launches(20, 2) == 9 + 2          # pairs, then two single steps
    assert bench.step_launches(1000, 4) == 15 * 16 + 9 + 1 + 2   # 15 graphs and 40 steps
    assert bench.step_launches(150, 1) == 150
    assert bench.observed_launches(20, 2) == 9 + 2 + 2
    assert bench.observed_launches(70, 4) == (16 + 2) + (3 + 2)
    assert bench.observed_launches(32, 1, stochastic=True) == 32 + 3


def test_single_steps_of_what_may_not_share_launches():
    case = {"nx": 4096, "ny": 1024, "ny_cl": 51}
    assert bench.steps_at_once(case, "fp32") == bench.steps_at_once(case, "bf16") == 2
    assert bench.steps_at_once(case, "fp64") == 1
    assert bench.steps_at_once(case, "fp16", "stochastic") == 1
    assert bench.steps_at_once(dict(case, periodic_x=1), "fp32") == 1
