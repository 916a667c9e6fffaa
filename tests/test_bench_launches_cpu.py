"""bench.py counts the launches, and the steps that a pass takes, as the
library plans them (csrc/step_plan.h, can_quad in csrc/api.cu)."""
import os
import re
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
        std::printf("%d %d %d %ld\n", most, open, n,
                    (long)pemlbm::plan_steps(most == 4, most >= 2, n, open, false).launches());
}
"""


def test_launches_of_a_run_follow_the_library(tmp_path):
    (tmp_path / "plan.cc").write_text(PROGRAM)
    subprocess.check_call(["g++", "-std=c++17", "-I", CSRC, str(tmp_path / "plan.cc"), "-o",
                           str(tmp_path / "plan")])
    out = subprocess.check_output([str(tmp_path / "plan")], text=True).splitlines()
    assert len(out) == 3 * 2 * 301
    for line in out:
        most, go_on, n, launches = map(int, line.split())
        assert bench.run_launches(n, most, bool(go_on)) == launches, line


def test_launches_of_calls():
    assert bench.step_launches(20, 2) == 9 + 2          # pairs, then two single steps
    assert bench.step_launches(1000, 4) == 15 * 16 + 9 + 1 + 2   # 15 graphs and 40 steps
    assert bench.step_launches(150, 1) == 150
    assert bench.observed_launches(20, 2) == 9 + 2 + 2
    assert bench.observed_launches(70, 4) == (16 + 2) + (3 + 2)
    assert bench.observed_launches(32, 1, stochastic=True) == 32 + 3


def test_steps_at_once_follow_the_library():
    launch = open(os.path.join(CSRC, "lbm_launch.h")).read()
    cols, rows = map(int, re.search(r"kQuadCols = (\d+), kQuadRows = (\d+)", launch).groups())
    api = open(os.path.join(CSRC, "api.cu")).read()
    a, b = map(int, re.search(r"blocks <= (\d+) \* (\d+);", api).groups())
    for nx, ny in ((200, 40), (1024, 256), (cols * 128, rows * 9), (cols * 128 + 1, rows * 9 + 5),
                   (cols * 152, rows * 8), (cols * 152, rows * 8 + 1), (4096, 1024)):
        most = 4 if -(-nx // cols) * -(-ny // rows) <= a * b else 2
        case = {"nx": nx, "ny": ny}
        assert bench.steps_at_once(case, "fp32") == bench.steps_at_once(case, "bf16") == most
        assert bench.steps_at_once(case, "fp64") == 1
        assert bench.steps_at_once(case, "fp16", "stochastic") == 1
        assert bench.steps_at_once(dict(case, periodic_x=1), "fp32") == 1
    assert bench.steps_at_once({"nx": 200, "ny": 40}, "fp32") == 4
    assert bench.steps_at_once({"nx": 4096, "ny": 1024}, "fp32") == 2
