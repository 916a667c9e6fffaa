"""How a run of steps is split into launches (csrc/step_plan.h), compiled for
the host: every step is taken, a run that ends here ends with a single step,
and where the buffers have to be kept an even number of steps is an even
number of launches."""
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2103_01444_gb300", "csrc")

PROGRAM = r"""
#include <cstdio>
#include "step_plan.h"
int main() {
  for (int kind = 0; kind < 3; ++kind)
    for (int open = 0; open < 2; ++open)
      for (int keep = 0; keep < 2; ++keep)
        for (int n = 0; n <= 300; ++n) {
          const pemlbm::StepPlan p = pemlbm::plan_steps(kind == 2, kind >= 1, n, open, keep);
          long taken = 0;
          for (long k = 0; k < p.launches(); ++k) taken += p.steps(k);
          std::printf("%d %d %d %d %ld %ld %ld %ld\n", kind, open, keep, n, (long)p.quads, (long)p.pairs,
                      (long)p.singles, taken);
        }
}
"""


@pytest.fixture(scope="module")
def plans(tmp_path_factory):
    d = tmp_path_factory.mktemp("plan")
    (d / "plan.cc").write_text(PROGRAM)
    subprocess.check_call(["g++", "-std=c++17", "-I", CSRC, str(d / "plan.cc"), "-o", str(d / "plan")])
    out = subprocess.check_output([str(d / "plan")], text=True)
    return [tuple(map(int, line.split())) for line in out.splitlines()]


def test_plans_take_every_step_and_end_with_a_single_one(plans):
    assert len(plans) == 3 * 2 * 2 * 301
    for kind, go_on, keep, n, quads, pairs, singles, taken in plans:
        assert min(quads, pairs, singles) >= 0
        assert taken == n == 4 * quads + 2 * pairs + singles
        assert quads == 0 or kind == 2
        assert pairs == 0 or kind >= 1
        if n and not go_on:
            assert singles >= 1


def test_an_even_number_of_steps_keeps_the_buffer(plans):
    for kind, go_on, keep, n, quads, pairs, singles, taken in plans:
        if keep:
            assert (quads + pairs + singles - n) % 2 == 0, (kind, go_on, n)
        # the graphs of 64 steps return to their buffer by themselves
        if go_on and n == 64:
            assert (quads + pairs + singles) % 2 == 0


SLOTS = r"""
#include <cstdio>
#include <vector>
#include "step_plan.h"
// calls of `n` steps of a batch of two pairable cases and one that is stepped
// one by one, as lbm_batch_step makes them: graphs captured
int captures(int n, int calls) {
  pemlbm::GraphSlots slots;
  std::vector<int> cur{0, 1, 0};
  int made = 0;
  for (int c = 0; c < calls; ++c) {
    int left = n;
    while (n >= 128 && left >= 66) {
      if (slots.find(cur) < 0) {
        slots.take(cur);
        ++made;
      }
      left -= 64;
    }
    for (int k = 0; k < 3; ++k) cur[k] ^= pemlbm::plan_steps(false, k < 2, left, false, false).launches() & 1;
  }
  return made;
}
int main() {
  for (int n = 128; n <= 600; ++n) std::printf("%d %d\n", n, captures(n, 40));
}
"""


def test_repeated_batch_calls_capture_two_graphs_at_most(tmp_path):
    (tmp_path / "slots.cc").write_text(SLOTS)
    subprocess.check_call(["g++", "-std=c++17", "-I", CSRC, str(tmp_path / "slots.cc"), "-o",
                           str(tmp_path / "slots")])
    out = subprocess.check_output([str(tmp_path / "slots")], text=True)
    made = dict(tuple(map(int, line.split())) for line in out.splitlines())
    assert len(made) == 473 and max(made.values()) <= 2
    assert made[130] == 1 and made[128] == 2   # 130 steps come back to their buffers, 128 swap them
