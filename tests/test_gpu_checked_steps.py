"""The kernels of several steps in the bounds-checked build.

A warp of the two-step kernel copies the next row's pulls into shared memory
while it works on this one.  Every copy has to be waited for before the warp
ends, since its shared memory then belongs to another block: the checked
library counts the rows asked for and the rows taken, and records a warp that
leaves with a row on its way.
"""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = r'''
from paper_2103_01444_gb300 import workloads as W
from paper_2103_01444_gb300.lbm import Batch, Domain, bounds_check

def check(what):
    v = bounds_check()
    assert v == 0, f"{what}: site {v >> 48}, value {v & ((1 << 48) - 1)}"

bounds_check()                                   # clears the record
# one strip and several, one chunk of rows and many, catalyst rows, walls
cases = [W.small_cathode(30, 24, 0), W.small_cathode(31, 25, 1), W.small_cathode(152, 64, 0, grains=True),
         W.small_cathode(331, 97, 1), W.cathode_blocks(2048, 500, Re=3.0), W.natural_convection_cavity(95)]
for precision in ("fp32", "bf16", "fp16"):
    for case in cases:
        label = f"{case['nx']}x{case['ny']} {precision}"
        d = Domain.from_case(case, precision=precision)
        d.step(3)                                # a pair and a single step
        check(label + " step")
        d.step_observe(8)                        # fours and pairs
        d.step(67)
        check(label + " observed")
        d.close()
    doms = [Domain.from_case(c, precision=precision) for c in cases[:4]]
    b = Batch(doms)
    for schedule in ("graph", "concurrent"):
        b.set_schedule(schedule)
        b.step(5)
        check(f"batch {schedule} {precision}")
    b.close()
    for d in doms:
        d.close()
print("CHECKED_OK")
'''


def test_steps_in_pairs_wait_for_every_row_they_asked_for():
    from paper_2103_01444_gb300.build import build
    lib = build(bounds_check=True)
    env = dict(os.environ, PEMLBM_LIB=lib, PYTHONPATH=ROOT)
    r = subprocess.run([sys.executable, "-c", CHILD], cwd=ROOT, env=env, capture_output=True,
                       text=True, timeout=900)
    assert r.returncode == 0 and "CHECKED_OK" in r.stdout, (r.stdout[-2000:], r.stderr[-4000:])
