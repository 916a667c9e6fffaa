"""Every way a run can be split into launches of four, two and one steps ends
with the bits of steps taken one by one."""
import numpy as np
import pytest

from paper_2103_01444_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def assert_same(many, one, label):
    np.testing.assert_array_equal(many.state(), one.state(), err_msg=label)
    a, b = many.fields(), one.fields()
    for key in a:
        np.testing.assert_array_equal(a[key], b[key], err_msg=f"{label} {key}")
    assert many.current_density()[:2] == one.current_density()[:2], label


@pytest.mark.parametrize("schedule", ["graph", "concurrent"])
def test_repeated_batch_calls(schedule):
    """Batch calls that end in the buffers they began in and calls that end in
    the other ones, again and again: the graphs of 64 steps start from both."""
    from paper_2103_01444_gb300.build import build
    from paper_2103_01444_gb300.lbm import Batch, Domain
    build()
    cases = [W.small_cathode(200, 40, 1), W.small_cathode(131, 37, 0, grains=True)]
    doms = [Domain.from_case(c, precision="fp32") for c in cases]
    b = Batch(doms)
    b.set_schedule(schedule)
    total = 0
    for n in (128, 128, 130, 129, 200, 128, 66):
        b.step(n)
        total += n
    for d, case in zip(doms, cases):
        one = Domain.from_case(case, precision="fp32")
        for _ in range(total):
            one.step(1)
        assert d.steps == total
        assert_same(d, one, f"{schedule} {case['nx']}x{case['ny']}")
    b.close()
