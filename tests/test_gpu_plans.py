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


def singles(case, precision, n):
    """A domain stepped n times one by one, and every step's read-out."""
    from paper_2103_01444_gb300.lbm import Domain
    d = Domain.from_case(case, precision=precision)
    seen = []
    for _ in range(n):
        d.step(1)
        seen.append(d.current_density(profile=False)[:2])
    return d, np.array(seen)


@pytest.mark.parametrize("precision", ["fp32", "bf16", "fp16"])
def test_every_split_of_a_short_run(precision):
    """On lattices that step in fours, 3 and 4 steps are one pair and single
    steps, 7 and 8 a four, a pair and single ones; strips of 30 columns, chunks of
    rows and every kind of boundary link."""
    from paper_2103_01444_gb300.build import build
    from paper_2103_01444_gb300.lbm import Domain
    build()
    cases = [W.small_cathode(nx, ny, k % 2, Re=3.0)
             for k, (nx, ny) in enumerate(((30, 24), (31, 25), (26, 61), (53, 30), (200, 40), (331, 97)))]
    cases += [W.small_cathode(152, 64, 0, grains=True), W.small_cathode(152, 65, 1, grains=True),
              dict(W.small_cathode(140, 31, 1), inlet="pressure", dp_in=5e-4),
              dict(W.small_cathode(140, 31, 0), alpha_a=0.5, V_op=1.0, scalar_advection=1),
              W.cathode_blocks(3001, 120, Re=3.0), W.natural_convection_cavity(95, heated_bottom=True),
              W.kang_surface_reaction(97, 48)]
    for case in cases:
        one, seen = singles(case, precision, 0)[0], np.zeros((0, 2))
        many = {n: Domain.from_case(case, precision=precision) for n in (3, 4, 7, 8)}
        watched = {n: Domain.from_case(case, precision=precision) for n in many}
        for n in range(1, 9):
            one.step(1)
            seen = np.append(seen, [one.current_density(profile=False)[:2]], 0)
            if n in many:
                label = f"{precision} {case['nx']}x{case['ny']} {n}"
                many[n].step(n)
                assert_same(many[n], one, label)
                i, heat = watched[n].step_observe(n)
                assert_same(watched[n], one, label)
                np.testing.assert_array_equal(np.stack([i, heat], 1), seen, err_msg=label)


@pytest.mark.parametrize("precision,nx", [("fp32", 1031), ("bf16", 2077)])
def test_pairs_on_lattices_larger_than_the_cache(precision, nx):
    """Above 96 MB the two-step kernel also asks the L2 cache for coming rows."""
    from paper_2103_01444_gb300.build import build
    from paper_2103_01444_gb300.lbm import Domain
    build()
    case = W.cathode_blocks(nx, 524, Re=3.0)
    one, seen = singles(case, precision, 5)
    many, watched = (Domain.from_case(case, precision=precision) for _ in range(2))
    many.step(5)
    i, heat = watched.step_observe(5)
    assert_same(many, one, precision)
    np.testing.assert_array_equal(watched.state(), one.state())
    np.testing.assert_array_equal(np.stack([i, heat], 1), seen)


def test_long_observed_runs_in_pairs():
    """More observed steps than a chunk holds, on a lattice that runs in pairs."""
    from paper_2103_01444_gb300.build import build
    from paper_2103_01444_gb300.lbm import Domain
    build()
    case = W.cathode_blocks(1024, 500, Re=3.0)
    one, seen = singles(case, "fp32", 150)
    d = Domain.from_case(case, precision="fp32")
    i, heat = d.step_observe(150)
    np.testing.assert_array_equal(np.stack([i, heat], 1), seen)
    assert_same(d, one, "observed")


def test_every_shape_of_the_single_step():
    from paper_2103_01444_gb300.build import build
    from paper_2103_01444_gb300.lbm import Domain
    build()
    for precision in ("fp32", "bf16", "fp64"):
        for case in (W.small_cathode(131, 37, 1), W.natural_convection_cavity(61)):
            doms = [Domain.from_case(case, precision=precision) for _ in range(8)]
            for v, d in enumerate(doms):
                d.set_variant(v)
                for _ in range(10):
                    d.step(1)
                np.testing.assert_array_equal(d.state(), doms[0].state(), err_msg=f"{precision} {v}")


@pytest.mark.parametrize("schedule", ["graph", "concurrent"])
@pytest.mark.parametrize("precision", ["fp32", "bf16", "fp16"])
def test_batches_in_pairs(precision, schedule):
    """Uneven cases in one batch, a long catalyst among them: the row chunk is
    the batch's, not the case's own."""
    from paper_2103_01444_gb300.build import build
    from paper_2103_01444_gb300.lbm import Batch, Domain
    build()
    cases = [W.small_cathode(331, 97, 1, Re=3.0), W.small_cathode(35, 24, 0, Re=3.0),
             W.cathode_blocks(3001, 120, Re=3.0), W.small_cathode(152, 64, 0, grains=True)]
    doms = [Domain.from_case(c, precision=precision) for c in cases]
    b = Batch(doms)
    b.set_schedule(schedule)
    for n in (3, 4, 11):
        b.step(n)
    for d, case in zip(doms, cases):
        one, _ = singles(case, precision, 18)
        assert_same(d, one, f"{precision} {schedule} {case['nx']}x{case['ny']}")
    b.close()


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
