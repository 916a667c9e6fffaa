"""Observed stepping with little room: shorter chunks, and no room for the
cells' values at all, give the results of the longest chunks."""
import numpy as np
import pytest

from paper_2103_01444_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def observe(case, precision, steps):
    from paper_2103_01444_gb300.build import build
    from paper_2103_01444_gb300.lbm import Domain
    build()
    d = Domain.from_case(case, precision=precision)
    out = [d.step_observe(n) for n in steps]
    i, heat = (np.concatenate([o[k] for o in out]) for k in range(2))
    return i, heat, d


@pytest.mark.parametrize("precision", ["fp32", "bf16", "fp64"])
@pytest.mark.parametrize("rows", [0, 1])
def test_short_chunks_and_none_observe_the_same(precision, rows, monkeypatch):
    steps = (7, 150, 66, 1, 35)
    case = W.small_cathode(131, 37, rows)
    i, heat, d = observe(case, precision, steps)
    state, now = d.state(), d.current_density()[:2]
    assert now == (i[-1], heat[-1])
    then = d.step_observe(5)
    # the slots of the sums are the call's first two allocations, then come a
    # column sum and the cells' values per chunk length; a domain makes 13
    # (no solids): 17 fails once (chunks of 32), 16+ always (none)
    for fail in ("17", "16+"):
        monkeypatch.setenv("PEMLBM_FAIL_ALLOC", fail)
        j, heat_j, e = observe(case, precision, steps)
        monkeypatch.delenv("PEMLBM_FAIL_ALLOC")
        np.testing.assert_array_equal(i, j)
        np.testing.assert_array_equal(heat, heat_j)
        np.testing.assert_array_equal(state, e.state())
        assert e.current_density()[:2] == now
        np.testing.assert_array_equal(e.step_observe(5), then)


def test_a_thick_catalyst_takes_no_more_than_its_share():
    """A lattice that is nearly all catalyst: the values kept beside it stay
    below a quarter of its two states and the shortest chunk's."""
    import torch
    case = W.cathode_blocks(2048, 1024, Re=3.0)
    rows = np.ones((1024, 2048))
    case = dict(case, ny_cl=900, ny_gdl=60, phi=0.5 * rows, K_cm2=1e-8 * rows)
    from paper_2103_01444_gb300.build import build
    from paper_2103_01444_gb300.lbm import Domain
    build()
    warm = Domain.from_case(case, precision="fp32")
    i, heat = warm.step_observe(70)      # (loads the kernels)
    d = Domain.from_case(case, precision="fp32")
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    j, heat_j = d.step_observe(70)
    held = before - torch.cuda.mem_get_info()[0]
    states = 2 * 96 * 2048 * 1024
    assert held < states / 4 + (8 << 20), held / states
    np.testing.assert_array_equal(i, j)
    np.testing.assert_array_equal(heat, heat_j)
    one = Domain.from_case(case, precision="fp32")
    seen = []
    for _ in range(12):
        one.step(1)
        seen.append(one.current_density(profile=False)[:2])
    np.testing.assert_array_equal(i[:12], [c[0] for c in seen])
