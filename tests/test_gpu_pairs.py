"""Several steps in one launch: runs that take their steps two or four at a
time must leave the states, read-outs and observed reactions of single steps,
bit for bit."""
import numpy as np
import pytest

from paper_2103_01444_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def set_ups():
    """Lattices around the strips of 30 columns and the chunks of rows of the
    two-step kernel and the 26 x 10 blocks of the four-step one, with every kind
    of boundary link; the last ones have too many blocks for four at a time."""
    out = []
    for nx, ny in ((30, 24), (31, 25), (26, 61), (53, 30), (200, 40), (331, 97)):
        out.append(("film", W.small_cathode(nx, ny, 0, Re=3.0)))
        out.append(("rows", W.small_cathode(nx, ny, 1, Re=3.0)))
    out.append(("grains", W.small_cathode(152, 64, 0, grains=True)))
    out.append(("pressure", dict(W.small_cathode(140, 31, 1), inlet="pressure", dp_in=5e-4)))
    out.append(("anodic", dict(W.small_cathode(140, 31, 0), alpha_a=0.5, V_op=1.0, scalar_advection=1)))
    out.append(("long", W.cathode_blocks(3001, 120, Re=3.0)))
    out.append(("long", W.small_cathode(2610, 127, 0, Re=3.0, grains=True, random_material=False)))
    out.append(("cavity", W.natural_convection_cavity(95, heated_bottom=True)))
    out.append(("cavity", W.natural_convection_cavity(601)))
    out.append(("kang", W.kang_surface_reaction(97, 48)))
    return out


@pytest.mark.parametrize("precision,rounding", [("fp32", "nearest"), ("bf16", "nearest"),
                                                ("fp16", "nearest"), ("fp16", "stochastic"),
                                                ("bf16", "stochastic"), ("fp64", "nearest")])
@pytest.mark.parametrize("n", [2, 5, 22])
def test_pairs_equal_single_steps(precision, rounding, n):
    from paper_2103_01444_gb300.build import build
    from paper_2103_01444_gb300.lbm import Domain
    build()
    for k, (name, case) in enumerate(set_ups()):
        if rounding == "stochastic" and case.get("kind"):
            continue
        make = lambda: Domain.from_case(case, precision=precision, rounding=rounding,  # noqa: E731
                                        interface_mode=k % 2)
        one, many, seen = make(), make(), make()
        currents = []
        for _ in range(n):
            one.step(1)
            currents.append(one.current_density(profile=False)[:2])
        many.step(n)
        i, heat = seen.step_observe(n)
        label = f"{name} {case['nx']}x{case['ny']}"
        for d in (many, seen):
            assert d.steps == n
            np.testing.assert_array_equal(d.state(), one.state(), err_msg=label)
            fa, fb = d.fields(), one.fields()
            for key in fa:
                np.testing.assert_array_equal(fa[key], fb[key], err_msg=f"{label} {key}")
            assert d.current_density()[:2] == currents[-1]
        np.testing.assert_array_equal(i, [c[0] for c in currents], err_msg=label)
        np.testing.assert_array_equal(heat, [c[1] for c in currents], err_msg=label)


def test_long_runs_cross_graph_replays():
    """Runs that replay the 64-step graph, observed or not, in one call or in
    several, end in the same state."""
    from paper_2103_01444_gb300.build import build
    from paper_2103_01444_gb300.lbm import Domain
    build()
    case = W.small_cathode(200, 40, 1)
    for precision in ("fp32", "fp64"):
        a, b, c = (Domain.from_case(case, precision=precision) for _ in range(3))
        a.step(341)
        for n in (130, 67, 1, 143):
            b.step(n)
        i = np.concatenate([c.step_observe(n)[0] for n in (200, 66, 75)])
        assert a.steps == b.steps == c.steps == 341 and i.shape == (341,)
        np.testing.assert_array_equal(a.state(), b.state())
        np.testing.assert_array_equal(a.state(), c.state())
        assert i[-1] == a.current_density()[0]
