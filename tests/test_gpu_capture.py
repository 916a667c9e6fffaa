"""Steps captured into a graph of the caller's: replays march on, alone and
with direct calls between them, and batches in steps of two keep their cases'
buffers."""
import numpy as np
import pytest

from paper_2103_01444_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def lattices():
    # in fours; in pairs (two states larger than the cache); one by one
    return [("fp32", W.small_cathode(200, 40, 1)), ("fp32", W.cathode_blocks(1024, 500, Re=3.0)),
            ("bf16", W.cathode_blocks(2048, 500, Re=3.0)), ("fp32", W.cathode_blocks(900, 225, Re=3.0)),
            ("fp64", W.small_cathode(96, 30, 0))]


@pytest.mark.parametrize("n", [4, 6, 8, 10, 12, 20])
def test_replays_of_a_captured_call_march_on(n):
    import torch
    from paper_2103_01444_gb300.build import build
    from paper_2103_01444_gb300.lbm import Domain
    build()
    for precision, case in lattices():
        stream = torch.cuda.Stream()
        d = Domain.from_case(case, precision=precision, stream=stream.cuda_stream)
        ref = Domain.from_case(case, precision=precision)
        d.step(3)
        ref.step(3)
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream):
            d.step(n)
        with torch.cuda.stream(stream):
            for _ in range(3):
                graph.replay()
        ref.step(3 * n)
        label = f"{precision} {case['nx']}x{case['ny']}"
        np.testing.assert_array_equal(d.state(), ref.state(), err_msg=label)
        assert d.current_density()[:2] == ref.current_density()[:2], label
        # direct calls of an even count leave the captured buffers in place
        i, _ = d.step_observe(n)
        d.step(n)
        j, _ = ref.step_observe(n)
        ref.step(n)
        np.testing.assert_array_equal(i, j, err_msg=label)
        with torch.cuda.stream(stream):
            graph.replay()
        ref.step(n)
        np.testing.assert_array_equal(d.state(), ref.state(), err_msg=label)


def test_batches_of_even_counts_keep_their_buffers():
    """Repeated batch calls of even counts, with captured single-domain steps
    of the same cases between them, end in the states of the domains stepped
    alone."""
    import torch
    from paper_2103_01444_gb300.build import build
    from paper_2103_01444_gb300.lbm import Batch, Domain
    build()
    cases = [W.small_cathode(200, 40, 1), W.small_cathode(131, 37, 0)]
    for schedule in ("graph", "concurrent"):
        stream = torch.cuda.Stream()
        doms = [Domain.from_case(c, precision="fp32", stream=stream.cuda_stream) for c in cases]
        refs = [Domain.from_case(c, precision="fp32") for c in cases]
        for d in doms:
            d.step(2)
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream):
            for d in doms:
                d.step(4)
        b = Batch(doms)
        b.set_schedule(schedule)
        taken = 2
        for n in (128, 8, 192, 4):
            b.step(n)
            with torch.cuda.stream(stream):
                graph.replay()
            taken += n + 4
        for d, r in zip(doms, refs):
            r.step(taken)
            np.testing.assert_array_equal(d.state(), r.state(), err_msg=schedule)
        b.close()
