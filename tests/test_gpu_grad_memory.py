"""Device memory that gradients leave with their domains: it is given back on
request, and bounded over all domains."""
import gc

import numpy as np
import pytest

from paper_2103_01444_gb300 import workloads as W

pytestmark = pytest.mark.gpu

MB = 1 << 20


def free_bytes():
    import torch
    torch.cuda.synchronize()
    return torch.cuda.mem_get_info()[0]


def domain(nx, ny, precision):
    from paper_2103_01444_gb300.build import build
    from paper_2103_01444_gb300.lbm import Domain
    build()
    d = Domain.from_case(W.cathode_blocks(nx, ny, Re=3.0), precision=precision)
    d.step(4)
    return d


def test_the_workspace_is_released_on_request():
    d = domain(1024, 256, "fp32")
    J, g = d.grad(0, 6)                  # (also loads the kernels)
    d.set_grad_memory(0)
    before = free_bytes()
    d.set_grad_memory(-1)
    assert d.grad(0, 6)[0] == J
    held = before - free_bytes()
    assert held > 96 * 4 * 1024 * 256    # four sets of adjoint populations stay
    d.set_grad_memory(0)
    assert before - free_bytes() < 8 * MB
    J0, g0 = d.grad(0, 6)                # nothing is kept while the limit is 0
    assert before - free_bytes() < 8 * MB
    assert J0 == J
    for k in ("phi", "K", "D_O2"):
        np.testing.assert_array_equal(g0[k], g[k])


def test_a_transposed_step_takes_one_state():
    """lbm_vjp takes (and leaves) one population state, not the two that a
    gradient steps between and a third one."""
    nx, ny = 1024, 256
    d = domain(nx, ny, "fp32")
    lam = np.random.default_rng(0).standard_normal((24, ny, nx))
    d.vjp(lam)                           # (loads the kernels)
    d.set_grad_memory(0)
    before = free_bytes()
    d.set_grad_memory(-1)
    d.vjp(lam)
    held = before - free_bytes()
    state, cells = 96 * nx * ny, nx * ny
    # four sets of adjoint populations, six fields, the listed index, one state
    assert held < 4 * state + 40 * cells + 1.5 * state, held / state
    J = d.grad(0, 6)[0]                  # a gradient takes its second state
    assert before - free_bytes() > 4 * state + 40 * cells + 1.5 * state
    d.set_grad_memory(0)
    assert d.grad(0, 6)[0] == J


def test_kept_workspaces_are_bounded_over_all_domains():
    import torch
    total = torch.cuda.mem_get_info()[1]
    # two workspaces of 0.7 of the bound each, at 1204 bytes per FP64 cell
    ny = 128
    nx = int(0.7 * total / 64 / 1204 / ny) // 64 * 64
    doms = [domain(nx, ny, "fp64") for _ in range(2)]
    for d in doms:
        d.grad(0, 3)                     # (loads the kernels)
        d.set_grad_memory(0)
        d.set_grad_memory(-1)
    before = free_bytes()
    J = [d.grad(0, 3)[0] for d in doms]
    held = before - free_bytes()
    assert total / 128 < held <= total / 64, held / total
    # the second domain's next call finds room once the first has let go
    doms[0].set_grad_memory(0)
    assert doms[1].grad(0, 3)[0] == J[1]
    assert total / 128 < before - free_bytes() <= total / 64
    for d in doms:
        d.close()
    gc.collect()
    assert free_bytes() >= before
