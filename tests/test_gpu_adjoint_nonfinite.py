"""A loss whose gradient is infinite at one particle: that particle's own dL/dq
takes no dipole of its own (nor of a particle at the same place), so it is what
it is without it, in the FP32-based modes and in FP64."""
import numpy as np
import pytest
import torch

from workloads import generators as G

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp32", "mixed_fp16", "fp64"])
def test_own_infinite_dipole_is_left_out(precision):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2512_09478_gb300 import Plan, build as B
    B.build()
    torch.cuda.set_device(0)
    n = 2000
    x, q = G.uniform_charges(n, 74)
    x[11] = x[7]  # a pair at one place
    dt = torch.float64 if precision == "fp64" else torch.float32
    xt, qt = (torch.tensor(a, dtype=dt, device="cuda") for a in (x, q))
    g = torch.tensor(np.random.default_rng(75).normal(size=(n, 3)), dtype=dt, device="cuda")
    g[7] = 0.0
    plan = Plan(p=4, leaf_cap=32, precision=precision, n_max=n, dtype=dt)
    plan.set_sources(xt, qt)
    plan.evaluate()
    dq0, _ = plan.backward(dL_dgrad=g)
    g[7] = float("inf")
    dq1, _ = plan.backward(dL_dgrad=g)
    assert torch.isfinite(dq0).all()
    assert dq1[7] == dq0[7] and dq1[11] == dq0[11]
    assert not torch.isfinite(dq1[:7]).any()  # everyone else feels it
