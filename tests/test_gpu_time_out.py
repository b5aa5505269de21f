"""The time-out path of both tensor-core M2L kernels: the 3xFP16 one of a mixed
plan's evaluate (slots split over CTAs, and whole tiles) and the exact-split one
of its backward.  With a bound of one poll every CTA gives up with copies and
MMAs in flight; it has to wait for them before it gives its shared and tensor
memory back, so that whatever runs next is right bit for bit.
"""
import numpy as np
import pytest
import torch

from workloads import generators as G

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2512_09478_gb300 import build as B
    B.build()
    torch.cuda.set_device(0)


@pytest.mark.parametrize("n", [20_000, 300_000])
def test_forward_and_adjoint_time_out_and_recover(n):
    from paper_2512_09478_gb300 import Plan
    x, q = G.uniform_charges(n, 51)
    xt, qt = (torch.tensor(a, dtype=torch.float32, device="cuda") for a in (x, q))
    w = torch.tensor(np.random.default_rng(52).normal(size=n), dtype=torch.float32, device="cuda")
    plan = Plan(p=4, leaf_cap=32, precision="mixed_fp16", n_max=n)
    plan.set_sources(xt, qt)
    pot, grad, _ = plan.evaluate()
    dq, dx = plan.backward(w, grad)
    assert plan.device_status() == 0
    for _ in range(3):
        plan.set_m2l_wait_bound(1)
        pot1, grad1, _ = plan.evaluate()
        assert plan.device_status() == 5      # KIFMM_ERR_TIMEOUT
        dq1, _ = plan.backward(w, grad)
        assert plan.device_status() == 5
        # callers that read no status (autograd) see it in the outputs
        assert torch.isnan(pot1).any() and torch.isnan(grad1).any() and torch.isnan(dq1).any()
        plan.set_m2l_wait_bound(0)
        pot2, grad2, _ = plan.evaluate()
        dq2, dx2 = plan.backward(w, grad2)
        assert plan.device_status() == 0
        for a, b in ((pot2, pot), (grad2, grad), (dq2, dq), (dx2, dx)):
            assert torch.equal(a, b)
