"""The M2L kernels at the edges of their tiles: surface orders whose expansion
lengths leave remainders in every blocking (n_s = 26, 98, 386: 16-column
groups, column blocks, 32-wide K blocks and chunks of them), trees of few
target tiles (the 189 slots split over CTAs) and of many, forward and adjoint.
"""
import numpy as np
import pytest
import torch

from oracle import oracle as O
from workloads import generators as G
from parity_helpers import rounding_floor

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2512_09478_gb300 import build as B
    B.build()
    torch.cuda.set_device(0)


def _plan(n, precision, p, M, **kw):
    from paper_2512_09478_gb300 import Plan
    return Plan(p=p, leaf_cap=M, max_depth=20, precision=precision, n_max=n,
                dtype=torch.float64 if precision == "fp64" else torch.float32, **kw)


def _dev(a, dtype):
    return torch.tensor(np.asarray(a), dtype=dtype, device="cuda")


@pytest.mark.parametrize("p", [3, 5, 9])
def test_fp64_and_fp32_orders(p):
    """FP64 against the oracle within the parity bar (1e-12, or 10x the
    method's rounding floor where that is larger); FP32 within the method's
    own error of the direct sum (10% and the budget of the other FP32 tests)."""
    x, q = G.uniform_charges(1500, 41)
    pot_o, grad_o, _ = O.kifmm(x, q, p=p, leaf_cap=16)
    bar_p, bar_g = rounding_floor(x, q, p, 16, pot_o, grad_o)
    plan = _plan(len(x), "fp64", p, 16)
    plan.set_sources(_dev(x, torch.float64), _dev(q, torch.float64))
    pot, grad, _ = plan.evaluate()
    assert O.rel_l2(pot.cpu().numpy(), pot_o) <= bar_p
    assert O.rel_l2(grad.cpu().numpy(), grad_o) <= bar_g
    x32, q32 = x.astype(np.float32).astype(np.float64), q.astype(np.float32).astype(np.float64)
    pd, gd = O.direct(x32, q32)
    po, go, _ = O.kifmm(x32, q32, p=p, leaf_cap=16)
    plan = _plan(len(x), "fp32", p, 16)
    plan.set_sources(_dev(x32, torch.float32), _dev(q32, torch.float32))
    pot, grad, _ = plan.evaluate()
    assert O.rel_l2(pot.double().cpu().numpy(), pd) <= 1.1 * O.rel_l2(po, pd) + 5e-6
    assert O.rel_l2(grad.double().cpu().numpy(), gd) <= 1.1 * O.rel_l2(go, gd) + 5e-6


@pytest.mark.parametrize("precision", ["fp64", "mixed_fp16"])
def test_adjoint_is_the_transpose(precision):
    """<w, A q> = <A^T w, q> with n_s = 98: to rounding in FP64, to the FP32
    modes' split of the mean (their adjoint transposes the plain method) else."""
    x, q = G.uniform_charges(3000, 42)
    w = np.random.default_rng(43).normal(size=len(x))
    plan = _plan(len(x), precision, 5, 16)
    dt = plan.dtype
    plan.set_sources(_dev(x, dt), _dev(q, dt))
    pot, grad, _ = plan.evaluate()
    dq, _ = plan.backward(_dev(w, dt), grad)
    a = float((_dev(w, dt).double() * pot.double()).sum())
    b = float((dq.double() * _dev(q, dt).double()).sum())
    scale = float(np.linalg.norm(w)) * float(pot.double().norm())
    assert abs(a - b) <= (1e-13 if precision == "fp64" else 1e-4) * scale


@pytest.mark.parametrize("precision,kernel,copies", [("mixed_fp16", "laplace", 24), ("fp32", "stokeslet", 24),
                                                     ("fp32", "stokeslet", 4)])
def test_one_system_alone_equals_its_copies(precision, kernel, copies):
    """One small system (slots split over CTAs, or narrow SIMT tiles) and many
    copies of it in one batch (whole tiles) run other launch shapes and the
    same sums in the same order: bit for bit the same outputs."""
    n, p, M = 4001, 4, 16
    x, q = G.uniform_charges(n, 44)
    x = _dev(x, torch.float32)
    q = _dev(q, torch.float32)
    if kernel == "stokeslet":
        q = _dev(np.random.default_rng(45).normal(size=(n, 3)), torch.float32)
    outs = []
    for k in (1, copies):
        plan = _plan(n * k, precision, p, M, kernel=kernel, n_systems_max=k)
        xs, qs = x.repeat(k, 1), q.repeat(k, *([1] * (q.dim() - 1)))
        for _ in range(2):  # the second build sorts the digits its own depth asks for
            plan.set_sources(xs, qs, [n * i for i in range(k + 1)])
        pot, grad, _ = plan.evaluate()
        assert plan.device_status() == 0
        outs.append((pot, grad))
    for i in (0, copies // 2, copies - 1):
        assert torch.equal(outs[1][0][n * i:n * (i + 1)], outs[0][0])
        if outs[0][1] is not None:
            assert torch.equal(outs[1][1][n * i:n * (i + 1)], outs[0][1])


@pytest.mark.parametrize("precision,p", [("fp64", 3), ("fp64", 6), ("fp32", 3), ("fp32", 4), ("mixed_fp16", 4),
                                         ("mixed_fp16", 5)])
def test_x_lists_at_every_block_width(precision, p):
    """P2L's block is n_s rounded up to a warp (32 to 160 threads here): a
    clustered cloud with W/X lists kept (direct_max = -1) against the direct
    sum, within the method's own error (10% and the FP32 budget)."""
    x = G.plummer(3000, 46)[0]
    q = np.random.default_rng(46).normal(size=len(x))
    x, q = x.astype(np.float32).astype(np.float64), q.astype(np.float32).astype(np.float64)
    pd, gd = O.direct(x, q)
    po, go, _ = O.kifmm(x, q, p=p, leaf_cap=16, direct_max=-1)
    plan = _plan(len(x), precision, p, 16, direct_max=-1)
    plan.set_sources(_dev(x, plan.dtype), _dev(q, plan.dtype))
    assert plan.tree_info()["n_x"] > 0
    pot, grad, _ = plan.evaluate()
    assert plan.device_status() == 0
    assert O.rel_l2(pot.double().cpu().numpy(), pd) <= 1.1 * O.rel_l2(po, pd) + 5e-6
    assert O.rel_l2(grad.double().cpu().numpy(), gd) <= 1.1 * O.rel_l2(go, gd) + 5e-6
