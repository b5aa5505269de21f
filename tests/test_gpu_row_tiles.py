"""The row products' tiles (M2M, L2L, the leaf pseudo-inverses and their
adjoints), each reached by a level of its own size.

The rule, for a level of `t` rows, `ld` output columns and 152 SMs:
  FP32  64-row tiles (k_rows_big) from 152 blocks on; below, tiles of 16 rows,
        or of 4 when the 16-row ones are fewer than 152;
  FP64  64-row tiles (k_rows_f64) from 304 blocks on, and at any size when a
        whole-input tile does not fit shared memory (a Stokeslet from p = 7 on);
        below, tiles of 16 rows, or of 4 when those are fewer than 608.
The cloud's levels of 8, 64, 512, 4096 and some 27 000 boxes take all three.
"""
import numpy as np
import pytest
import torch

from oracle import oracle as O
from workloads import generators as G
from parity_helpers import rounding_floor

pytestmark = pytest.mark.gpu

SMS = 152


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2512_09478_gb300 import build as B
    B.build()
    O.build()
    torch.cuda.set_device(0)


def _up(a, b):
    return -(-a // b)


def _fp32_tile(t, ld):
    nc = min(range(5, 0, -1), key=lambda c: _up(ld, 32 * c) * c)  # the least padding, the wider on a tie
    if _up(t, 64) * _up(ld, 32 * nc) >= SMS:
        return "64 rows"
    return "4 rows" if _up(t, 16) * _up(ld, 32) < SMS else "16 rows"


def _fp64_tile(t, n):
    nkp = _up(n, 16) * 16
    if _up(t, 64) * _up(n, 160) >= 2 * SMS or 8 * (nkp * 32 + 16 * (nkp + 4)) > 200 * 1024:
        return "64 rows"
    return "4 rows" if _up(t, 16) * _up(n, 32) < 4 * SMS else "16 rows"


def _cloud():
    x, q = G.uniform_charges(40_000, 71)
    return x.astype(np.float32).astype(np.float64), q.astype(np.float32).astype(np.float64)


def _run(x, q, precision, p, M):
    from paper_2512_09478_gb300 import Plan
    dt = torch.float64 if precision == "fp64" else torch.float32
    plan = Plan(p=p, leaf_cap=M, precision=precision, n_max=len(x), dtype=dt)
    xt, qt = (torch.tensor(a, dtype=dt, device="cuda") for a in (x, q))
    plan.set_sources(xt, qt)
    pot, grad, _ = plan.evaluate()
    w = torch.tensor(np.random.default_rng(72).normal(size=len(x)), dtype=dt, device="cuda")
    dq, _ = plan.backward(w, grad)
    assert plan.device_status() == 0
    # <w, A q> = <A^T w, q>: the adjoint's row products
    a, b = float((w.double() * pot.double()).sum()), float((dq.double() * qt.double()).sum())
    scale = float(w.double().norm()) * float(pot.double().norm())
    assert abs(a - b) <= (1e-13 if precision == "fp64" else 1e-4) * scale
    return plan, pot.double().cpu().numpy(), grad.double().cpu().numpy()


@pytest.mark.parametrize("p", [4, 5])  # n_s = 56 and 98: 16-byte aligned rows and not
def test_fp32_levels(p):
    x, q = _cloud()
    plan, pot, grad = _run(x, q, "fp32", p, 4)
    ns = 6 * (p - 1) ** 2 + 2
    sizes = np.bincount(plan.tree()["level"])[1:]
    assert {_fp32_tile(int(t), ns + 1) for t in sizes} == {"4 rows", "16 rows", "64 rows"}
    pd, gd = O.direct(x, q)
    po, go, _ = O.kifmm(x, q, p=p, leaf_cap=4)
    assert O.rel_l2(pot, pd) <= 1.1 * O.rel_l2(po, pd) + 5e-6
    assert O.rel_l2(grad, gd) <= 1.1 * O.rel_l2(go, gd) + 5e-6


def test_fp64_levels():
    x, q = _cloud()
    plan, pot, grad = _run(x, q, "fp64", 5, 4)
    sizes = np.bincount(plan.tree()["level"])[1:]
    assert {_fp64_tile(int(t), 98) for t in sizes} == {"4 rows", "16 rows", "64 rows"}
    po, go, _ = O.kifmm(x, q, p=5, leaf_cap=4)
    bar_p, bar_g = rounding_floor(x, q, 5, 4, po, go)
    assert O.rel_l2(pot, po) <= bar_p and O.rel_l2(grad, go) <= bar_g


def test_fp64_rows_too_long_for_a_whole_input_tile():
    """Stokeslet, p = 7: 654 inputs, 64-row tiles on levels of a few boxes;
    against the oracle as the other Stokeslet orders are."""
    from paper_2512_09478_gb300 import Plan
    p, M, n = 7, 32, 1500
    assert _fp64_tile(8, 654) == "64 rows" and _fp64_tile(8, 456) == "4 rows"
    x, f = G.uniform_charges(n, 3)[0], np.random.default_rng(4).normal(size=(n, 3))
    u_o = O.kifmm_stokes(x, f, p=p, leaf_cap=M)
    bar = 1e-12
    for a, b in ((3.0, 0.1234567), (0.7, -0.3141592)):
        bar = max(bar, 10 * O.rel_l2(a * O.kifmm_stokes(a * x + b, f, p=p, leaf_cap=M), u_o))
    plan = Plan(p=p, leaf_cap=M, precision="fp64", n_max=n, dtype=torch.float64, kernel="stokeslet")
    plan.set_sources(torch.tensor(x, device="cuda"), torch.tensor(f, device="cuda"))
    u = plan.evaluate()[0]
    assert plan.device_status() == 0
    assert O.rel_l2(u.cpu().numpy(), u_o) <= bar
