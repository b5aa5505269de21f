"""The leaf kernel's tuner times the plan's default table beside the candidates:
an FP64 plan, whose default (eight targets per pass) is none of them, keeps it
where it is the fastest."""
import pytest
import torch

from workloads import generators as G

pytestmark = pytest.mark.gpu


def test_fp64_tuning_keeps_the_default_where_it_wins():
    """Leaves of up to 64 points, 512 and 64 of them: the fastest candidate takes
    2.5 times as long (679 us against 265 on this shape)."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2512_09478_gb300 import Plan, build as B
    B.build()
    torch.cuda.set_device(0)
    x, q = G.uniform_charges(4096, 73)
    xt, qt = (torch.tensor(a, device="cuda") for a in (x, q))
    plans = [Plan(p=4, leaf_cap=64, precision="fp64", n_max=len(x), dtype=torch.float64, autotune=t)
             for t in (False, True)]
    outs = []
    for plan in plans:
        for _ in range(2):
            plan.set_sources(xt, qt)
        for _ in range(2):
            outs.append(plan.evaluate()[:2])
    tiles = [plan.tuning()["leaf_tiles"] for plan in plans]
    assert plans[1].tuning()["tuned_leaf"] and tiles[1] == tiles[0]
    # the same table, the same sums
    assert all(torch.equal(a, b) for o in outs[1:] for a, b in zip(o, outs[0]))
