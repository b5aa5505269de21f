"""set_sources on a device that is nearly full.  Whichever allocation is refused,
the call reports KIFMM_ERR_CUDA or does without the buffer; the plan then takes
the next sources as if nothing had happened.  The room left is swept from a few
megabytes to more than the whole tree needs, so the refusal falls on the list
arrays, the expansions' slices, the tiles and the partial products in turn.
"""
import numpy as np
import pytest
import torch

from workloads import generators as G

pytestmark = pytest.mark.gpu

ROOM = [(2 << 20) * m for m in (1, 2, 3, 4, 6, 8, 12, 16, 24, 32, 48, 64, 96, 128, 192, 256, 512)]


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2512_09478_gb300 import build as B
    B.build()
    torch.cuda.set_device(0)


def _hog(room):
    """Tensors over all free device memory but `room` bytes, as far as the
    allocator goes."""
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    held, ask = [], torch.cuda.mem_get_info()[0] - room
    while ask >= 4 << 20:
        try:
            held.append(torch.empty(ask, dtype=torch.uint8, device="cuda"))
            ask = torch.cuda.mem_get_info()[0] - room
        except torch.OutOfMemoryError:
            ask = ask // 4 * 3
    return held


class _Set:
    def __init__(self, n, dtype, kernel, seed):
        x, q = G.uniform_charges(n, seed)
        if kernel == "stokeslet":
            q = np.random.default_rng(seed).normal(size=(n, 3))
        self.x, self.q = (torch.tensor(a, dtype=dtype, device="cuda") for a in (x, q))
        self.w = torch.tensor(np.random.default_rng(seed + 1).normal(size=n), dtype=dtype, device="cuda")
        self.out = [torch.empty(n, *s, dtype=dtype, device="cuda") for s in ((), (3,), (), (3,), (3,))]

    def run(self, plan, kernel):
        """The outputs on this set, in buffers of its own (nothing is allocated
        here); the second build sorts the digits this tree's depth asks for."""
        for _ in range(2):
            plan.set_sources(self.x, self.q)
        pot, grad, dq, dx, vel = self.out
        if kernel == "stokeslet":
            plan.evaluate(pot=vel)
            return [vel]
        plan.evaluate(pot=pot, grad=grad)
        plan.backward(self.w, grad, dq=dq, dx=dx)
        return [pot, grad, dq, dx]


@pytest.mark.parametrize("precision,kernel,reuse", [("mixed_fp16", "laplace", True), ("fp64", "laplace", False),
                                                    ("fp32", "laplace", True), ("fp32", "stokeslet", False)])
def test_a_refused_allocation_leaves_a_plan_that_works(precision, kernel, reuse):
    from paper_2512_09478_gb300 import KifmmError, Plan
    dtype = torch.float64 if precision == "fp64" else torch.float32
    small, big = _Set(1500, dtype, kernel, 61), _Set(20_000, dtype, kernel, 63)
    mk = lambda: Plan(p=4, leaf_cap=8, precision=precision, kernel=kernel, n_max=len(big.x), dtype=dtype,
                      reuse_lists=reuse)
    ref = {}
    for s in (small, big):
        plan = mk()
        ref[s] = [t.cpu() for t in s.run(plan, kernel)]
        assert plan.device_status() == 0
        plan.close()
    # (on the host: no device memory for the comparison).  A tree without room
    # for its partial products adds in another order: rounding, no more.
    tol = 1e-12 if precision == "fp64" else 1e-5

    def same(plan, s):
        got = [t.cpu() for t in s.run(plan, kernel)]
        return all(((a - b).norm() <= tol * b.norm()).item() for a, b in zip(got, ref[s]))

    base = _hog(6 << 30)
    refused = 0
    for room in ROOM:
        plan = mk()
        assert same(plan, small)
        hog = _hog(room)
        try:
            assert same(plan, big), room
        except KifmmError as e:
            assert e.code == 3, room            # KIFMM_ERR_CUDA
            refused += 1
            try:
                assert same(plan, small), room  # in what the refused call gave back
            except KifmmError as e2:
                assert e2.code == 3, room
        del hog
        torch.cuda.empty_cache()
        assert same(plan, small), room
        assert same(plan, big), room
        assert plan.device_status() == 0
        plan.close()
    del base
    torch.cuda.empty_cache()
    assert 0 < refused < len(ROOM)  # the sweep met both outcomes


@pytest.mark.parametrize("precision,kernel", [("mixed_fp16", "laplace"), ("fp64", "laplace"), ("fp32", "laplace"),
                                              ("fp64", "stokeslet")])
def test_the_bits_do_not_depend_on_the_room_for_partial_products(precision, kernel):
    """The partial products of the slot splits are the last thing set_sources
    asks for, and the kernels do without them: whatever room there is, a tree
    that builds gives the same bits, forward and adjoint."""
    from paper_2512_09478_gb300 import KifmmError, Plan
    dtype = torch.float64 if precision == "fp64" else torch.float32
    big = _Set(12_000, dtype, kernel, 65)
    mk = lambda: Plan(p=4, leaf_cap=8, precision=precision, kernel=kernel, n_max=len(big.x), dtype=dtype)
    plan = mk()
    ref = [t.cpu() for t in big.run(plan, kernel)]
    plan.close()
    base = _hog(6 << 30)
    taken = set()
    for room in (m << 20 for m in range(16, 640, 24)):
        plan = mk()
        hog = _hog(room)
        before = torch.cuda.mem_get_info()[0]
        try:
            got = [t.cpu() for t in big.run(plan, kernel)]
            taken.add((before - torch.cuda.mem_get_info()[0]) >> 21)
            assert all(torch.equal(a, b) for a, b in zip(got, ref)), room
            assert plan.device_status() == 0
        except KifmmError as e:
            assert e.code == 3, room
        del hog
        torch.cuda.empty_cache()
        plan.close()
    del base
    torch.cuda.empty_cache()
    assert len(taken) > 1  # with the buffer and without


def test_partial_products_are_bounded():
    """A tree of some 5000 boxes at p = 8: unbounded, the 189 slots' partial
    products of its 40 tiles would take 1.2 GB."""
    from paper_2512_09478_gb300 import Plan
    x, q = G.uniform_charges(120_000, 67)
    xt, qt = (torch.tensor(a, dtype=torch.float32, device="cuda") for a in (x, q))
    plan = Plan(p=8, leaf_cap=64, precision="mixed_fp16", n_max=len(x))
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    plan.set_sources(xt, qt)
    taken = before - torch.cuda.mem_get_info()[0]
    nb = plan.tree_info()["n_boxes"]
    # per box (a quarter more boxes than there are): lists 1.6 KB, eight
    # expansions of 296 values, their 16-bit slices; leaf pass lists
    per_box = 1700 + 8 * 4 * 297 + 2 * 2 * 320 + 3 * 2 * 320
    assert taken <= 1.25 * (nb + 256) * per_box + 8 * 6 * len(x) / 8 + (640 << 20) + (64 << 20)
