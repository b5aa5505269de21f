"""The SIMT M2L (FP32 Stokeslet and FP32 periodic cells): every column-block
width its rule picks, rows that are 16-byte aligned and not, and the slot split
in one round and in three, against the unsplit form bit for bit."""
import numpy as np
import pytest
import torch

from test_gpu_out_of_memory import ROOM, _hog
from workloads import generators as G

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2512_09478_gb300 import build as B
    B.build()
    torch.cuda.set_device(0)


class _Set:
    """Sources and output buffers on the device (nothing is allocated in run)."""

    def __init__(self, kernel, n, seed, dtype=torch.float32):
        x = G.uniform_charges(n, seed)[0].astype(np.float32)
        rng = np.random.default_rng(seed)
        q = rng.normal(size=(n, 3)) if kernel == "stokeslet" else np.repeat([1.0, -1.0], n // 2)
        self.kernel = kernel
        self.x, self.q = (torch.tensor(a.astype(np.float32), dtype=dtype, device="cuda") for a in (x, q))
        self.out = torch.empty(n, 3, dtype=dtype, device="cuda")

    def run(self, plan):
        """Velocities, or gradients (a periodic potential's offset comes from the
        far-image operator); on the host."""
        for _ in range(2):  # the second build sorts the digits this tree's depth asks for
            plan.set_sources(self.x, self.q)
        plan.evaluate(**({"pot": self.out} if self.kernel == "stokeslet" else {"grad": self.out, "want_pot": False}))
        assert plan.device_status() == 0
        return self.out.cpu().double()


def _plan(kernel, n, p, M, precision):
    from paper_2512_09478_gb300 import Plan
    return Plan(p=p, leaf_cap=M, precision=precision, n_max=n, kernel=kernel,
                dtype=torch.float64 if precision == "fp64" else torch.float32,
                cell=0.0 if kernel == "stokeslet" else 1.0, pinv_eps=1e-9 if precision == "fp64" else 0.0)


# outputs of the M2L, n (+ 1): 9, 27, 57, 99, 153, 219 and 24, 78, 168, 294
@pytest.mark.parametrize("kernel,p", [("laplace", p) for p in (2, 3, 4, 5, 6, 7)] +
                         [("stokeslet", p) for p in (2, 3, 4, 5)])
def test_every_width_against_another_kernel(kernel, p):
    """A mixed plan (periodic) and an FP64 plan of the same truncation
    (Stokeslet) run other M2L kernels on the same method; what remains is FP32
    rounding, 1e-5 to 1e-6 at these orders.  Bar 1e-4: a row, column or slot out
    of place is of order one."""
    other = "fp64" if kernel == "stokeslet" else "mixed_fp16"
    ref = _Set(kernel, 3000, 81, torch.float64 if other == "fp64" else torch.float32).run(
        _plan(kernel, 3000, p, 16, other))
    got = _Set(kernel, 3000, 81).run(_plan(kernel, 3000, p, 16, "fp32"))
    assert ((got - ref).norm() <= 1e-4 * ref.norm()).item()


# 576 and 4672 targets: at p = 6 (periodic) 70 and 565 MB of partial products
@pytest.mark.parametrize("kernel,p,n", [("laplace", 4, 3000), ("laplace", 6, 3000), ("laplace", 6, 30_000),
                                        ("laplace", 7, 30_000), ("stokeslet", 3, 3000), ("stokeslet", 4, 30_000)])
def test_split_equals_unsplit(kernel, p, n):
    """Whatever room there is for the partial products: one round, three, none."""
    from paper_2512_09478_gb300 import KifmmError
    src, few = _Set(kernel, n, 82), _Set(kernel, 64, 83)
    plan = _plan(kernel, n, p, 16, "fp32")
    ref = src.run(plan)
    plan.close()
    base = _hog(4 << 30)
    taken = set()
    for room in ROOM:
        plan = _plan(kernel, n, p, 16, "fp32")
        few.run(plan)
        hog = _hog(room)
        before = torch.cuda.mem_get_info()[0]
        try:
            got = src.run(plan)
            taken.add((before - torch.cuda.mem_get_info()[0]) >> 22)
            assert torch.equal(got, ref), room
        except KifmmError as e:
            assert e.code == 3, room
        del hog
        torch.cuda.empty_cache()
        plan.close()
    del base
    torch.cuda.empty_cache()
    assert len(taken) > 1  # split and not
