"""Slabs too large for the small-grid kernels (tests/test_gpu_slab.py has the others) against the FP64 oracle
on the whole grid: the marching kernels on a slab's local grid.  tests/test_launches_host.py holds the local
grids against the kernel each takes.  Relative L2: FP64 1e-12, FP32 2e-5."""
import numpy as np
import pytest

from paper_2412_16845_gb300 import gks as G
from paper_2412_16845_gb300 import slab
from paper_2412_16845_gb300 import workloads as wl
from tests.oracle_runs import oracle_cart_run, rel_l2
from tests.test_gpu_slab import _exchange_local

pytestmark = pytest.mark.gpu

TOL = {"fp64": 1e-12, "fp32": 2e-5}
# whole grid, ranks, local grid of the first rank (two ghost layers on each shared side), kernel
SLABS = [((3700, 13), 2, False, "fp32", (3700, 9), "cart2d_tau0_kernel"),
         ((3700, 13), 2, True, "fp64", (3700, 11), "cart2d_tau0_f64_kernel"),
         ((60, 9, 616), 2, False, "fp64", (60, 9, 310), "cart3d_tau0_f64_kernel"),
         ((64, 30, 176), 2, False, "fp32", (64, 30, 90), "cart3d_tau0_kernel")]


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2412_16845_gb300 import build
    build.build()


@pytest.mark.parametrize("n,world,ring,precision,local,kernel", SLABS)
def test_slabs_match_the_oracle(n, world, ring, precision, local, kernel):
    import torch
    dim, cells = len(n), int(np.prod(n))
    rng = np.random.default_rng(dim)
    bc = ["nrbc"] * (2 * dim)
    if ring:
        bc[-2:] = ["periodic"] * 2
    h = 1.0 / n[0]
    w = wl.CartWorkload(name="slab", dim=dim, n=n, lo=(0.0,) * dim, hi=tuple(h * v for v in n), bc=tuple(bc),
                        cfl=0.4, steps=0, eps=rng.uniform(1.0, 3.0, cells), mu=None,
                        fields0=rng.standard_normal((3 if dim == 2 else 6, cells)), jz_mask=None, src=None,
                        c_lattice=1.0)
    plans = [slab.partition(n[-1], world, r, ring) for r in range(world)]
    assert plans[0].n_local == local[-1]
    solvers = [slab.SlabSolver(w, p, precision=precision, backend="gloo") for p in plans]
    steps = 2
    for _ in range(steps):
        for s in solvers:
            G.gks_step(s.ctx, 1)
        _exchange_local(solvers)
    torch.cuda.synchronize()
    got = np.zeros_like(w.fields0)
    for s in solvers:
        got[:, s.ids[s.owned]] = s.read_owned()
        s.close()
    ref, _ = oracle_cart_run(w, steps, c=1.0)
    assert rel_l2(got, ref) <= TOL[precision], rel_l2(got, ref)
