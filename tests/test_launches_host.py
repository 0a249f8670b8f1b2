"""What the host side launches, without a GPU (tests/fake_cuda.py)."""
import numpy as np
import pytest

from paper_2412_16845_gb300 import workloads as wl
from paper_2412_16845_gb300.gks import GKSSolver
from tests.fake_cuda import _fake_library, fake  # noqa: F401

SIDE = {"n": "nrbc", "p": "periodic", "m": "pec"}


def _grid(n, bc, limiter=None, phm=None):
    cells = int(np.prod(n))
    nc = (3 if len(n) == 2 else 6) + ((len(n) - 1) if phm else 0)
    w = wl.CartWorkload(name="host", dim=len(n), n=n, lo=(0.0,) * len(n),
                        hi=tuple(v / n[0] for v in n), bc=tuple(SIDE[b] for b in bc), cfl=0.25, steps=0,
                        eps=np.ones(cells), mu=None, fields0=np.zeros((nc, cells)), jz_mask=None,
                        src=None, c_lattice=1.0, limiter=limiter)
    w.phm = phm
    return w


# every launcher that needs more than 48 KB of shared memory: n, sides, limiter, cleaning, kappa, precision
BIG = [
    ((64, 64), "pppp", None, None, 0.0, "fp64", "cart2d_small_kernel"),
    ((100, 100), "nnnn", "vanleer", None, 0.0, "fp32", "cart2d_small_kernel"),
    ((40, 30, 20), "nnmmpp", None, None, 0.0, "fp32", "cart3d_small_kernel"),
    ((40, 30, 20), "nnnnnn", "vanleer", None, 0.0, "fp64", "cart3d_small_kernel"),
    ((33, 9, 600), "nnmmnn", None, None, 0.0, "fp64", "cart3d_tau0_f64_kernel"),
    ((90, 80, 70), "nnppnn", None, None, 0.0, "fp32", "cart3d_tau0_kernel"),
    ((30, 20, 10), "nnnnnn", None, (0.7, 1.3), 0.0, "fp32", "cart3d_phm_tau0_kernel"),
    ((30, 20, 10), "mmnnnn", "vanleer", (0.7, 1.3), 0.0, "fp64", "cart3d_phm_tau0_kernel"),
    ((200, 90), "nnnn", None, None, 0.05, "fp32", "cart2d_step_kernel_s"),
    ((200, 90), "nnnn", None, (0.0, 1.0), 0.05, "fp32", "cart2d_psi_step_kernel_s"),
    ((40, 30, 20), "nnppnn", None, None, 0.05, "fp32", "cart3d_side_kernel"),
    ((40, 30, 20), "mmnnnn", None, None, 0.05, "fp32", "cart3d_step_kernel"),
]


@pytest.mark.parametrize("n,bc,limiter,phm,kappa,precision,kernel", BIG)
def test_a_second_device_gets_its_shared_memory(fake, n, bc, limiter, phm, kappa, precision, kernel):
    """The limit of dynamic shared memory is a setting of each device: a step that ran on one device runs
    on the next one, and again on the first."""
    for device in (0, 1, 0, 3):
        fake.set_device(device)
        s = GKSSolver.from_workload(_grid(n, bc, limiter, phm), precision=precision, kappa=kappa)
        fake.launched()
        s.step(2)
        names = fake.launched()
        s.close()
        assert names and all(kernel in k for k in names), names
