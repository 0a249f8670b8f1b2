"""GPU parity of the kernels that kappa > 0 takes on 2-D grids, against the FP64 oracle at kappa = 0.05:
the staged kernel (FP32, mu = 1; strips of 63 columns, chunks of 8 rows or more) with open and closed
sides, and windowed steps through every kernel.  Relative L2: FP32 2e-5, FP64 1e-12."""
import numpy as np
import pytest

from paper_2412_16845_gb300 import workloads as wl
from paper_2412_16845_gb300.gks import GKSSolver, gks_step_window
from tests.oracle_runs import oracle_cart_run, rel_l2

pytestmark = pytest.mark.gpu

TOL = {"fp64": 1e-12, "fp32": 2e-5}
KAPPA = 0.05


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2412_16845_gb300 import build
    build.build()


def _grid(n, bc, seed, source=True, limiter=None, mu=False):
    rng = np.random.default_rng(seed)
    cells = n[0] * n[1]
    mask = np.where(rng.random(cells) < 0.04, rng.uniform(-3, 3, cells), 0.0) if source else None
    sides = tuple({"n": "nrbc", "p": "periodic", "m": "pec"}[b] for b in bc)
    return wl.CartWorkload(name="general", dim=2, n=n, lo=(0.0, 0.0), hi=(1.0, 1.2 * n[1] / n[0]), bc=sides,
                           cfl=0.4, steps=0, eps=rng.uniform(1.0, 4.0, cells),
                           mu=rng.uniform(1.0, 2.0, cells) if mu else None,
                           fields0=rng.standard_normal((3, cells)), jz_mask=mask, src=(1.0, 20.0, 0.02, 0.02),
                           c_lattice=0.0, limiter=limiter)


# widths below, at and past one strip, faces of the high side on either half of a lane's pair, one and two
# rows, several chunks with an odd last one
STAGED = [((64, 47), "nnnn"), ((59, 9), "nnnn"), ((63, 2), "nnnn"), ((127, 130), "nnnn"), ((33, 40), "nnnn"),
          ((32, 5), "nnnn"), ((1, 7), "nnnn"), ((3, 1), "nnnn"), ((200, 3), "nnpp"), ((7, 300), "nnpp"),
          ((45, 2), "nnpp"), ((64, 47), "mmmm"), ((33, 9), "mmnn"), ((63, 2), "nnmm"), ((2, 7), "mmmm"),
          ((127, 130), "mmpp"), ((32, 5), "nmnn")]


@pytest.mark.parametrize("n,bc", STAGED)
def test_staged_kernel(n, bc):
    w = _grid(n, bc, seed=n[0] + 1000 * n[1])
    s = GKSSolver.from_workload(w, precision="fp32", kappa=KAPPA)
    s.step(13)
    out, c = s.read_fields(), s.info()["c"]
    s.close()
    ref, _ = oracle_cart_run(w, 13, kappa=KAPPA, c=c)
    assert rel_l2(out, ref) <= TOL["fp32"], rel_l2(out, ref)


# (the kernel each takes: staged, paired, scalar with mu, scalar FP64; kappa = 0: the two marches)
WINDOWS = [("fp32", KAPPA, "nnnn", None, False), ("fp32", KAPPA, "mmmm", None, False),
           ("fp32", KAPPA, "ppnn", None, False), ("fp32", KAPPA, "nnnn", "vanleer", False),
           ("fp32", KAPPA, "nnnn", None, True), ("fp64", KAPPA, "nnnn", None, False),
           ("fp32", 0.0, "ppnn", None, False), ("fp64", 0.0, "nnpp", None, False)]


@pytest.mark.parametrize("precision,kappa,bc,limiter,mu", WINDOWS)
def test_windowed_steps(precision, kappa, bc, limiter, mu):
    """After k steps over a window the cells at least 2 k inside it are those of the whole grid."""
    nx, ny, k = 190, 110, 3
    x0, x1, y0, y1 = 61, 170, 21, 96
    w = _grid((nx, ny), bc, seed=5, limiter=limiter, mu=mu)
    s = GKSSolver.from_workload(w, precision=precision, kappa=kappa)
    gks_step_window(s.ctx, k, x0, x1, y0, y1)
    out, c = s.read_fields(), s.info()["c"]
    s.close()
    ref, _ = oracle_cart_run(w, k, kappa=kappa, c=c)
    inner = (slice(None), slice(y0 + 2 * k, y1 - 2 * k), slice(x0 + 2 * k, x1 - 2 * k))
    o, r = (f.reshape(3, ny, nx)[inner] for f in (out, ref))
    assert rel_l2(o, r) <= TOL[precision], rel_l2(o, r)
