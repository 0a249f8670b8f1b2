"""GPU parity of the marching kernels for tau = 0 (2-D and 3-D) against the FP64 oracle on grids past the
rules of the small-grid kernels, at the widths, heights and depths where their strips, tiles and chunks begin
and end.  tests/test_launches_host.py holds the same grids against the kernel that each takes.  Relative L2:
FP64 1e-12, FP32 2e-5."""
import numpy as np
import pytest

from paper_2412_16845_gb300 import workloads as wl
from paper_2412_16845_gb300.gks import GKSSolver
from tests.oracle_runs import oracle_cart_run, rel_l2

pytestmark = pytest.mark.gpu

TOL = {"fp64": 1e-12, "fp32": 2e-5}

# 2-D: FP32 strips of 62 columns, four to a tile; FP64 strips of 30 or 62; chunks of 2 rows or more
MARCH_2D = [((61, 1300), "nnnn", None), ((62, 1300), "nnpp", None), ((63, 1301), "mnnn", None),
            ((30, 1900), "ppnn", None), ((31, 1900), "mmmm", None), ((2, 3700), "mmnn", None),
            ((1, 3700), "nnnn", None), ((3, 3701), "pppp", None), ((248, 373), "nnnn", None),
            ((249, 371), "nmnm", None), ((247, 373), "mnpp", None), ((310, 300), "ppmm", None),
            ((3700, 1), "nnnn", None), ((3700, 2), "mmpp", None), ((3700, 3), "ppmm", None),
            ((3701, 4), "pppp", None), ((63, 1303), "nnnn", "vanleer"), ((250, 370), "pppp", "vanleer"),
            ((3650, 5), "mmmm", "vanleer")]

# 3-D, FP64: strips of 30 cells, up to 8 rows and any number of planes per warp; FP32: tiles of 64 columns x
# 10 rows, chunks of planes (open and periodic sides)
MARCH_3D = [((33, 9, 600), "nnmmpp", None, "fp64"), ((60, 17, 170), "mmmmnn", None, "fp64"),
            ((90, 17, 120), "nnmmpp", None, "fp64"), ((60, 9, 310), "ppnnmn", None, "fp64"),
            ((33, 9, 601), "nnnnnn", "vanleer", "fp64"), ((59, 2, 1400), "mmnnpp", None, "fp64"),
            ((9, 400, 60), "nnmmnn", None, "fp64"), ((600, 33, 9), "mmnnpp", None, "fp64"),
            ((97, 89, 91), "nnmmnn", None, "fp64"),        # chunks of 4 rows x 7 planes
            ((65, 51, 50), "nnppnn", None, "fp32"), ((129, 41, 31), "ppnnpp", None, "fp32"),
            ((63, 1, 2600), "nnppnn", None, "fp32"), ((64, 30, 90), "nnnnnn", None, "fp32")]

# 3-D grids of several tiles per SM that take one tile per CTA all the same: FP64, and FP32 where the march
# does not run (limiter, walls)
TILES_3D = [((57, 43, 66), "nnnnnn", "vanleer", "fp32"), ((48, 50, 47), "mmnmpp", None, "fp32"),
            ((61, 40, 33), "nmppmm", "vanleer", "fp32"), ((63, 41, 30), "nnmmpp", None, "fp64"),
            ((45, 34, 27), "nnpppp", None, "fp32")]


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2412_16845_gb300 import build
    build.build()


def grid(n, bc, limiter=None, seed=0):
    rng = np.random.default_rng(seed + sum(n))
    cells = int(np.prod(n))
    mask = np.zeros(cells)
    at = rng.choice(cells, size=cells // 30, replace=False)
    mask[at] = rng.uniform(-3, 3, at.size)
    sides = tuple({"n": "nrbc", "p": "periodic", "m": "pec"}[b] for b in bc)
    hi = tuple(v / n[0] * (1.2 if a == 1 else 1.0) for a, v in enumerate(n))
    return wl.CartWorkload(name="march", dim=len(n), n=n, lo=(0.0,) * len(n), hi=hi, bc=sides, cfl=0.4, steps=0,
                           eps=rng.uniform(1.0, 4.0, cells), mu=None,
                           fields0=rng.standard_normal((3 if len(n) == 2 else 6, cells)), jz_mask=mask,
                           src=(1.0, 20.0, 0.02, 0.02), c_lattice=0.0, limiter=limiter)


def _check(w, precisions, steps):
    out = {}
    for precision in precisions:
        s = GKSSolver.from_workload(w, precision=precision)
        s.step(steps)
        out[precision], c = s.read_fields(), s.info()["c"]
        s.close()
    ref, _ = oracle_cart_run(w, steps, c=c)
    for precision, f in out.items():
        assert rel_l2(f, ref) <= TOL[precision], (precision, rel_l2(f, ref))


@pytest.mark.parametrize("n,bc,limiter", MARCH_2D)
def test_2d(n, bc, limiter):
    _check(grid(n, bc, limiter), ("fp32", "fp64"), 5)


@pytest.mark.parametrize("n,bc,limiter,precision", MARCH_3D + TILES_3D)
def test_3d(n, bc, limiter, precision):
    _check(grid(n, bc, limiter), (precision,), 2 if np.prod(n) < 300000 else 1)
