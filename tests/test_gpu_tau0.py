"""GPU parity of the kernels for tau = 0 (the default kappa) with mu = 1 against the FP64 oracle, at the
sizes where their tiles, strips and chunks begin and end.  Tolerances (relative L2) are those of every
other path: FP64 <= 1e-12, FP32 <= 2e-5."""
import numpy as np
import pytest

from paper_2412_16845_gb300 import workloads as wl
from paper_2412_16845_gb300.gks import GKSSolver, gks_step_window
from tests.oracle_runs import oracle_cart_run, rel_l2

pytestmark = pytest.mark.gpu

TOL = {"fp64": 1e-12, "fp32": 2e-5}


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2412_16845_gb300 import build
    build.build()


def _grid(n, bc, seed, source=True, limiter=None, stretch=1.2):
    rng = np.random.default_rng(seed)
    cells = int(np.prod(n))
    nc = 3 if len(n) == 2 else 6
    mask = None
    if source:
        mask = np.zeros(cells)
        at = rng.choice(cells, size=max(1, cells // 30), replace=False)
        mask[at] = rng.uniform(-3, 3, at.size)
    hi = tuple(v / n[0] * (stretch if a == 1 else 1.0) for a, v in enumerate(n))
    return wl.CartWorkload(name="tau0", dim=len(n), n=n, lo=(0.0,) * len(n), hi=hi, bc=bc, cfl=0.4,
                           steps=0, eps=rng.uniform(1.0, 4.0, cells), mu=None,
                           fields0=rng.standard_normal((nc, cells)), jz_mask=mask,
                           src=(1.0, 20.0, 0.02, 0.02), c_lattice=0.0, limiter=limiter)


def _check(w, precision, steps, march=False):
    """march: windowed steps over the whole grid, which small grids do not take several at a time."""
    s = GKSSolver.from_workload(w, precision=precision)
    if march:
        gks_step_window(s.ctx, steps, 0, w.n[0], 0, w.n[1])
    else:
        s.step(steps)
    out = s.read_fields()
    c = s.info()["c"]
    s.close()
    ref, _ = oracle_cart_run(w, steps, c=c)
    assert rel_l2(out, ref) <= TOL[precision], rel_l2(out, ref)


# 2-D: FP32 strips of 62 columns, four to a tile; FP64 strips of 30 or 62; chunks of 2 rows or more
@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("n,bc", [
    ((61, 5), "nnnn"), ((62, 2), "nnpp"), ((63, 1), "nnnn"), ((30, 33), "ppnn"), ((31, 3), "mmmm"),
    ((248, 9), "nnnn"), ((249, 9), "nmnm"), ((247, 12), "mnpp"), ((310, 7), "ppmm"), ((125, 4), "pppp"),
    ((2, 40), "mmnn"), ((1, 3), "nnnn"), ((3, 2), "pppp"), ((500, 70), "nnnn"),
])
def test_2d_tiles(n, bc, precision):
    sides = tuple({"n": "nrbc", "p": "periodic", "m": "pec"}[b] for b in bc)
    _check(_grid(n, sides, seed=n[0] + 7 * n[1]), precision, 9, march=True)


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("n,bc", [((63, 9), "nrbc"), ((250, 6), "periodic"), ((130, 17), "pec")])
def test_2d_limited_tiles(n, bc, precision):
    _check(_grid(n, (bc,) * 4, seed=n[0], limiter="vanleer"), precision, 9, march=True)


# several steps per launch on small grids: tiles of 4 to 24 cells, 1 to 8 steps, walls inside a margin
@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("n,bc,steps,limiter", [
    ((64, 64), "pppp", 19, None), ((100, 100), "nnnn", 23, None), ((41, 77), "mmnn", 8, None),
    ((5, 3), "nmpp", 11, None), ((1, 1), "nnnn", 3, None), ((2, 2), "mmmm", 7, None),
    ((17, 90), "ppmn", 1, None), ((33, 20), "nnmm", 9, "vanleer"), ((3, 50), "pppp", 16, "vanleer"),
])
def test_2d_small_grids(n, bc, steps, limiter, precision):
    sides = tuple({"n": "nrbc", "p": "periodic", "m": "pec"}[b] for b in bc)
    _check(_grid(n, sides, seed=n[0] + 3 * n[1], limiter=limiter), precision, steps)


def test_2d_extreme_permittivity_keeps_its_results():
    """eps beyond 2^+-100 leaves the FP32 tau = 0 kernel (its reciprocal needs normal numbers); FP64 is
    the reference here, since the oracle's sums over velocities cancel at such eps."""
    w = _grid((64, 20), ("nrbc",) * 4, seed=3, source=False)
    w.eps[100] = 1e32
    w.c_lattice = 1.0
    out = {}
    for precision in ("fp64", "fp32"):
        s = GKSSolver.from_workload(w, precision=precision)
        s.step(5)
        out[precision] = s.read_fields()
        s.close()
    assert rel_l2(out["fp32"], out["fp64"]) <= 2e-5


# 3-D small grids: one tile per CTA
@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("n,bc,limiter", [
    ((45, 34, 27), "nnpppp", None), ((17, 5, 9), "mmnnpp", None), ((1, 1, 1), "pppppp", None),
    ((30, 3, 2), "nmppmn", None), ((20, 20, 20), "nnnnnn", "vanleer"), ((2, 33, 7), "ppmmnn", "vanleer"),
])
def test_3d_small_grids(n, bc, limiter, precision):
    sides = tuple({"n": "nrbc", "p": "periodic", "m": "pec"}[b] for b in bc)
    _check(_grid(n, sides, seed=n[0] + n[1], limiter=limiter), precision, 6)


# The marching kernels, on grids just past what takes one tile per CTA.  FP64: strips of 30 cells, up
# to 8 rows and any number of planes per warp; FP32: tiles of 64 columns x 10 rows, chunks of planes.
@pytest.mark.parametrize("n,bc,precision,limiter", [
    ((31, 73, 72), "nnmmpp", "fp64", None), ((121, 41, 33), "ppnnnm", "fp64", "vanleer"),
    ((59, 2, 1400), "mmnnpp", "fp64", None), ((65, 51, 50), "nnppnn", "fp32", None),
    ((129, 41, 31), "ppnnpp", "fp32", None), ((63, 1, 2600), "nnppnn", "fp32", None),
])
def test_3d_marching_tiles(n, bc, precision, limiter):
    sides = tuple({"n": "nrbc", "p": "periodic", "m": "pec"}[b] for b in bc)
    _check(_grid(n, sides, seed=sum(n), limiter=limiter), precision, 2)


# divergence cleaning, 3-D: tiles of 30 x 10 (FP32) or 30 x 6 (FP64) columns, chunks of planes
@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("n,bc,limiter", [
    ((30, 10, 7), "nnnnnn", None), ((31, 11, 6), "mnnmnn", None), ((29, 7, 5), "ppnnmm", None),
    ((61, 21, 40), "nnppnn", None), ((1, 1, 1), "nnnnnn", None), ((2, 13, 1), "mmnnpp", None),
    ((33, 6, 9), "nmppnn", "vanleer"), ((30, 31, 3), "pppppp", "vanleer"),
])
def test_3d_cleaning_tiles(n, bc, limiter, precision):
    sides = tuple({"n": "nrbc", "p": "periodic", "m": "pec"}[b] for b in bc)
    w = _grid(n, sides, seed=sum(n) + 11, limiter=limiter)
    rng = np.random.default_rng(n[0])
    w.fields0 = np.concatenate([w.fields0, rng.standard_normal((2, w.fields0.shape[1]))])
    w.phm, w.cfl = (0.7, 1.3), 0.25
    _check(w, precision, 5)
