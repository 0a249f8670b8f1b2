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


def _states(w, precision, *offsets):
    """Host buffers for states of w that start `offset` bytes past a 16-byte boundary."""
    from paper_2412_16845_gb300 import gks
    s = GKSSolver.from_workload(w, precision=precision)
    _, nbytes = gks.gks_state_layout(s.ctx)
    s.close()
    bufs = [np.zeros(nbytes + 64, dtype=np.uint8) for _ in offsets]
    return bufs, [(b.ctypes.data + 31) // 16 * 16 + o for b, o in zip(bufs, offsets)]


# kernels that copy rows by tensor maps need 16 bytes, those that load pairs need a pair, the rest a value
@pytest.mark.parametrize("precision,kappa,bc,src,dst,kernel", [
    ("fp32", 0.0, "nnnn", 0, 4, "cart2d_tau0_kernel"),
    ("fp32", 0.0, "nnnn", 8, 8, "cart2d_step_kernel_p"),
    ("fp32", 0.05, "nnnn", 0, 4, "cart2d_step_kernel_s"),
    ("fp32", 0.05, "nnnn", 8, 8, "cart2d_step_kernel_p"),
    ("fp32", 0.05, "ppnn", 4, 0, None),
    ("fp32", 0.05, "ppnn", 0, 4, None),
    ("fp64", 0.0, "nnnn", 8, 8, "cart2d_tau0_f64_kernel"),
    ("fp64", 0.05, "nnnn", 8, 0, None),
    ("fp64", 0.05, "nnnn", 0, 0, "cart2d_step_kernel"),
])
def test_a_callers_state_goes_to_a_kernel_that_takes_its_alignment(fake, precision, kappa, bc, src, dst, kernel):
    from paper_2412_16845_gb300 import gks
    w = _grid((4000, 3), bc)                          # too wide for the kernel of small grids
    keep, (p, q) = _states(w, precision, src, dst)
    s = GKSSolver.from_workload(w, precision=precision, kappa=kappa)
    fake.launched()
    if kernel is None:
        with pytest.raises(gks.GksError):
            gks.gks_step_state_window(s.ctx, p, q, 0, 0, 40, 0, 3)
        assert not fake.launched()
    else:
        gks.gks_step_state_window(s.ctx, p, q, 0, 0, 40, 0, 3)
        assert [kernel + "I" in k or kernel + "E" in k for k in fake.launched()] == [True]
    s.close()


@pytest.mark.parametrize("precision,kappa,lam,out,kernel", [
    ("fp32", 0.0, 0, 4, "adjoint_tau0_kernel"),
    ("fp32", 0.0, 8, 8, "adjoint_lambda_kernel"),     # accepted before the march by tensor copies came
    ("fp32", 0.05, 8, 0, "adjoint_lambda_kernel"),
    ("fp32", 0.05, 0, 4, None),
    ("fp64", 0.0, 8, 0, None),
    ("fp64", 0.0, 0, 0, "adjoint_lambda_kernel"),
])
def test_a_callers_lambda_goes_to_a_kernel_that_takes_its_alignment(fake, precision, kappa, lam, out, kernel):
    from paper_2412_16845_gb300 import gks
    w = _grid((40, 30), "nnpp")
    keep, (p, q) = _states(w, precision, lam, out)
    s = GKSSolver.from_workload(w, precision=precision, kappa=kappa)
    gks.gks_set_objective(s.ctx, None, None)
    fake.launched()
    if kernel is None:
        with pytest.raises(gks.GksError):
            gks.gks_adjoint_step(s.ctx, None, None, p, q, None, False)
        assert not fake.launched()
    else:
        gks.gks_adjoint_step(s.ctx, None, None, p, q, None, False)
        names = fake.launched()
        assert len(names) >= 1 and kernel in names[0], names
    s.close()


def test_a_failed_change_of_materials_keeps_extreme_permittivities_off_the_fast_reciprocals(fake):
    """set_materials that uploads eps and then finds no memory for mu: the context holds the new eps."""
    from paper_2412_16845_gb300 import gks
    w = _grid((40, 30), "nnnn")
    s = GKSSolver.from_workload(w, precision="fp32")
    fake.launched()
    s.step(1)
    assert "cart2d_small_kernel" in fake.launched()[0]
    fake.fail_allocation(0)
    with pytest.raises(gks.GksError):
        s.set_materials(np.full(1200, 1e-35), np.ones(1200))
    fake.fail_allocation(-1)
    fake.dll.cudaGetLastError()                       # the runtime's own record of the failed allocation
    fake.launched()
    s.step(1)
    assert "cart2d_step_kernel_s" in fake.launched()[0]
    s.set_materials(np.ones(1200))
    fake.launched()
    s.step(1)
    assert "cart2d_small_kernel" in fake.launched()[0]
    s.close()


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("n", [(1, 1), (5, 3), (64, 64), (100, 100), (173, 211), (288, 300), (290, 280), (24, 3600),
                               (24, 3700), (320, 280), (500, 300), (4000, 2)])
def test_every_step_of_a_2d_grid_takes_the_same_arithmetic(fake, n, precision):
    """Whole steps, in any number at a time and with a probe, windowed steps and steps between a caller's
    states: either all take the kernel of small grids or all the march."""
    from paper_2412_16845_gb300 import gks
    w = _grid(n, "nnpp" if n[1] > 1 else "nnnn")
    s = GKSSolver.from_workload(w, precision=precision)
    keep, (p, q) = _states(w, precision, 0, 0)
    fake.launched()
    for k in (1, 2, 3, 8, 11):
        s.step(k)
    x1, y1 = (n[0] + 1) // 2, (n[1] + 1) // 2
    gks.gks_step_window(s.ctx, 3, 0, n[0], 0, n[1])
    gks.gks_step_window(s.ctx, 2, 0, x1, 0, y1)
    gks.gks_step_state_window(s.ctx, p, q, 0, 0, x1, 0, y1)
    names = fake.launched()
    gks.gks_set_objective(s.ctx, [0], [0])
    s.step(5)
    names += [k for k in fake.launched() if "objective" not in k]
    s.close()
    small = sum("cart2d_small_kernel" in k for k in names)
    assert small in (0, len(names)), names
    assert (small > 0) == (-(-n[0] // 24) * -(-n[1] // 24) <= 152), n      # one 24 x 24 tile per SM at most


def _kernel_of(fake, n, bc, limiter, precision, kappa=0.0):
    s = GKSSolver.from_workload(_grid(n, bc, limiter), precision=precision, kappa=kappa)
    fake.launched()
    s.step(1)
    names = fake.launched()
    s.close()
    return names[0]


# what was timed (us a step): the faster one of one tile per CTA and of the kernel the step takes otherwise
@pytest.mark.parametrize("n,bc,limiter,precision,small", [
    ((64, 64, 64), "nnnnnn", None, "fp64", True),           # 162, march 261
    ((80, 80, 80), "nnnnnn", None, "fp64", True),           # 321, 331
    ((90, 80, 70), "nnnnnn", None, "fp64", False),          # 342, 308
    ((130, 118, 97), "nnnnnn", None, "fp64", False),        # 985, 929
    ((33, 9, 600), "nnnnnn", None, "fp64", False),          # 175, 162
    ((64, 64, 64), "nnnnnn", "vanleer", "fp64", True),      # 361, 493
    ((80, 80, 80), "nnnnnn", "vanleer", "fp64", False),     # 720, 620
    ((40, 40, 40), "nnnnnn", None, "fp32", True),           # 8.0, 9.8
    ((56, 48, 40), "nnnnnn", None, "fp32", False),          # 10.8, 9.8
    ((56, 48, 40), "nnnnnn", "vanleer", "fp32", True),      # 11.7, general kernel 23.0
    ((64, 64, 64), "mmmmmm", None, "fp32", True),           # 22.1, 35.3
    ((90, 80, 70), "mmmmmm", None, "fp32", False),          # 44.8, 43.7
])
def test_3d_rule_takes_the_faster_kernel(fake, n, bc, limiter, precision, small):
    assert ("cart3d_small_kernel" in _kernel_of(fake, n, bc, limiter, precision)) == small


def test_45_34_27_takes_the_tile_that_was_fastest(fake):
    """8 x 4 x 4 tiles: 7.0 us a step; 4 x 4 x 4: 9.1, 8 x 8 x 4: 7.6, 8 x 8 x 8: 7.9."""
    assert "cart3d_small_kernelIfLi2E" in _kernel_of(fake, (45, 34, 27), "nnpppp", None, "fp32")


def test_the_parity_grids_take_the_kernels_they_are_for(fake):
    """The grids of tests/test_gpu_tau0_march.py, test_gpu_slab_march.py and test_gpu_cart2d_general.py."""
    from tests import test_gpu_cart2d_general as general
    from tests import test_gpu_slab_march as slabs
    from tests import test_gpu_tau0_march as march
    for n, bc, limiter in march.MARCH_2D:
        assert "cart2d_tau0_kernel" in _kernel_of(fake, n, bc, limiter, "fp32"), n
        assert "cart2d_tau0_f64_kernel" in _kernel_of(fake, n, bc, limiter, "fp64"), n
    for n, bc, limiter, precision in march.MARCH_3D:
        kernel = "cart3d_tau0_f64_kernel" if precision == "fp64" else "cart3d_tau0_kernel"
        assert kernel in _kernel_of(fake, n, bc, limiter, precision), n
    for n, bc, limiter, precision in march.TILES_3D:
        assert "cart3d_small_kernel" in _kernel_of(fake, n, bc, limiter, precision), n
    for n, bc in general.STAGED:
        assert "cart2d_step_kernel_s" in _kernel_of(fake, n, bc, None, "fp32", general.KAPPA), n
    for _, _, _, precision, local, kernel in slabs.SLABS:
        assert kernel in _kernel_of(fake, local, "nn" * len(local), None, precision), local
