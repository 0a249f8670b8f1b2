"""GPU tests of the adjoint for tau = 0 and of the design problem around it: streams, windows, periodic
sides, both precisions."""
import numpy as np
import pytest

from paper_2412_16845_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2412_16845_gb300 import build
    build.build()


def _design(nx, ny, bc, steps, design, probe, seed=4):
    """A design problem with random fields and eps; design and probe are boxes ((x0, x1), (y0, y1))."""
    rng = np.random.default_rng(seed)

    def cells(b):
        return (np.arange(*b[1])[:, None] * nx + np.arange(*b[0])[None, :]).ravel()
    return wl.CartWorkload(name="design", dim=2, n=(nx, ny), lo=(0.0, 0.0), hi=(1.0, ny / nx), bc=bc, cfl=0.5,
                           steps=steps, eps=rng.uniform(1.0, 3.0, nx * ny), mu=None,
                           fields0=rng.standard_normal((3, nx * ny)), jz_mask=None, src=None,
                           c_lattice=1.0, probe=cells(probe), design=cells(design).astype(np.int64))


OPEN = ("nrbc",) * 4


def test_gradient_on_another_stream():
    """A problem on its own stream, called while the caller's stream is still busy, gives the gradient of a
    problem on the current stream, bit for bit."""
    import torch
    from paper_2412_16845_gb300.adjoint import DesignProblem
    w = _design(300, 200, OPEN, 40, ((100, 180), (60, 120)), ((190, 200), (90, 99)))
    e = w.eps[w.design]
    p = DesignProblem(w, precision="fp32")
    J0, g0 = p.value_and_grad(e)
    p.close()
    for busy in (False, True):
        p = DesignProblem(w, precision="fp32", stream=torch.cuda.Stream())
        if busy:
            torch.cuda._sleep(200_000_000)                    # about 0.1 s on the caller's stream
        J = p.forward(e)
        if busy:
            torch.cuda._sleep(200_000_000)
        g = p.backward().cpu().numpy()
        p.close()
        assert J == J0 and np.array_equal(g, g0)


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_an_empty_probe_has_a_zero_gradient(precision):
    from paper_2412_16845_gb300.adjoint import DesignProblem
    w = _design(40, 30, OPEN, 9, ((10, 20), (8, 15)), ((30, 31), (5, 6)))
    w.probe = w.probe[:0]
    p = DesignProblem(w, precision=precision, checkpoint_every=4)
    J, g = p.value_and_grad(w.eps[w.design])
    p.close()
    assert J == 0.0 and g.size == w.design.size and not g.any()


def test_a_callers_states_between_16_byte_boundaries():
    """FP32 states 8 bytes past a 16-byte boundary: the adjoint and the step run without tensor copies and
    agree with the aligned calls to rounding."""
    import torch
    from paper_2412_16845_gb300 import gks
    w = _design(70, 40, OPEN, 1, ((10, 20), (8, 15)), ((30, 31), (5, 6)))
    s = gks.GKSSolver.from_workload(w, precision="fp32")
    gks.gks_set_objective(s.ctx, None, None)
    n, _ = gks.gks_state_layout(s.ctx)
    x = torch.zeros(n, device="cuda")
    gks.gks_copy_state(s.ctx, x.data_ptr())
    out = []
    for off in (0, 2):
        src, dst, lam = (torch.zeros(n + 4, device="cuda")[off:off + n] for _ in range(3))
        src.copy_(x)
        gks.gks_step_state_window(s.ctx, src.data_ptr(), dst.data_ptr(), 0, 0, 70, 0, 40)
        gks.gks_adjoint_step(s.ctx, None, None, src.data_ptr(), lam.data_ptr(), None, False)
        gks.gks_sync(s.ctx)
        out.append((dst.clone(), lam.clone()))
    s.close()
    for a, b in zip(out[0], out[1]):
        assert float((a - b).norm()) <= 2e-5 * float(a.norm()) and float(a.norm()) > 0


def _random_state(s, rng, dtype):
    """A random state in the context's layout, zero in the padding."""
    import torch
    from paper_2412_16845_gb300 import gks
    n, _ = gks.gks_state_layout(s.ctx)
    mask = torch.zeros(n, dtype=dtype, device="cuda")
    s.write_fields(np.ones((3, s.ncell)))
    gks.gks_copy_state(s.ctx, mask.data_ptr())
    x = torch.as_tensor(rng.standard_normal(n), device="cuda").to(dtype)
    gks.gks_sync(s.ctx)
    return x * mask


PERIODIC = ("periodic",) * 4
X_PERIODIC = ("periodic", "periodic", "nrbc", "nrbc")
Y_PERIODIC = ("nrbc", "nrbc", "periodic", "periodic")


# warps of 61 columns, four to a CTA, chunks of 4 rows or more; one to three rows
@pytest.mark.parametrize("bc", [OPEN, PERIODIC, X_PERIODIC, Y_PERIODIC])
@pytest.mark.parametrize("n", [(61, 5), (62, 3), (60, 2), (244, 41), (245, 2), (37, 1), (1, 9), (2, 2), (130, 90),
                               (306, 200)])
def test_fp32_transpose_identity(n, bc):
    """<L x, y> = <x, L^T y>.  Every value of L x and L^T y is a sum of some 40 products of norm about 2 in
    FP32: 40 x 2^-24 x 2 = 5e-6 of |x| |y|, with all errors of one sign."""
    import torch
    from paper_2412_16845_gb300 import gks
    w = _design(n[0], n[1], bc, 1, ((0, 1), (0, 1)), ((0, 1), (0, 1)))
    s = gks.GKSSolver.from_workload(w, precision="fp32")
    gks.gks_set_objective(s.ctx, None, None)
    rng = np.random.default_rng(n[0] + 7 * n[1])
    x, y = (_random_state(s, rng, torch.float32) for _ in range(2))
    gks.gks_load_state(s.ctx, x.data_ptr(), 0)
    s.step(1)
    Lx, LTy = torch.zeros_like(x), torch.zeros_like(x)
    gks.gks_copy_state(s.ctx, Lx.data_ptr())
    gks.gks_adjoint_step(s.ctx, None, None, y.data_ptr(), LTy.data_ptr(), None, False)
    gks.gks_sync(s.ctx)
    s.close()
    a, b = float((Lx.double() * y.double()).sum()), float((x.double() * LTy.double()).sum())
    assert abs(a - b) <= 5e-6 * float(x.double().norm()) * float(y.double().norm()), (a, b)


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("bc", [OPEN, PERIODIC, X_PERIODIC])
@pytest.mark.parametrize("window", [(37, 202, 21, 150), (0, 61, 0, 3), (238, 300, 100, 180), (101, 102, 77, 78)])
def test_windowed_adjoint_is_the_whole_one_inside(window, bc, precision):
    import torch
    from paper_2412_16845_gb300 import gks
    nx, ny = 300, 180
    x0, x1, y0, y1 = window
    w = _design(nx, ny, bc, 1, ((20, 290), (1, 170)), ((30, 250), (0, 130)))
    s = gks.GKSSolver.from_workload(w, precision=precision)
    gks.gks_set_objective(s.ctx, w.probe, w.design)
    dtype = torch.float64 if precision == "fp64" else torch.float32
    rng = np.random.default_rng(2)
    V, lam = (_random_state(s, rng, dtype) for _ in range(2))
    V1 = torch.zeros_like(V)
    gks.gks_step_state_window(s.ctx, V.data_ptr(), V1.data_ptr(), 0, 0, nx, 0, ny)
    out = []
    for win in ((0, nx, 0, ny), window):
        l, g = torch.zeros_like(V), torch.zeros(w.design.size, dtype=torch.float64, device="cuda")
        gks.gks_adjoint_step_window(s.ctx, V.data_ptr(), V1.data_ptr(), lam.data_ptr(), l.data_ptr(), g.data_ptr(),
                                    True, *win)
        gks.gks_load_state(s.ctx, l.data_ptr(), 1)
        out.append((s.read_fields().reshape(3, ny, nx), g.cpu().numpy()))
    s.close()
    (l0, g0), (l1, g1) = out
    inside = (w.design % nx >= x0) & (w.design % nx < x1) & (w.design // nx >= y0) & (w.design // nx < y1)
    tol = 1e-14 if precision == "fp64" else 1e-6
    a, b = (v[:, y0:y1, x0:x1] for v in (l0, l1))
    assert np.abs(a - b).max() <= tol * np.abs(a).max() and np.abs(a).max() > 0
    if inside.any():
        assert np.abs(g0[inside] - g1[inside]).max() <= tol * np.abs(g0).max()
    assert not g1[~inside].any()


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("bc,design,probe,acts", [
    (OPEN, ((40, 60), (30, 50)), ((70, 74), (40, 44)), True),
    (OPEN, ((40, 60), (30, 50)), ((88, 91), (33, 36)), True),             # windows of a few columns
    (OPEN, ((5, 15), (30, 50)), ((105, 108), (40, 44)), False),           # no window at all
    (PERIODIC, ((2, 12), (3, 15)), ((112, 117), (80, 86)), True),         # reached across the sides only
    (X_PERIODIC, ((2, 12), (30, 45)), ((112, 117), (36, 40)), True),
    (Y_PERIODIC, ((50, 70), (1, 9)), ((52, 60), (84, 89)), True),
    (PERIODIC, ((2, 12), (3, 15)), ((58, 62), (43, 47)), False),
])
def test_gradient_is_that_of_whole_grid_steps(bc, design, probe, acts, precision):
    """DesignProblem (recomputed windows, lambda windows) against stored states and whole-grid adjoint steps."""
    import torch
    from paper_2412_16845_gb300 import gks
    from paper_2412_16845_gb300.adjoint import DesignProblem
    steps = 20
    w = _design(120, 90, bc, steps, design, probe)
    p = DesignProblem(w, precision=precision, checkpoint_every=6)
    J, g = p.value_and_grad(w.eps[w.design])
    p.close()
    s = gks.GKSSolver.from_workload(w, precision=precision, c_lattice=1.0)
    gks.gks_set_objective(s.ctx, w.probe, w.design)
    n, _ = gks.gks_state_layout(s.ctx)
    dtype = torch.float64 if precision == "fp64" else torch.float32
    V = [torch.zeros(n, dtype=dtype, device="cuda") for _ in range(steps + 1)]
    gks.gks_copy_state(s.ctx, V[0].data_ptr())
    for k in range(steps):
        s.step(1)
        gks.gks_copy_state(s.ctx, V[k + 1].data_ptr())
    assert gks.gks_objective(s.ctx) == J
    lam, lam2 = torch.zeros_like(V[0]), torch.zeros_like(V[0])
    ref = torch.zeros(w.design.size, dtype=torch.float64, device="cuda")
    gks.gks_adjoint_seed(s.ctx, V[steps].data_ptr(), lam.data_ptr())
    for k in range(steps - 1, -1, -1):
        gks.gks_adjoint_step(s.ctx, V[k].data_ptr(), V[k + 1].data_ptr(), lam.data_ptr(), lam2.data_ptr(),
                             ref.data_ptr(), k >= 1)
        lam, lam2 = lam2, lam
    gks.gks_sync(s.ctx)
    s.close()
    ref = ref.cpu().numpy()
    assert np.linalg.norm(g - ref) <= (1e-13 if precision == "fp64" else 1e-5) * np.linalg.norm(ref)
    assert bool(ref.any()) == acts


def test_a_failed_context_has_no_gradient():
    """With the context's flag set (here by a state that is not finite; a wait that ran out sets it too)
    gks_guard_gradient makes a gradient NaN, and leaves it once fields are written."""
    import torch
    from paper_2412_16845_gb300 import gks
    w = _design(70, 40, OPEN, 1, ((10, 20), (8, 15)), ((30, 31), (5, 6)))
    s = gks.GKSSolver.from_workload(w, precision="fp32")
    g = torch.arange(700, dtype=torch.float64, device="cuda")

    def guarded(n):
        h = g.clone()
        gks.gks_guard_gradient(s.ctx, h.data_ptr(), n)
        torch.cuda.synchronize()
        return h.cpu().numpy()
    assert np.array_equal(guarded(700), np.arange(700.0))
    bad = w.fields0.copy()
    bad[0, 5] = np.inf
    s.write_fields(bad)
    s.step(1)
    h = guarded(513)
    assert np.isnan(h[:513]).all() and np.array_equal(h[513:], np.arange(513.0, 700.0))
    with pytest.raises(gks.GksError):
        gks.gks_sync(s.ctx)
    s.write_fields(w.fields0)
    assert np.array_equal(guarded(700), np.arange(700.0))
    s.close()
