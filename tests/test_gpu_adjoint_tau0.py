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
