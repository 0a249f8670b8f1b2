"""The host side of DesignProblem without a GPU (tests/fake_cuda.py): streams, errors, windows."""
import numpy as np
import pytest

from paper_2412_16845_gb300 import workloads as wl
from tests.fake_cuda import _fake_library, fake, fake_torch  # noqa: F401


def _workload(nx=40, ny=32, bc=("nrbc",) * 4, steps=20, design=((8, 16), (6, 14)), probe=((24, 27), (15, 18))):
    def cells(b):
        return (np.arange(*b[1])[:, None] * nx + np.arange(*b[0])[None, :]).ravel()
    return wl.CartWorkload(name="design", dim=2, n=(nx, ny), lo=(0.0, 0.0), hi=(1.0, ny / nx), bc=bc, cfl=0.5,
                           steps=steps, eps=np.full(nx * ny, 2.0), mu=None, fields0=np.zeros((3, nx * ny)),
                           jz_mask=None, src=None, c_lattice=1.0, probe=cells(probe), design=cells(design))


def _problem(w, **kw):
    from paper_2412_16845_gb300.adjoint import DesignProblem
    return DesignProblem(w, **kw)


@pytest.mark.parametrize("own", [False, True])
def test_buffers_live_on_the_problems_stream(fake_torch, own):
    """Every buffer that kernels on the problem's stream write is made (and filled) on that stream, and the
    caller's stream waits for the gradient, whichever stream is current at each call."""
    t = fake_torch
    side = t.Stream(t, "side")
    p = _problem(_workload(), **({"stream": side} if own else {}))
    mine = "side" if own else "caller"
    for name in ("caller", "another"):
        t.current = t.Stream(t, name)
        p.forward(p.base_eps[p.design])
        g = p.backward()
        assert set(t.made) == {mine}, t.made
        assert t.current.name == name
        if name != mine:
            assert (name, mine) in t.waits and name in g.streams
    p.close()


@pytest.mark.parametrize("kernel", [b"adjoint_tau0_kernel", b"cart2d_tau0_kernel"])
def test_a_wait_that_ran_out_in_backward_is_an_error(fake, fake_torch, kernel):
    """The lambda march and the recomputed steps have bounded waits; a wrong gradient is not returned."""
    from paper_2412_16845_gb300 import gks
    p = _problem(_workload(nx=400, ny=300))           # (smaller grids recompute without waits)
    p.forward(p.base_eps[p.design])
    fake.give_up(kernel)
    with pytest.raises(gks.GksError) as e:
        p.backward()
    assert e.value.status == gks.GKS_E_TIMEOUT
    p.close()


@pytest.mark.parametrize("late", [False, True])
def test_autograd_reports_a_wait_that_ran_out(fake, fake_torch, late):
    from paper_2412_16845_gb300 import adjoint, gks
    p = _problem(_workload(nx=400, ny=300))
    e = fake_torch.tensor(p.base_eps[p.design], requires_grad=True)
    J = adjoint._autograd_class().apply(e, p)
    if not late:
        J.backward()
        assert e.grad.shape == e.shape
    else:
        fake.give_up(b"adjoint_tau0_kernel")
        with pytest.raises(gks.GksError) as err:
            J.backward()
        assert err.value.status == gks.GKS_E_TIMEOUT
    p.close()


@pytest.mark.parametrize("bc", [("nrbc",) * 4, ("periodic",) * 4])
def test_an_empty_probe_has_a_zero_gradient(fake, fake_torch, bc):
    """gks_set_objective takes an empty probe: J = 0, and no lambda acts anywhere."""
    w = _workload(bc=bc)
    w.probe = np.zeros(0, dtype=np.int64)
    p = _problem(w)
    J = p.forward(p.base_eps[p.design])
    g = p.backward()
    assert J == 0.0 and g.t.shape == (p.design.size,) and not g.t.any()
    p.close()
