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
    assert "guard_gradient_kernel" in fake.launched()[-1]    # for a gradient that is used without the check
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


def _context(precision="fp32", n=(40, 30), **kw):
    from paper_2412_16845_gb300 import gks
    s = gks.GKSSolver(gks.SolverSpec(dim=len(n), n=n, lo=(0.0,) * len(n), hi=(1.0,) * len(n),
                                     bc=kw.pop("bc", ("nrbc",) * (2 * len(n))), cfl=0.3, precision=precision, **kw))
    _, nbytes = gks.gks_state_layout(s.ctx)
    bufs = [np.zeros(nbytes + 32, dtype=np.uint8) for _ in range(4)]
    return s, bufs, [(b.ctypes.data + 15) // 16 * 16 for b in bufs]


BAD_WINDOWS = [(-1, 4, 0, 4), (0, 41, 0, 4), (0, 4, -1, 4), (0, 4, 0, 31), (5, 5, 0, 4), (6, 5, 0, 4), (0, 4, 7, 7)]


@pytest.mark.parametrize("window", BAD_WINDOWS)
def test_windows_outside_the_grid_are_refused(fake, window):
    from paper_2412_16845_gb300 import gks
    s, keep, (a, b, c, d) = _context()
    gks.gks_set_objective(s.ctx, [3], [4])
    with pytest.raises(gks.GksError) as e:
        gks.gks_step_state_window(s.ctx, a, b, 0, *window)
    assert e.value.status == gks.GKS_E_ARG
    with pytest.raises(gks.GksError) as e:
        gks.gks_adjoint_step_window(s.ctx, a, b, c, d, a, True, *window)
    assert e.value.status == gks.GKS_E_ARG
    assert not fake.launched()[1:]                     # (the fill of eps at creation)
    s.close()


def test_arguments_of_the_window_calls(fake):
    from paper_2412_16845_gb300 import gks
    s, keep, (a, b, c, d) = _context()
    gks.gks_set_objective(s.ctx, [3], [4])
    win = (0, 40, 0, 30)
    for src, dst, step in ((None, b, 0), (a, None, 0), (a, a, 0), (a, b, -1), (a + 2, b, 0), (a, b + 1, 0)):
        with pytest.raises(gks.GksError) as e:
            gks.gks_step_state_window(s.ctx, src, dst, step, *win)
        assert e.value.status == gks.GKS_E_ARG
    for vn, vn1, lin, lout, g in ((None, b, c, d, a), (a, None, c, d, a), (a, b, None, d, a), (a, b, c, None, a),
                                  (a, b, c, c, a), (a, b, c, d, None), (a, b, c + 2, d, a)):
        with pytest.raises(gks.GksError) as e:
            gks.gks_adjoint_step_window(s.ctx, vn, vn1, lin, lout, g, True, *win)
        assert e.value.status == gks.GKS_E_ARG
    s.close()
    # what the whole-grid calls refuse
    for kw, step_too in (({"n": (8, 8, 8)}, True), ({"phm": (0.0, 1.0)}, True), ({"limiter": "vanleer"}, False),
                         ({"bc": ("pec", "pec", "nrbc", "nrbc")}, False)):
        s, keep, (a, b, c, d) = _context(**kw)
        with pytest.raises(gks.GksError) as e:
            gks.gks_adjoint_step_window(s.ctx, a, b, c, d, a, False, 0, 4, 0, 4)
        assert e.value.status == gks.GKS_E_UNSUPPORTED
        if step_too:
            with pytest.raises(gks.GksError) as e:
                gks.gks_step_state_window(s.ctx, a, b, 0, 0, 4, 0, 4)
            assert e.value.status == gks.GKS_E_UNSUPPORTED
        s.close()


def _brute_lambda(p, w):
    """Cells where lambda^n is not zero and acts on the gradient, by dilating masks two cells a step."""
    nx, ny = w.n
    per = (w.bc[0] == "periodic", w.bc[2] == "periodic")

    def grow(m):
        for axis, wrap in ((1, per[0]), (0, per[1])):
            acc = m.copy()
            for k in (1, 2):
                for sgn in (1, -1):
                    r = np.roll(m, sgn * k, axis=axis)
                    if not wrap:
                        idx = [slice(None)] * 2
                        idx[axis] = slice(0, k) if sgn > 0 else slice(-k, None)
                        r[tuple(idx)] = False
                    acc |= r
            m = acc
        return m
    lam, act = [None] * (p.N + 1), [None] * (p.N + 1)
    m = np.zeros((ny, nx), bool)
    m.ravel()[w.probe] = True
    for n in range(p.N, -1, -1):
        lam[n] = m
        m = grow(m)
    # lambda^n acts on the gradient through lambda^k, k <= n, beside a design cell (k's step reads two cells)
    a = np.zeros((ny, nx), bool)
    a.ravel()[w.design] = True
    for n in range(0, p.N + 1):
        a = grow(a) if n else a
        act[n] = a
    return lam, act


@pytest.mark.parametrize("bc", [("nrbc",) * 4, ("periodic",) * 4, ("periodic", "periodic", "nrbc", "nrbc")])
@pytest.mark.parametrize("design,probe", [
    (((8, 16), (6, 14)), ((24, 27), (15, 18))), (((1, 4), (2, 5)), ((36, 39), (28, 31))),
    (((30, 40), (0, 3)), ((0, 2), (0, 2))), (((5, 6), (5, 6)), ((33, 34), (25, 26))),
])
def test_lambda_windows_hold_every_cell_that_acts(fake_torch, bc, design, probe):
    w = _workload(bc=bc, steps=14, design=design, probe=probe)
    p = _problem(w)
    lam, act = _brute_lambda(p, w)
    for n in range(p.N):
        need = lam[n] & act[n]
        win = p._lambda_window(n)
        if win is None:
            assert not need.any(), n
            continue
        x0, x1, y0, y1 = win
        need[y0:y1, x0:x1] = False
        assert not need.any(), (n, win)
    p.close()
