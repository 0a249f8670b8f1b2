"""Steps over the whole grid, steps over a window and steps between a caller's states give the same bits, on
grids that take several steps per launch too: a state recomputed by windowed steps is the state that the
forward pass had."""
import numpy as np
import pytest

from paper_2412_16845_gb300 import workloads as wl
from paper_2412_16845_gb300 import gks
from paper_2412_16845_gb300.gks import GKSSolver

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2412_16845_gb300 import build
    build.build()


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("n,bc,limiter,source", [
    ((64, 64), "pppp", None, False), ((100, 100), "nnnn", None, True), ((41, 77), "mmnn", None, True),
    ((5, 3), "nmpp", None, False), ((33, 20), "nnmm", "vanleer", True), ((3, 50), "pppp", "vanleer", False),
    ((130, 90), "ppnn", None, True), ((500, 300), "nnnn", None, True),
])
def test_windowed_steps_repeat_the_bits(n, bc, limiter, source, precision):
    import torch
    rng = np.random.default_rng(n[0])
    cells = n[0] * n[1]
    mask = np.where(rng.random(cells) < 0.05, rng.uniform(-3, 3, cells), 0.0) if source else None
    sides = tuple({"n": "nrbc", "p": "periodic", "m": "pec"}[b] for b in bc)
    w = wl.CartWorkload(name="bits", dim=2, n=n, lo=(0.0, 0.0), hi=(1.0, 1.2 * n[1] / n[0]), bc=sides, cfl=0.4,
                        steps=0, eps=rng.uniform(1.0, 4.0, cells), mu=None,
                        fields0=rng.standard_normal((3, cells)), jz_mask=mask, src=(1.0, 20.0, 0.02, 0.02),
                        c_lattice=0.0, limiter=limiter)
    s = GKSSolver.from_workload(w, precision=precision)
    size, _ = gks.gks_state_layout(s.ctx)
    dtype = torch.float64 if precision == "fp64" else torch.float32
    buf = [torch.zeros(size, dtype=dtype, device="cuda") for _ in range(2)]
    gks.gks_copy_state(s.ctx, buf[0].data_ptr())
    s.step(13)
    whole = s.read_fields()
    s.write_fields(w.fields0)
    gks.gks_step_window(s.ctx, 13, 0, n[0], 0, n[1])
    assert np.array_equal(s.read_fields(), whole)
    for k in range(13):
        gks.gks_step_state_window(s.ctx, buf[k % 2].data_ptr(), buf[1 - k % 2].data_ptr(), k, 0, n[0], 0, n[1])
    gks.gks_load_state(s.ctx, buf[1].data_ptr(), 13)
    assert np.array_equal(s.read_fields(), whole)
    if n[0] > 20 and n[1] > 16:                         # one step over an inner window
        x0, x1, y0, y1 = 5, n[0] - 7, 3, n[1] - 4
        s.write_fields(w.fields0)
        gks.gks_copy_state(s.ctx, buf[0].data_ptr())
        s.step(1)
        one = s.read_fields().reshape(3, n[1], n[0])[:, y0:y1, x0:x1]
        gks.gks_step_state_window(s.ctx, buf[0].data_ptr(), buf[1].data_ptr(), 0, x0, x1, y0, y1)
        gks.gks_load_state(s.ctx, buf[1].data_ptr(), 1)
        assert np.array_equal(s.read_fields().reshape(3, n[1], n[0])[:, y0:y1, x0:x1], one)
    s.write_fields(w.fields0)
    for _ in range(13):
        s.step(1)
    assert np.array_equal(s.read_fields(), whole)
    s.close()
