"""The time of a 3-D cleaning step on grids that end inside a tile: open and closed sides cost about what
periodic sides do (copies for unused columns past an open side once made the step twice as long)."""
import numpy as np
import pytest

from paper_2412_16845_gb300 import workloads as wl
from paper_2412_16845_gb300.gks import GKSSolver

pytestmark = pytest.mark.gpu


def _time(n, side):
    import torch
    rng = np.random.default_rng(2)
    cells = int(np.prod(n))
    w = wl.CartWorkload(name="sides", dim=3, n=n, lo=(0.0,) * 3, hi=tuple(v / n[0] for v in n), bc=(side,) * 6,
                        cfl=0.25, steps=0, eps=rng.uniform(1.0, 4.0, cells), mu=None,
                        fields0=0.1 * rng.standard_normal((8, cells)), jz_mask=None, src=None, c_lattice=0.0)
    w.phm = (0.7, 1.3)
    s = GKSSolver.from_workload(w, precision="fp32", stream=torch.cuda.current_stream().cuda_stream)
    s.step(10)
    best = 1e9
    for _ in range(5):
        a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
        torch.cuda.synchronize()
        a.record()
        s.step(50)
        b.record()
        torch.cuda.synchronize()
        best = min(best, a.elapsed_time(b))
    s.close()
    return best


@pytest.mark.parametrize("n", [(32, 32, 32), (100, 90, 80), (8, 8, 8)])
def test_sides_cost_alike(n):
    periodic = _time(n, "periodic")
    assert _time(n, "nrbc") <= 1.4 * periodic
    assert _time(n, "pec") <= 1.6 * periodic            # plus the mirror images
