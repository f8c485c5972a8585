"""The flow kernels that take four cells in x per thread (whole float4 rows,
16-byte aligned fields) against the one-cell kernels, which the same grid takes
when a field starts 4 bytes off a 16-byte boundary: the velocity after every
predictor and projection, forced and not, on grids from a single quad per row,
with heights that leave partial columns.  Both do the same float32 stencils, so
they differ by the rounding of a few operations: 1e-6 relative.  (The pressure
enters the next predictor; against float64 it is held in the flow tests.)"""
import pytest
import torch

from paper_1612_03399_gb300 import _lib
from paper_1612_03399_gb300 import workloads as W

pytestmark = pytest.mark.gpu
DEV = "cuda"


def field(n, g, off):
    """A contiguous random field that starts `off` floats past an aligned address."""
    t = torch.empty(n[0] * n[1] * n[2] + 4, device=DEV)[off:off + n[0] * n[1] * n[2]]
    t.copy_(torch.randn(t.shape, generator=g, device="cpu"))
    return t.view(n[2], n[1], n[0])


def fields(n, off, seed=3):
    g = torch.Generator().manual_seed(seed)
    return [field(n, g, off) for _ in range(7)]


def rel(a, b):
    a, b = (torch.stack(list(t)).double() for t in (a, b))
    return float((a - b).norm() / b.norm())


@pytest.mark.parametrize("n", [(4, 4, 4), (8, 5, 4), (36, 7, 33), (40, 36, 20), (128, 9, 11)])
@pytest.mark.parametrize("forced", [False, True])
def test_quads_match_single_cells(n, forced):
    L = tuple(k / max(n) for k in n)
    dt, nu = 0.05 / max(n), 0.01
    out = []
    for off in (0, 1):
        flow = _lib.Flow(W.Grid(n, L), nu=nu, dt=dt)
        u, v, w, p, fx, fy, fz = fields(n, off)
        assert (u.data_ptr() % 16 == 0) == (off == 0)
        states = []
        for l in range(3):
            flow.predict(l, (u, v, w), p)
            states.append([t.clone() for t in (u, v, w)])
            flow.project(l, (u, v, w), p, f=(fx, fy, fz) if forced else None,
                         f_scale=dt if forced else 0.0)
            states.append([t.clone() for t in (u, v, w)])
        out.append(states)
    for a, b in zip(*out):
        assert rel(a, b) <= 1e-6
