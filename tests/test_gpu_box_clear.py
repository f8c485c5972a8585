"""The clear of patches that took the global path (a bounding box each, widened to
whole float4s where the rows allow): a step elsewhere leaves in the force fields
exactly what a fresh context leaves there (float32 order of the atomics: 1e-6), for
boxes across the periodic boundary, rows of whole float4s and not, boxes as wide as
the grid, and fields that start off a 16-byte boundary."""
import numpy as np
import pytest
import torch

from paper_1612_03399_gb300 import _lib
from paper_1612_03399_gb300 import workloads as W

import helpers as H

pytestmark = pytest.mark.gpu
DEV = "cuda"


@pytest.mark.parametrize("nx,ny,nz,radius,off", [
    (128, 96, 100, 38, 0), (126, 96, 100, 38, 0), (125, 97, 99, 30, 0), (64, 60, 62, 45, 0),
    (61, 60, 62, 45, 0), (128, 96, 100, 38, 1)])
def test_boxes_are_cleared(nx, ny, nz, radius, off):
    rng = np.random.default_rng(4)
    n = (nx, ny, nz)
    grid = W.Grid(n, tuple(k / 128 for k in n))
    v, t = W.icosphere(3)
    bodies = []
    for c in ((0.05, 0.1, 0.9), (0.6, 0.5, 0.5)):
        c = np.array(c) * grid.L
        bodies.append(W.Body(rest=c + radius / 128 * v @ W.random_rotation(rng), tri=t, origin=c))
    fields = W.sample_field(W.fourier_modes(6, 3, 1.0, rng), grid, device=DEV)

    def zeros():
        size = nx * ny * nz
        return tuple(torch.zeros(size + 4, device=DEV)[off:off + size].view(nz, ny, nx)
                     for _ in range(3))

    ctx, fresh = (_lib.Context(bodies, grid) for _ in range(2))
    x, _ = ctx.init_state()
    vel = torch.tensor(rng.uniform(-0.2, 0.2, tuple(x.shape)), dtype=torch.float32, device=DEV)
    y = x + torch.tensor(rng.uniform(-9, 9, (3, 1)) / 128, dtype=torch.float32, device=DEV)
    x1, v1, f, f2 = torch.empty_like(x), torch.empty_like(x), zeros(), zeros()
    ctx.step(x, vel, fields, x1, v1, f)
    assert ctx.counters()["marker_box_fallbacks"] > 0
    ctx.step(y, vel, fields, x1, v1, f)
    fresh.step(y, vel, fields, x1, v1, f2)
    ctx.check_device_error()
    fresh.check_device_error()
    assert H.rel_l2(torch.stack(f).cpu(), torch.stack(f2).cpu()) <= 1e-6
    assert bool(((torch.stack(f) == 0) == (torch.stack(f2) == 0)).all())
