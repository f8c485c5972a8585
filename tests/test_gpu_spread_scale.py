"""The fixed-point scale of the fused spread against the tile-owned spread (38-bit
contributions).  The scale comes from the sum of a block's |c_l F|: its unit is at
most 2^-22 of a mean contribution's bound, a rounding 0.29 units rms, so for supports
whose |phi| is about 0.1 of its bound a field's relative error is about 5e-7: bar
1e-6, also for patches of few, large contributions (faces of several cells), which
the largest contribution alone would scale to 2 .. 3e-6."""
import numpy as np
import pytest
import torch

from paper_1612_03399_gb300 import _lib
from paper_1612_03399_gb300 import workloads as W

import helpers as H

pytestmark = pytest.mark.gpu
DEV = "cuda"


@pytest.mark.parametrize("nx", [128, 126])
@pytest.mark.parametrize("count,radius", [(1, 16), (6, 11), (6, 16), (6, 20)])
def test_scale_of_few_large_drops(count, radius, nx, record_error):
    rng = np.random.default_rng(12)
    n = (nx, 120, 124)
    grid = W.Grid(n, tuple(k / 128 for k in n))
    v, t = W.icosphere(3)
    bodies = []
    for _ in range(count):
        c = rng.uniform(0, 1, 3) * grid.L
        bodies.append(W.Body(rest=c + radius / 128 * v @ W.random_rotation(rng), tri=t, origin=c))
    fields = W.sample_field(W.fourier_modes(8, 3, 1.0, rng), grid, device=DEV)
    out = []
    for variant in (1, 2):
        ctx = _lib.Context(bodies, grid, spread_variant=variant)
        x, _ = ctx.init_state()
        vel = torch.full_like(x, 0.1)
        f = tuple(torch.zeros_like(g) for g in fields)
        ctx.step(x, vel, fields, torch.empty_like(x), torch.empty_like(x), f)
        ctx.check_device_error()
        out.append(torch.stack(f).cpu())
    e = H.rel_l2(*out)
    record_error("f", e)
    assert e <= 1e-6
