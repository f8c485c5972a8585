"""Widths of the MLS weight past any use: from alpha = 1e6 on the weights of a
support are equal to float32 rounding, so wider ones give the same interpolation,
traction and force fields (1e-6), up to widths whose exponent no longer has a
float32 or float64 value."""
import numpy as np
import pytest
import torch

from paper_1612_03399_gb300 import _lib
from paper_1612_03399_gb300 import workloads as W

import helpers as H

pytestmark = pytest.mark.gpu
DEV = "cuda"


@pytest.mark.parametrize("alpha", [1e10, 1e18, 1e20, 1e160])
def test_wide_weights(alpha):
    c = np.array([0.5, 0.5, 0.5])
    v, t = W.icosphere(3)
    bodies = [W.Body(rest=c + 0.2 * v, tri=t, origin=c)]
    grid = W.Grid((48, 40, 44), (1.0, 40 / 48, 44 / 48))
    fields = W.sample_field(W.fourier_modes(6, 3, 1.0, np.random.default_rng(2)), grid, device=DEV)
    out = []
    for a in (1e6, alpha):
        ctx = _lib.Context(bodies, grid, alpha=a)
        x, vel = ctx.init_state()
        U, Fm, Fe = ctx.interpolate(x, vel, fields)
        f = tuple(torch.zeros_like(g) for g in fields)
        ctx.spread(x, Fm, f)
        ctx.check_device_error()
        out.append([t.double().cpu() for t in (U, Fm, Fe, torch.stack(f))])
    for a, b in zip(*out):
        assert bool(torch.isfinite(b).all()) and H.rel_l2(b, a) <= 1e-6
