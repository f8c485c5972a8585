"""The tile-owned spread where a tile's nodes meet themselves: grids from the
smallest period, one node longer than a tile and with partial last tiles in
every direction, markers in every cell and across the seams, against the FP64
oracle away from nearest-node switches (bar 1e-5 as in the parity tests), and a
clear-mode step against a fresh context (bitwise, as documented)."""
import numpy as np
import pytest
import torch

from oracle import ibm_oracle as O
from paper_1612_03399_gb300 import _lib
from paper_1612_03399_gb300 import workloads as W

import helpers as H

pytestmark = pytest.mark.gpu
DEV = "cuda"


@pytest.mark.parametrize("n", [(4, 4, 4), (16, 8, 8), (17, 9, 9), (18, 10, 10), (15, 7, 33),
                               (32, 5, 17), (33, 24, 4)])
def test_tile_spread_edges(n, record_error):
    rng = np.random.default_rng(2)
    L = tuple(k / max(n) for k in n)
    v, t = W.icosphere(2)
    bodies = []
    for _ in range(3):
        c = rng.uniform(0, 1, 3) * L
        bodies.append(W.Body(rest=c + 0.45 * v * np.array(L), tri=t, origin=c))
    wl = W.Workload(name="edges", bodies=bodies, grid=W.Grid(n, L), field={"kind": "uniform", "U": (0.1, -0.2, 0.3)})
    make = lambda: _lib.Context(wl.bodies, wl.grid, dt=wl.dt, mu=wl.mu, alpha=wl.alpha,
                                spread_variant=2)
    zeros = lambda: tuple(torch.zeros((n[2], n[1], n[0]), device=DEV) for _ in range(3))
    ctx = make()
    x, v0 = ctx.init_state()
    xs = H.to_abs(wl, H.split_state(ctx, wl, x))
    keep = H.tie_mask(wl, xs)
    Fm = rng.standard_normal((ctx.F, 3)) * keep[:, None]
    F = torch.tensor(np.ascontiguousarray(Fm.T), dtype=torch.float32, device=DEV)
    f = zeros()
    ctx.spread(x, F, f)
    P, A = [], []
    for i, b in enumerate(H.oracle_bodies(wl)):
        C, _, Al = O.face_geometry(xs[i], b.tri)
        P.append(C)
        A.append(Al)
    ref = O.spread(torch.tensor(F.double().cpu().numpy().T), torch.cat(P), torch.cat(A), wl.grid.n,
                   wl.grid.h, wl.alpha)
    e = H.rel_l2(torch.stack(f).double().cpu(), ref)
    record_error("f", e)
    assert e <= 1e-5
    # clear mode: a step here, then elsewhere, leaves what a fresh context leaves there
    fields = W.sample_field(wl.field, wl.grid, device=DEV)
    y = x + torch.tensor(rng.uniform(-1, 1, (3, 1)) * L[0], dtype=torch.float32, device=DEV)
    x1, v1 = torch.empty_like(x), torch.empty_like(x)
    f, f2 = zeros(), zeros()
    ctx.step(x, v0, fields, x1, v1, f)
    ctx.step(y, v0, fields, x1, v1, f)
    fresh = make()
    fresh.step(y, v0, fields, x1, v1, f2)
    ctx.check_device_error()
    fresh.check_device_error()
    assert all(torch.equal(a, b) for a, b in zip(f, f2))
