"""The marker kernel's launch shapes (two staging buffers, one, fewer blocks
per SM, the global path) on drops whose patches touch more and more nodes per
face, on grids with and without whole float4 rows: interpolation and probe
traction against the FP64 oracle away from nearest-node switches (bar 1e-5 as
in the parity tests), the fused step's spread against interpolation and spread
called one after the other (the same contributions rounded to the same fixed
point: only the float32 order of the patches' merges differs, 1e-6), and a
second step's clear against a fresh context (the same bound)."""
import numpy as np
import pytest
import torch

from oracle import ibm_oracle as O
from paper_1612_03399_gb300 import _lib
from paper_1612_03399_gb300 import workloads as W

import helpers as H

pytestmark = pytest.mark.gpu
DEV = "cuda"


def drops(count, radius, nx):
    rng = np.random.default_rng(11)
    n = (nx, 64, 60)
    L = tuple(k / 64 for k in n)
    v, t = W.icosphere(3)
    bodies = []
    for _ in range(count):
        c = rng.uniform(0, 1, 3) * L
        bodies.append(W.Body(rest=c + radius / 64 * v @ W.random_rotation(rng), tri=t, origin=c))
    return W.Workload(name="drops", bodies=bodies, grid=W.Grid(n, L),
                      field=W.fourier_modes(6, 3, 1.0, rng))


def zeros(wl):
    n = wl.grid.n
    return tuple(torch.zeros((n[2], n[1], n[0]), device=DEV) for _ in range(3))


# drops, radius in cells, nx, faces per patch: about 8, 8, 22, 38 nodes per face
# (two buffers, one buffer, 16 warps per SM), one block per SM with more rows
# than the footprint record holds, and more rows than any table
@pytest.mark.parametrize("count,radius,nx,patch", [
    (1, 6, 64, 256), (16, 6, 50, 128), (16, 14, 64, 128), (16, 21, 66, 128), (1, 22, 64, 256),
    (2, 22, 61, 256), (1, 29, 64, 256)])
def test_launch_shapes(count, radius, nx, patch, record_error):
    wl = drops(count, radius, nx)
    make = lambda: _lib.Context(wl.bodies, wl.grid, dt=wl.dt, mu=wl.mu, alpha=wl.alpha,
                                marker_patch=patch)
    ctx = make()
    fields = H.fields_for(wl, DEV)
    rng = np.random.default_rng(5)
    x, _ = ctx.init_state()
    v = torch.tensor(rng.uniform(-0.2, 0.2, (3, ctx.V)), dtype=torch.float32, device=DEV)
    U, Fm, Fe = ctx.interpolate(x, v, fields)
    xs = H.to_abs(wl, H.split_state(ctx, wl, x))
    keep = H.tie_mask(wl, xs)
    ob = H.oracle_bodies(wl)
    vs = [torch.tensor(a) for a in H.split_state(ctx, wl, v)]
    out = O.step(ob, xs, vs, tuple(t.double().cpu() for t in fields), H.oracle_params(wl),
                 with_spread=False)
    for name, g in (("U", U), ("F_ext_face", Fe)):
        e = H.rel_l2(g.double().cpu().numpy().T[keep], out[name].numpy()[keep])
        record_error(name, e)
        assert e <= 1e-5, (name, e)
    # the fused step's spread is that of the two calls
    f, f2 = zeros(wl), zeros(wl)
    x1, v1 = torch.empty_like(x), torch.empty_like(v)
    direct = [ctx.counters()["marker_box_fallbacks"]]
    ctx.step(x, v, fields, x1, v1, f)
    direct.append(ctx.counters()["marker_box_fallbacks"])
    ctx.spread(x, Fm, f2)
    direct.append(ctx.counters()["marker_box_fallbacks"])
    same = direct[1] - direct[0] == direct[2] - direct[1]
    assert H.rel_l2(torch.stack(f).cpu(), torch.stack(f2).cpu()) <= (1e-6 if same else 1e-5)
    # a second step elsewhere leaves nothing of the first behind
    y = x + torch.tensor(rng.uniform(-3, 3, (3, 1)) / 64, dtype=torch.float32, device=DEV)
    ctx.step(y, v, fields, x1, v1, f)
    fresh, f2 = make(), zeros(wl)
    fresh.step(y, v, fields, x1, v1, f2)
    ctx.check_device_error()
    fresh.check_device_error()
    assert H.rel_l2(torch.stack(f).cpu(), torch.stack(f2).cpu()) <= 1e-6
