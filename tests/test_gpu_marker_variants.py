"""The marker kernel's variants for many blocks (more than 512 faces per SM:
closed bodies without pressure; everything else) against the variant for few, which
the parity tests hold against the FP64 oracle: one context with all bodies
against contexts with a few of them each.  The variants run the same float32
operations, contracted differently by the compiler: state, interpolation and
loads to 1e-6.  The force fields against the tile-owned spread, an algorithm of its
own with 38-bit contributions (the parity bar 1e-5: the marker kernel rounds a
contribution to 2^-22 of its block's largest).  Drops of 7 cells (two staging
buffers) and 13 (one), rows of whole float4s and not."""
import numpy as np
import pytest
import torch

from paper_1612_03399_gb300 import _lib
from paper_1612_03399_gb300 import workloads as W

import helpers as H

pytestmark = pytest.mark.gpu
DEV = "cuda"


def bodies_of(radius, grid, rng, sheets):
    v, t = W.icosphere(3)
    out = []
    for k in range(64):
        c = rng.uniform(0, 1, 3) * grid.L
        if sheets and k % 16 == 0:
            sv, st, rim = W.elliptic_sheet(radius / 128, 0.7 * radius / 128, 1500, rng, jitter=0.1)
            out.append(W.Body(rest=c + sv, tri=st, origin=c, closed=False, clamped=rim, ks=5.0,
                              kb=0.3, kA=0.0, kv=0.0, spring_model=1))
        else:
            out.append(W.Body(rest=c + radius / 128 * v @ W.random_rotation(rng), tri=t, origin=c))
    return out


@pytest.mark.parametrize("sheets", [False, True])
@pytest.mark.parametrize("radius,nx", [(7, 128), (13, 128), (7, 126), (13, 126)])
def test_many_blocks_match_few(radius, nx, sheets, record_error):
    rng = np.random.default_rng(8)
    n = (nx, 120, 124)
    grid = W.Grid(n, tuple(k / 128 for k in n))
    bodies = bodies_of(radius, grid, rng, sheets)
    fields = W.sample_field(W.fourier_modes(8, 3, 1.0, rng), grid, device=DEV)
    p = W.sample_pressure(W.pressure_modes(8, 3, 1.0, rng), grid, device=DEV) if sheets else None
    kw = dict(dt=1e-3)
    ctx = _lib.Context(bodies, grid, **kw)
    assert ctx.F > 512 * torch.cuda.get_device_properties(0).multi_processor_count
    x, _ = ctx.init_state()
    v = torch.tensor(rng.uniform(-0.2, 0.2, (3, ctx.V)), dtype=torch.float32, device=DEV)
    a = torch.tensor(rng.uniform(-1, 1, (3, ctx.V)), dtype=torch.float32, device=DEV) if sheets else None
    zeros = lambda: tuple(torch.zeros_like(g) for g in fields)

    def run(c, x, v, a, f):
        out = [torch.empty_like(x), torch.empty_like(x)]
        c.step(x, v, fields, out[0], out[1], f, p=p, accel=a)
        out += list(c.interpolate(x, v, fields, p=p, accel=a))
        c.check_device_error()
        return out

    f = zeros()
    whole = run(ctx, x, v, a, f)
    parts, at = [], 0
    for k in range(0, len(bodies), 8):
        c = _lib.Context(bodies[k:k + 8], grid, **kw)
        s = slice(at, at + c.V)
        at += c.V
        parts.append(run(c, x[:, s].contiguous(), v[:, s].contiguous(),
                         a[:, s].contiguous() if sheets else None, zeros()))
    for i, name in enumerate(("x", "v", "U", "F_marker", "F_ext")):
        e = H.rel_l2(whole[i].cpu(), torch.cat([q[i] for q in parts], 1).cpu())
        record_error(name, e)
        assert e <= 1e-6, name
    f2 = zeros()
    run(_lib.Context(bodies, grid, spread_variant=2, **kw), x, v, a, f2)
    e = H.rel_l2(torch.stack(f).cpu(), torch.stack(f2).cpu())
    record_error("f", e)
    assert e <= 1e-5


@pytest.mark.parametrize("radius", [7, 13])
def test_coupled_forcing_matches_tile_spread(radius):
    """The coupled step's forcing with cached row tables against the tile-owned
    spread, an algorithm of its own (parity bar 1e-5)."""
    rng = np.random.default_rng(9)
    n = (128, 120, 124)
    grid = W.Grid(n, tuple(k / 128 for k in n))
    bodies = bodies_of(radius, grid, rng, False)
    u0 = W.sample_field(W.fourier_modes(8, 3, 1.0, rng), grid, device=DEV)
    out = []
    for variant in (1, 2):
        ctx = _lib.Context(bodies, grid, dt=1e-3, mu=0.01, spread_variant=variant)
        flow = _lib.Flow(grid, nu=0.01, dt=1e-3)
        x, v = ctx.init_state()
        u, p = tuple(g.clone() for g in u0), torch.zeros_like(u0[0])
        f = tuple(torch.zeros_like(g) for g in u0)
        x1, v1 = torch.empty_like(x), torch.empty_like(v)
        flow.step(u, p, ctx=ctx, x=x, v=v, x_out=x1, v_out=v1, f=f)
        ctx.check_device_error()
        out.append([torch.stack(u).cpu(), torch.stack(f).cpu(), v1.cpu()])
        flow.close()
    for a, b in zip(*out):
        assert H.rel_l2(a, b) <= 1e-5
