"""The Poisson solve with its z direction by recursions: projections against the
FP64 flow oracle (the flow tests' bars: velocity 1e-5, pressure_ok) for column
lengths around the segments' 16 entries up to the longest (511, 512), and
for a thin domain (by transforms)."""
import pytest
import torch

from oracle import ns_oracle as N
from paper_1612_03399_gb300 import _lib
from paper_1612_03399_gb300 import workloads as W

from test_gpu_flow import curl_field, fields_dev, pressure_ok, rel, stack_cpu, to_dev

pytestmark = pytest.mark.gpu
DT = torch.float64


@pytest.mark.parametrize("n", [(8, 6, 4), (9, 5, 15), (8, 8, 16), (7, 6, 17), (20, 33, 144), (8, 6, 511),
                               (6, 8, 512), (120, 6, 8)])
def test_projection_matches_oracle(n, record_error):
    grid = W.Grid(n, tuple(k / 40 for k in n))
    fo = N.Flow(grid.n, grid.L, nu=0.02, dt=1e-2)
    g = torch.Generator().manual_seed(4)
    u0 = torch.stack([torch.randn((n[2], n[1], n[0]), generator=g, dtype=DT) for _ in range(3)])
    u0 = stack_cpu(fields_dev(u0))
    p0 = torch.zeros((n[2], n[1], n[0]), dtype=DT)
    fl = _lib.Flow(grid, nu=fo.nu, dt=fo.dt)
    for l in range(3):
        u, p = fields_dev(u0), to_dev(p0)
        fl.predict(l, fields_dev(0 * u0), to_dev(p0))   # the substep order
        fl.project(l, u, p)
        uo, po = N.project(fo, l, u0, p0)
        eu = rel(stack_cpu(u), uo)
        ep, pok = pressure_ok(p.double().cpu(), po, float(u0.abs().max()), min(grid.h), fo.dt, [l])
        record_error(f"u{l}", eu)
        record_error(f"p{l}", ep)
        assert eu <= 1e-5 and pok, (l, eu, ep)
