"""The projection on stretched cells and short columns against the FP64 flow
oracle.  The float32 error of u is that of a handful of roundings per direction
(the differences, two transforms of log2 n stages, the column solve), well below
sixteen units of 2^-24 of |u| whatever the cells' shape: bar 1e-6, on a random
field, where every wavelength counts alike."""
import pytest
import torch

from oracle import ns_oracle as N
from paper_1612_03399_gb300 import _lib
from paper_1612_03399_gb300 import workloads as W

from test_gpu_flow import fields_dev, rel, stack_cpu, to_dev

pytestmark = pytest.mark.gpu
DT = torch.float64


@pytest.mark.parametrize("n,cell", [
    ((32, 32, 32), (1, 1, 1)), ((32, 32, 32), (1, 1, 4)), ((32, 32, 32), (1, 1, 16)),
    ((32, 30, 33), (1, 1, 64)), ((24, 26, 40), (4, 1, 1)), ((24, 26, 40), (1, 8, 3)),
    ((33, 32, 31), (1, 1, 0.25)), ((4, 4, 4), (1, 1, 1)), ((4, 5, 6), (1, 1, 30)),
    ((12, 10, 512), (1, 1, 2)), ((8, 64, 50), (1, 1, 1.3))])
def test_projection_on_stretched_cells(n, cell, record_error):
    grid = W.Grid(n, tuple(k * c / 40 for k, c in zip(n, cell)))
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
        uo, _ = N.project(fo, l, u0, p0)
        e = rel(stack_cpu(u), uo)
        record_error(f"u{l}", e)
        assert e <= 1e-6, l
