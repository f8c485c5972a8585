"""The viscous solve by recursions along the lines: each substep's predictor
against the FP64 flow oracle (relative L2 <= 1e-5, the flow tests' bar) over line
lengths from the smallest to ragged ones longer than a block's tile.  At nu = 0.5
every substep takes the recursions, at 5.0 (c = 21, 5, 13) substeps 0 and 2 are
past their range and take the transforms."""
import pytest
import torch

from oracle import ns_oracle as N
from paper_1612_03399_gb300 import _lib
from paper_1612_03399_gb300 import workloads as W

from test_gpu_flow import curl_field, fields_dev, rel, stack_cpu, to_dev

pytestmark = pytest.mark.gpu
DT = torch.float64


@pytest.mark.parametrize("nu", [0.5, 5.0])
@pytest.mark.parametrize("n", [(4, 5, 6), (9, 7, 4), (33, 40, 65), (40, 36, 20), (70, 31, 12)])
def test_line_solves_match_oracle(n, nu, record_error):
    grid = W.Grid(n, tuple(k / 40 for k in n))
    fo = N.Flow(grid.n, grid.L, nu=nu, dt=1e-2)
    u0 = curl_field(grid.n, grid.h, 1)
    p0 = torch.zeros((n[2], n[1], n[0]), dtype=DT)
    fl = _lib.Flow(grid, nu=nu, dt=fo.dt)
    u, p = fields_dev(u0), to_dev(p0)
    uo, Hp = u0.clone(), None
    for l in range(3):
        fl.predict(l, u, p)
        us, Hp = N.predict(fo, l, uo, p0, Hp)
        e = rel(stack_cpu(u), us)
        record_error(f"u{l}", e)
        assert e <= 1e-5, l
        uo = us
