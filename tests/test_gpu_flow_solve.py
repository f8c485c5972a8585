"""The real-space viscous solve at the edges of its tiles and walks: each
substep's predictor against the FP64 flow oracle (relative L2 <= 1e-5, the flow
tests' bar), rows of whole float4s and not, fewer cells than a tile and one more,
half widths from 0 up to 8."""
import pytest
import torch

from oracle import ns_oracle as N
from paper_1612_03399_gb300 import _lib
from paper_1612_03399_gb300 import workloads as W

from test_gpu_flow import curl_field, fields_dev, rel, stack_cpu, to_dev

pytestmark = pytest.mark.gpu
DT = torch.float64


@pytest.mark.parametrize("nu", [0.0, 1e-4, 2e-3, 0.01, 0.02, 0.03])
@pytest.mark.parametrize("n", [(17, 18, 19), (20, 17, 33), (33, 32, 31), (36, 33, 70), (64, 65, 17)])
def test_real_space_solves_match_oracle(n, nu, record_error):
    grid = W.Grid(n, tuple(k / 40 for k in n))
    fo = N.Flow(grid.n, grid.L, nu=nu, dt=1e-2)
    u0 = curl_field(grid.n, grid.h, 1)
    p0 = torch.zeros((n[2], n[1], n[0]), dtype=DT)
    fl = _lib.Flow(grid, nu=nu, dt=fo.dt)
    assert any(w >= 0 for w in fl.solve_widths())
    u, p = fields_dev(u0), to_dev(p0)
    uo, Hp = u0.clone(), None
    for l in range(3):
        fl.predict(l, u, p)
        us, Hp = N.predict(fo, l, uo, p0, Hp)
        e = rel(stack_cpu(u), us)
        record_error(f"u{l}", e)
        assert e <= 1e-5, l
        uo = us
