"""The viscous solve on grids with one direction shorter than the filters the
others ask for: the real-space solve is taken only where 2W + 1 <= n_d holds in
every direction for the W it uses (the widths are checked before anything runs),
and each substep's predictor agrees with the FP64 flow oracle (relative L2 <=
1e-5, the flow tests' bar)."""
import pytest
import torch

from oracle import ns_oracle as N
from paper_1612_03399_gb300 import _lib
from paper_1612_03399_gb300 import workloads as W

from test_gpu_flow import curl_field, documented_widths, fields_dev, rel, stack_cpu, to_dev

pytestmark = pytest.mark.gpu
DT = torch.float64


@pytest.mark.parametrize("nu", [0.0, 0.002, 0.02, 0.03])
@pytest.mark.parametrize("n", [(64, 64, 5), (40, 36, 7), (5, 40, 36), (40, 9, 36), (64, 20, 11),
                               (17, 15, 13)])
def test_short_directions_match_oracle(n, nu, record_error):
    grid = W.Grid(n, tuple(k / 40 for k in n))
    fo = N.Flow(grid.n, grid.L, nu=nu, dt=1e-2)
    fl = _lib.Flow(grid, nu=nu, dt=fo.dt)
    own = documented_widths(grid, nu, fo.dt)   # the largest of the directions' own widths
    assert fl.solve_widths() == tuple(w if 2 * w + 1 <= min(n) else -1 for w in own)
    u0 = curl_field(grid.n, grid.h, 1)
    p0 = torch.zeros((n[2], n[1], n[0]), dtype=DT)
    u, p = fields_dev(u0), to_dev(p0)
    uo, Hp = u0.clone(), None
    for l in range(3):
        fl.predict(l, u, p)
        us, Hp = N.predict(fo, l, uo, p0, Hp)
        e = rel(stack_cpu(u), us)
        record_error(f"u{l}", e)
        assert e <= 1e-5, l
        uo = us
