"""Force patches around the largest float4 layout a block can hold beside its
static shared memory (patches of 684 vertices of this body need 227 KB for it):
created, with the layout that fits, and internal forces against the FP64 oracle
(bar 1e-5 as in the parity tests); past what the adjoint's narrow layout can hold
the library says so."""
import numpy as np
import pytest

from paper_1612_03399_gb300 import _lib
from paper_1612_03399_gb300 import workloads as W

import helpers as H

pytestmark = pytest.mark.gpu


def scene():
    c = np.array([0.5, 0.5, 0.5])
    v, t = W.icosphere(4)
    return W.Workload(name="limits", bodies=[W.Body(rest=c + 0.2 * v, tri=t, origin=c)],
                      grid=W.Grid((32, 32, 32)), field={"kind": "shear"})


@pytest.mark.parametrize("patch", [680, 683, 684, 685, 690])
def test_forces_at_the_limit(patch, record_error):
    wl = scene()
    ctx = _lib.Context(wl.bodies, wl.grid, patch_size=patch)
    x = H.state_tensor(wl, H.rel_positions(wl, W.perturb_positions(wl, 0.1, 3, stretch=0.1)))
    F = ctx.compute_forces(x)
    ref = H.oracle_bodies(wl)[0].internal_forces(H.to_abs(wl, H.split_state(ctx, wl, x))[0]).numpy()
    e = H.rel_l2(H.split_state(ctx, wl, F)[0], ref)
    record_error("F", e)
    assert e <= 1e-5


def test_oversized_patches_are_named():
    wl = scene()
    with pytest.raises(_lib.IBMError, match="lower patch_size"):
        _lib.Context(wl.bodies, wl.grid, patch_size=1200)
