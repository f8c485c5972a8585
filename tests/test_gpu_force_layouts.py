"""The force kernel's block sizes and shared-memory layouts: internal forces and
energies of a deformed drop and a clamped open sheet for patches from the
smallest to the largest that fits (whose positions and slots no longer fit as
float4), against the FP64 oracle (bar 1e-5 as in the parity tests)."""
import numpy as np
import pytest
import torch

from paper_1612_03399_gb300 import _lib
from paper_1612_03399_gb300 import workloads as W

import helpers as H

pytestmark = pytest.mark.gpu


def scene():
    rng = np.random.default_rng(6)
    c = np.array([0.5, 0.5, 0.5])
    v, t = W.icosphere(4)
    sv, st, rim = W.elliptic_sheet(0.2, 0.15, 1500, rng, jitter=0.1)
    bodies = [W.Body(rest=c + 0.2 * v * np.array([1.2, 1.0, 0.9]), tri=t, origin=c),
              W.Body(rest=c + sv, tri=st, origin=c, closed=False, clamped=rim, ks=5.0, kb=0.3,
                     kA=0.0, kv=0.0, spring_model=1)]
    return W.Workload(name="layouts", bodies=bodies, grid=W.Grid((32, 32, 32)),
                      field={"kind": "shear"})


def largest_patch(wl):
    for p in range(800, 512, -16):
        try:
            return _lib.Context(wl.bodies, wl.grid, patch_size=p)
        except _lib.IBMError:
            continue
    raise RuntimeError("no patch above 512 fits")


@pytest.mark.parametrize("patch", [32, 96, 224, 384, "largest"])
def test_forces_and_energies(patch, record_error):
    wl = scene()
    ctx = largest_patch(wl) if patch == "largest" else _lib.Context(wl.bodies, wl.grid,
                                                                    patch_size=patch)
    xs = W.perturb_positions(wl, 0.1, 3, stretch=0.1)
    x = H.state_tensor(wl, H.rel_positions(wl, xs))
    F, E = ctx.compute_forces(x, energy=True)
    assert torch.equal(F, ctx.compute_forces(x))
    got = H.split_state(ctx, wl, F)
    ax = H.to_abs(wl, H.split_state(ctx, wl, x))
    for i, b in enumerate(H.oracle_bodies(wl)):
        ref = b.internal_forces(ax[i]).numpy()
        e = H.rel_l2(got[i], ref)
        record_error(f"F[{i}]", e)
        assert e <= 1e-5
        t = b.energy_terms(ax[i])
        for j, k in enumerate(("We", "Wb", "Wa", "WA", "Wv")):
            assert float(E[i, j]) == pytest.approx(float(t[k]), rel=1e-5, abs=1e-12), k
