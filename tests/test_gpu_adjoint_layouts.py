"""The force adjoint's shared-memory layouts and block sizes: one step's adjoint
of a deformed drop and a clamped open sheet for patches from the smallest to the
largest that fits, against reverse mode of the FP64 oracle (bars of the adjoint
parity test: 1e-4 of the non-trivial part and of the constants' cotangents).
The flow is linear, which MLS reproduces whatever nodes the markers pick."""
import numpy as np
import pytest
import torch

from paper_1612_03399_gb300 import _lib
from paper_1612_03399_gb300 import workloads as W

import helpers as H
from test_gpu_adjoint import DEV, PARAMS, oracle_vjp
from test_gpu_force_layouts import largest_patch, scene

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def reference():
    wl = scene()
    x = H.rel_positions(wl, W.perturb_positions(wl, 0.05, 20, stretch=0.05))
    rng = np.random.default_rng(9)
    V = sum(len(b.rest) for b in wl.bodies)
    gxn, gvn = (torch.tensor(rng.standard_normal((3, V)), dtype=torch.float32) for _ in range(2))
    return wl, x, gxn, gvn, {}


@pytest.mark.parametrize("patch", [32, 224, 384, "largest"])
def test_backward(patch, reference, record_error):
    wl, rel, gxn, gvn, want = reference
    ctx = largest_patch(wl) if patch == "largest" else _lib.Context(wl.bodies, wl.grid,
                                                                    patch_size=patch)
    x = H.state_tensor(wl, rel)
    fields = H.fields_for(wl, DEV)
    gx, gv, gp = ctx.backward(x, fields, gxn.to(DEV), gvn.to(DEV))
    ctx.check_device_error()
    gxn_b, gvn_b = ([torch.tensor(a) for a in H.split_state(ctx, wl, g)] for g in (gxn, gvn))
    if not want:
        xs = H.to_abs(wl, H.split_state(ctx, wl, x))
        want["all"] = oracle_vjp(wl, H.oracle_bodies(wl), xs, [torch.zeros_like(t) for t in xs],
                                 tuple(f.double().cpu() for f in fields), gxn_b, gvn_b)
    ogx, ogv, ogp = want["all"]
    got_x, got_v, gp = H.split_state(ctx, wl, gx), H.split_state(ctx, wl, gv), gp.cpu().numpy()
    for i, b in enumerate(wl.bodies):
        e = H.rel_l2(got_x[i] - gxn_b[i].numpy(), ogx[i] - gxn_b[i].numpy())
        record_error(f"gx[{i}]", e)
        assert e <= 1e-4
        assert H.rel_l2(got_v[i], ogv[i]) <= 1e-6
        for k, name in enumerate(PARAMS):
            if b.closed or name != "kv":
                e = abs(gp[i, k] - ogp[i, k]) / max(abs(ogp[i, k]), 1e-30)
                record_error(f"g{name}[{i}]", e)
                assert e <= 1e-4, (i, name)
