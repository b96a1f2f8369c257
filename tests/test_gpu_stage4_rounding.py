"""The RK4 combination's third adds no systematic error. A state multiplied by the FP32 constant 1/3
(3e-8 too large) grows by that share every step; rounded to nearest it only walks.

Bound, from the arithmetic alone: N steps of a sweep round a value about 4 N times (once per
stage), each by at most 2^-24 of it, without a preferred sign: 2^-24 sqrt(4 N) = 5.3e-6 for 2000
steps. The gradients are products of two such sweeps over the whole time window. With the
constant alone they were 6.9e-6 and 8.5e-6 off."""
import os

import numpy as np
import pytest

import fwi_inputs as fi
from helpers import rel_l2

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

GOLDEN = os.path.join(os.path.dirname(__file__), "golden", "long_run_grf_16x16x8.npz")


def test_long_run_gradients_without_drift():
    from paper_1504_08340_gb300 import Context

    gold = np.load(GOLDEN)
    w = fi.grf_16x16x8()
    bound = 2.0 ** -24 * np.sqrt(4 * w.nsteps)
    lam, mu = (np.ascontiguousarray(a, dtype=np.float32) for a in fi.medium(w, "trial"))
    with Context(w.nx, w.ny, w.nz, w.npml, w.h, w.dt, w.nsteps, rho=w.rho) as ctx:
        ctx.set_material(lam, mu)
        ctx.set_sources(w.sources(), w.source_dirs(), "ricker", w.ricker())
        ctx.set_receivers(w.receivers())
        obs = torch.tensor(gold["observed"][None], device="cuda").contiguous()
        J, gl, gm = ctx.adjoint_gradient(obs)
    assert abs(J - float(gold["J"])) < bound * float(gold["J"])
    assert rel_l2(gl.cpu().numpy(), gold["g_lambda"]) < bound
    assert rel_l2(gm.cpu().numpy(), gold["g_mu"]) < bound
