"""Kernel timing by class: point loads and samples that take a kernel of their own are counted and
timed in class 2, and in no other; where the stage kernels apply them there is none."""
import numpy as np
import pytest

import fwi_inputs as fi

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("inside_pml", [False, True])
def test_point_kernels_are_class_two(inside_pml):
    from paper_1504_08340_gb300 import Context

    w = fi.tiny(nx=3, ny=3, nz=2, npml=2, nsteps=12, f0=30.0)
    p = 2 * w.npml
    lam, mu = (np.ascontiguousarray(a, dtype=np.float32) for a in fi.medium(w, "true"))
    with Context(w.nx, w.ny, w.nz, w.npml, w.h, w.dt, w.nsteps, rho=w.rho) as ctx:
        ctx.set_material(lam, mu)
        # a source on a node of the PML kernel, which does not apply points
        ctx.set_sources([(p - 1, p + 3, 2) if inside_pml else (p + 3, p + 2, 1)], [(0.0, 0.0, 1.0)], "ricker", w.ricker())
        ctx.set_receivers([(p + 2, p + 2, 0)])
        ctx.reset_timing()
        ctx.set_timing(True)
        ctx.forward(0, 1)
        ctx.set_timing(False)
        ms, launches = zip(*(ctx.timing(k) for k in range(4)))
    stages = 4 * w.nsteps
    assert launches[0] == stages and ms[0] > 0
    assert launches[1] == 0
    if inside_pml:
        assert launches[2] == stages and 0 < ms[2] < ms[0]
        assert launches[3] == 5 * stages  # interior, shell, face, PML, points
    else:
        assert launches[2] == 0 and ms[2] == 0
        assert launches[3] == 4 * stages
