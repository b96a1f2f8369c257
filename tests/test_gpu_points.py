"""Point loads and receiver samples on every node set a stage kernel writes: interior, interface
shell, free top face outside the interior, and nodes inside the PML, with a receiver on a source
node, against the FP64 oracle. The tolerances are those of the other parity tests: traces
1e-5, J 2e-5, gradients 1e-4 relative L2."""
import numpy as np
import pytest

import fwi_inputs as fi
from helpers import rel_l2

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

# offsets from the interior's corner node (2 npml, 2 npml, 0), in nodes
INTERIOR, SHELL, TOP_FACE, DEEP = (3, 2, 1), (0, 3, 0), (-2, 3, 0), (-1, 3, 2)


@pytest.mark.parametrize("source", [INTERIOR, SHELL, TOP_FACE, DEEP])
@pytest.mark.parametrize("sweep", ["direct", "graph", "persistent"])
def test_points_on_every_node_set(oracle_mod, source, sweep):
    from paper_1504_08340_gb300 import Context

    w = fi.tiny(nx=3, ny=3, nz=2, npml=2, nsteps=40, f0=30.0)
    p = 2 * w.npml
    node = lambda o: (p + o[0], p + o[1], o[2])  # noqa: E731
    src = np.array([node(source), node(INTERIOR)])  # two shots in one batch
    rec = np.array([node(o) for o in (INTERIOR, SHELL, TOP_FACE, DEEP, (2, 2, 0), (4, 7, 5))])
    dirs = np.array([[0.2, -0.3, 1.0], [0.0, 0.0, 1.0]])
    lam, mu = (np.ascontiguousarray(a, dtype=np.float32) for a in fi.medium(w, "true"))
    obs = np.stack([fi.synthetic_traces(w.nsteps, len(rec), 5 + s, scale=1e-7) for s in range(2)])
    obs = np.ascontiguousarray(obs, dtype=np.float32)

    o = oracle_mod.Oracle(w.nx, w.ny, w.nz, w.npml, h=w.h, rho=w.rho)
    o.set_material(lam.astype(np.float64), mu.astype(np.float64))
    rn = [o.node_id(*r) for r in rec]
    J, gl, gm, traces = 0.0, 0.0, 0.0, []
    for s in range(2):
        j, a, b, t = o.misfit_and_gradient(w.dt, w.nsteps, [o.node_id(*src[s])], dirs[s], rn, obs[s].astype(np.float64),
                                           "ricker", w.ricker())
        J, gl, gm = J + j, gl + a, gm + b
        traces.append(t)
    with Context(w.nx, w.ny, w.nz, w.npml, w.h, w.dt, w.nsteps, rho=w.rho) as ctx:
        ctx.set_material(lam, mu)
        ctx.set_sources(src, dirs, "ricker", w.ricker())
        ctx.set_receivers(rec)
        ctx.set_shot_batch(2)
        if sweep == "graph":
            ctx.set_graphs(True)
        elif sweep == "persistent":
            ctx.set_persistent(True)
        got = ctx.forward(0, 2)
        Jg, glg, gmg = ctx.adjoint_gradient(obs, 0, 2)
        assert np.array_equal(ctx.forward(0, 2), got)
    for s in range(2):
        assert rel_l2(got[s], traces[s]) < 1e-5
    assert Jg == pytest.approx(J, rel=2e-5)
    assert rel_l2(glg, gl) < 1e-4 and rel_l2(gmg, gm) < 1e-4


def test_points_of_a_large_batch():
    """A batch whose nodes exceed the limit up to which the stage kernels apply the points takes
    the kernel of its own after each stage: traces and gradient of such a batch against those of
    one shot at a time, traces bitwise (the two add and read the same values)."""
    from paper_1504_08340_gb300 import Context

    w = fi.box_8x8x4()
    shots, steps = 640, 6  # 640 x 12,615 nodes > 8,000,000
    lam, mu = (np.ascontiguousarray(a, dtype=np.float32) for a in fi.medium(w, "true"))
    rng = np.random.default_rng(3)
    p = 2 * w.npml
    src = np.stack([rng.integers(2, p + 20, shots), rng.integers(2, p + 20, shots), rng.integers(0, 12, shots)], axis=1)
    src[:3] = [(p + 4, p + 4, 0), (2, 9, 0), (2, 9, 3)]  # interior, free top face in the PML, inside the PML
    rec = np.array([(p + 4, p + 4, 0), (2, 9, 0), (2, 9, 3), (p, p + 3, 2)])
    obs = torch.zeros((shots, steps + 1, len(rec), 3), dtype=torch.float32, device="cuda")
    with Context(w.nx, w.ny, w.nz, w.npml, w.h, w.dt, steps, rho=w.rho) as ctx:
        ctx.set_material(lam, mu)
        ctx.set_sources(src, np.tile([0.1, 0.2, 1.0], (shots, 1)), "ricker", (100.0, 0.001, 1e3))
        ctx.set_receivers(rec)
        one = [ctx.forward(s, 1) for s in range(3)]
        g1 = [ctx.adjoint_gradient(obs[s:s + 1].contiguous(), s, 1)[1].cpu().numpy() for s in range(3)]
        ctx.set_shot_batch(shots)
        assert shots * ctx.nnode > 8_000_000
        many = ctx.forward(0, shots)
        assert np.abs(many).max() > 0
        for s in range(3):
            assert np.array_equal(many[s], one[s][0])
        ctx.set_shot_batch(1)
        total = sum(ctx.adjoint_gradient(obs[s:s + 1].contiguous(), s, 1)[1].cpu().numpy() for s in range(shots))
        ctx.set_shot_batch(shots)
        g = ctx.adjoint_gradient(obs, 0, shots)[1].cpu().numpy()
    assert rel_l2(g, total) < 1e-12  # FP64 sums of the same FP32 products in another order
    assert all(np.isfinite(x).all() for x in g1)
