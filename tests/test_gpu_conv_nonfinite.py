"""Non-finite values in the preconditioner's convolutions. A NaN stays where the sums that use
it are: it must reach the outputs (a ReLU that turned it into zero would hide a failed layer,
and the loss would stay finite) and no others."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from test_gpu_precond import _bf16, _f32, _lib, _p, _s, _vals  # noqa: E402


@pytest.mark.parametrize("relu", [0, 1])
@pytest.mark.parametrize("cin,cout,shape,at", [(3, 5, (4, 19, 11), (2, 7, 4)), (20, 40, (5, 16, 8), (0, 0, 0)),
                                               (4, 17, (3, 33, 17), (2, 32, 16))])
def test_forward_keeps_a_nan_in_its_stencil(relu, cin, cout, shape, at):
    rng = np.random.default_rng(cin + cout)
    lib = _lib()
    x = rng.standard_normal((cin, *shape))
    wd, _ = _bf16(rng.standard_normal((cout, cin, 27)) / np.sqrt(27 * cin))
    bd = _f32(rng.standard_normal(cout).astype(np.float32))

    def run(values):
        xd, _ = _bf16(values)
        y = torch.empty((cout, *shape), dtype=torch.bfloat16, device="cuda")
        assert lib.fwi_nn_conv3d_forward(_p(xd), _p(wd), _p(bd), cin, cout, *shape, relu, _p(y), _s()) == 0
        return _vals(y)

    clean = run(x)
    assert np.isfinite(clean).all()
    x[cin // 2][at] = np.nan
    got = run(x)
    near = np.zeros(shape, bool)
    near[tuple(slice(max(a - 1, 0), a + 2) for a in at)] = True
    assert np.isnan(got[:, near]).all()
    assert np.array_equal(got[:, ~near], clean[:, ~near])


def test_network_loss_shows_a_nan_of_the_input():
    from paper_1504_08340_gb300.precond import UNet

    net = UNet(4, 2, (6, 8, 10), (9, 17, 13), seed=3)
    gen = torch.Generator().manual_seed(5)
    x = torch.randn((4, 9, 17, 13), generator=gen).to("cuda")
    t = torch.randn((2, 9, 17, 13), generator=gen).to("cuda")
    with torch.no_grad():
        assert bool(torch.isfinite(net(x)).all())
        x[1, 4, 8, 6] = float("nan")
        assert bool(torch.isnan(net(x)).any())
    assert np.isnan(net.train_step(x, t))


@pytest.mark.parametrize("value", [float("nan"), float("inf")])
@pytest.mark.parametrize("cin,cout,shape", [(3, 5, (4, 19, 11)), (40, 3, (3, 16, 13)), (2, 45, (2, 33, 8)),
                                            (3, 2, (3, 32, 16))])
def test_weight_gradient_of_a_non_finite_edge(cin, cout, shape, value):
    # one non-finite x at a corner, an edge or inside the grid: the taps that use it are not
    # finite, the others are the FP64 sums. Tolerance as in test_gpu_precond.py.
    lib = _lib()
    gen = torch.Generator(device="cuda").manual_seed(cin + cout)
    dy = torch.randn((cout, *shape), generator=gen, device="cuda")
    base = torch.randn((cin, *shape), generator=gen, device="cuda").to(torch.bfloat16)
    D, H, W = shape
    work = torch.empty(lib.fwi_nn_conv3d_backward_weight_work(cin, cout, *shape), dtype=torch.float32, device="cuda")
    for at in [(0, 0, 0), (1, 5, W - 1), (D - 1, H - 1, 3), (1, H - 1, W - 1), (D - 1, 7, 4), (0, 2, 0)]:
        x = base.clone()
        ci = cin - 1
        x[ci][at] = value
        dw = torch.empty((cout, cin, 27), device="cuda")
        db = torch.empty(cout, device="cuda")
        assert lib.fwi_nn_conv3d_backward_weight(_p(dy), _p(x), cin, cout, *shape, _p(dw), _p(db), _p(work), _s()) == 0
        flat = dy.double().reshape(cout, -1)
        pad = torch.nn.functional.pad(base.double(), (1, 1, 1, 1, 1, 1))
        ref = torch.stack([flat @ pad[:, a:a + D, b:b + H, c:c + W].reshape(cin, -1).T
                           for a in range(3) for b in range(3) for c in range(3)], dim=2)
        for t in range(27):  # the voxel that reads x[at] with tap t
            p = (at[0] + 1 - t // 9, at[1] + 1 - t // 3 % 3, at[2] + 1 - t % 3)
            if all(0 <= q < n for q, n in zip(p, shape)):
                ref[:, ci, t] = float("nan")
        finite = torch.isfinite(ref)
        assert torch.equal(torch.isfinite(dw), finite), at
        err = (dw.double() - ref)[finite].norm() / ref[finite].norm()
        assert float(err) < 1e-5, (at, float(err))
        assert torch.isfinite(db).all()
