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
