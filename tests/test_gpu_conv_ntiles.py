"""Convolutions of more GEMM output channels than one tile of them (256) on grids with more tiles
than the GPU holds blocks: a block goes from one tile of channels to the next, and takes the new
channels' biases while the MMAs of its next tile run. Against the FP64 oracle with the tolerances of
test_gpu_precond.py; every pass twice, bit for bit."""
import numpy as np
import pytest

from helpers import rel_l2

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle import precond as P  # noqa: E402
from test_gpu_precond import _bf16, _bwd_data_tol, _f32, _lib, _p, _s, _vals  # noqa: E402


def _twice(make, call):
    """The outputs of two calls into fresh buffers, the same bit for bit."""
    outs = []
    for _ in range(2):
        out = make()
        assert call(*out) == 0
        outs.append(out)
    for a, b in zip(*outs):
        assert torch.equal(a.view(torch.int16), b.view(torch.int16))
    return outs[0]


@pytest.mark.parametrize("many,few,shape", [(300, 3, (2, 160, 161)), (520, 2, (5, 90, 95))])
def test_block_walks_over_channel_tiles(many, few, shape):
    rng = np.random.default_rng(many)
    lib = _lib()
    vox = lambda c, t: (torch.empty((c, *shape), dtype=t, device="cuda"),)  # noqa: E731
    # forward, `many` output channels, with a bias that differs from channel to channel
    xd, xv = _bf16(rng.standard_normal((few, *shape)))
    wd, wv = _bf16(rng.standard_normal((many, few, 27)) / np.sqrt(27 * few))
    b = (3 + np.arange(many) % 7 + rng.standard_normal(many)).astype(np.float32)
    bd = _f32(b)
    y, = _twice(lambda: vox(many, torch.bfloat16),
                lambda o: lib.fwi_nn_conv3d_forward(_p(xd), _p(wd), _p(bd), few, many, *shape, 0, _p(o), _s()))
    ref = P.conv3d(xv, wv, b.astype(np.float64))
    assert np.all(np.abs(_vals(y) - ref) <= 2.0 ** -8 * np.abs(ref) + 1e-5)
    # backward data to `many` input channels, and that layer's weight gradient
    wd, wv = _bf16(rng.standard_normal((few, many, 27)) / np.sqrt(27 * many))
    dy = rng.standard_normal((few, *shape)).astype(np.float32)
    dyd = _f32(dy)
    dx, = _twice(lambda: vox(many, torch.float32),
                 lambda o: lib.fwi_nn_conv3d_backward_data(_p(dyd), _p(wd), many, few, *shape, _p(o), _s()))
    assert rel_l2(dx.cpu().numpy(), P.conv3d_backward_data(dy.astype(np.float64), wv, many)) < _bwd_data_tol(few)
    xd, xv = _bf16(rng.standard_normal((many, *shape)))
    work = torch.empty(lib.fwi_nn_conv3d_backward_weight_work(many, few, *shape), dtype=torch.float32, device="cuda")
    dw, db = _twice(lambda: (torch.empty((few, many, 27), device="cuda"), torch.empty(few, device="cuda")),
                    lambda o, p: lib.fwi_nn_conv3d_backward_weight(_p(dyd), _p(xd), many, few, *shape, _p(o), _p(p),
                                                                   _p(work), _s()))
    dw_ref, db_ref = P.conv3d_backward_weight(dy.astype(np.float64), xv)
    assert rel_l2(dw.cpu().numpy(), dw_ref) < 1e-5
    assert rel_l2(db.cpu().numpy(), db_ref) < 1e-5


def test_fewer_channels_take_no_longer():
    # 8 -> 16 channels are a seventh of the work of 28 -> 28. With a grid of more blocks than the GPU holds
    # at once, each owning its share of the tiles, they took a third longer.
    lib = _lib()
    shape = (65, 129, 129)

    def best(cin, cout):
        x = torch.zeros((cin, *shape), dtype=torch.bfloat16, device="cuda")
        w = torch.zeros((cout, cin, 27), dtype=torch.bfloat16, device="cuda")
        y = torch.empty((cout, *shape), dtype=torch.bfloat16, device="cuda")
        ms = []
        for _ in range(12):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            for _ in range(10):
                assert lib.fwi_nn_conv3d_forward(_p(x), _p(w), None, cin, cout, *shape, 1, _p(y), _s()) == 0
            b.record()
            b.synchronize()
            ms.append(a.elapsed_time(b))
        return min(ms)

    assert best(8, 16) < best(28, 28)
