"""The convolutions of the learned preconditioner (fwi_precond.h) against the FP64 oracle on
grids where the tile kernels' paths change: more tiles than blocks, ragged plane chunks, several
channel passes, each form of the weight gradient.

Tolerances as in test_gpu_precond.py, whose arithmetic argument holds on these sizes too: a
forward output is an FP32 sum rounded to BF16, the backward sums are FP32."""
import numpy as np
import pytest

from helpers import rel_l2

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle import precond as P  # noqa: E402
from test_gpu_precond import _bf16, _bwd_data_tol, _f32, _lib, _p, _s, _vals  # noqa: E402


@pytest.mark.parametrize("cin,cout,shape", [(5, 6, (13, 129, 137)), (100, 3, (6, 65, 129)), (45, 50, (3, 17, 33)),
                                            (3, 4, (17, 129, 137))])
def test_convolutions_on_many_tiles(cin, cout, shape):
    # more tiles than blocks on the GPU, so that a block walks several (ragged plane chunks and
    # tile edges among them); several passes over the channel groups; a weight gradient of one
    # tap group per kz and of three taps, of one and of two gradient row tiles, with its partial
    # sums in the caller's scratch and in its own; the last grid's gradient is split by a launch
    # of its own. A second call gives the same bits.
    rng = np.random.default_rng(cin + 7 * cout)
    lib = _lib()
    xd, xv = _bf16(rng.standard_normal((cin, *shape)))
    wd, wv = _bf16(rng.standard_normal((cout, cin, 27)) / np.sqrt(27 * cin))
    b = rng.standard_normal(cout).astype(np.float32)
    y = torch.empty((cout, *shape), dtype=torch.bfloat16, device="cuda")
    bd = _f32(b)
    assert lib.fwi_nn_conv3d_forward(_p(xd), _p(wd), _p(bd), cin, cout, *shape, 0, _p(y), _s()) == 0
    y2 = torch.empty_like(y)
    assert lib.fwi_nn_conv3d_forward(_p(xd), _p(wd), _p(bd), cin, cout, *shape, 0, _p(y2), _s()) == 0
    assert torch.equal(y.view(torch.int16), y2.view(torch.int16))
    ref, got = P.conv3d(xv, wv, b.astype(np.float64)), _vals(y)
    assert np.all(np.abs(got - ref) <= 2.0 ** -8 * np.abs(ref) + 1e-5)
    dy = rng.standard_normal((cout, *shape)).astype(np.float32)
    dyd = _f32(dy)
    dx = torch.empty((cin, *shape), dtype=torch.float32, device="cuda")
    assert lib.fwi_nn_conv3d_backward_data(_p(dyd), _p(wd), cin, cout, *shape, _p(dx), _s()) == 0
    assert rel_l2(dx.cpu().numpy(), P.conv3d_backward_data(dy.astype(np.float64), wv, cin)) < _bwd_data_tol(cout)
    work = torch.empty(lib.fwi_nn_conv3d_backward_weight_work(cin, cout, *shape), dtype=torch.float32, device="cuda")
    dw = torch.empty((cout, cin, 27), dtype=torch.float32, device="cuda")
    db = torch.empty(cout, dtype=torch.float32, device="cuda")
    assert lib.fwi_nn_conv3d_backward_weight(_p(dyd), _p(xd), cin, cout, *shape, _p(dw), _p(db), _p(work), _s()) == 0
    dw_ref, db_ref = P.conv3d_backward_weight(dy.astype(np.float64), xv)
    assert rel_l2(dw.cpu().numpy(), dw_ref) < 1e-5
    assert rel_l2(db.cpu().numpy(), db_ref) < 1e-5
