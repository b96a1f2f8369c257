"""Pooling and upsampling on grids of small planes, whose blocks take several (channel, z) planes,
on more planes than one grid dimension takes, and at the change from one form to the other.
Forward: the sums of up to eight BF16 values in FP32, so within half a BF16 step of FP64; backward
and upsampling: single products and sums of eight, 1e-6 relative."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle import precond as P  # noqa: E402
from test_gpu_precond import _bf16, _f32, _lib, _p, _s, _vals  # noqa: E402

CASES = [(3, 5, 1, 1), (2, 301, 3, 2), (5, 7, 4, 4), (2, 3, 16, 8), (2, 3, 43, 3), (2, 5, 16, 16), (1, 4, 17, 31),
         (60000, 2, 12, 11)]


@pytest.mark.parametrize("C,D,H,W", CASES)
def test_small_planes(C, D, H, W):
    rng = np.random.default_rng(C * D + H * W)
    lib = _lib()
    fine, coarse = (C, D, H, W), (C, (D + 1) // 2, (H + 1) // 2, (W + 1) // 2)
    xd, xv = _bf16(rng.standard_normal(fine))
    y = torch.empty(coarse, dtype=torch.bfloat16, device="cuda")
    assert lib.fwi_nn_pool2_forward(_p(xd), *fine, _p(y), _s()) == 0
    ref = P.pool2(xv)
    assert np.all(np.abs(_vals(y) - ref) <= 2.0 ** -8 * np.abs(ref) + 1e-6)
    cd, cv = _bf16(rng.standard_normal(coarse))
    up = torch.empty(fine, dtype=torch.bfloat16, device="cuda")
    assert lib.fwi_nn_upsample2_forward(_p(cd), *fine, _p(up), _s()) == 0
    assert np.array_equal(_vals(up), P.upsample2(cv, fine[1:]))
    gc, gf = rng.standard_normal(coarse).astype(np.float32), rng.standard_normal(fine).astype(np.float32)
    for acc in (0, 1):
        dx0 = rng.standard_normal(fine).astype(np.float32)
        dx = _f32(dx0)
        assert lib.fwi_nn_pool2_backward(_p(_f32(gc)), *fine, acc, _p(dx), _s()) == 0
        want = P.pool2_backward(gc.astype(np.float64), fine[1:]) + acc * dx0
        assert np.allclose(dx.cpu().numpy(), want, rtol=1e-6, atol=1e-6)
        dc0 = rng.standard_normal(coarse).astype(np.float32)
        dc = _f32(dc0)
        assert lib.fwi_nn_upsample2_backward(_p(_f32(gf)), *fine, acc, _p(dc), _s()) == 0
        want = P.upsample2_backward(gf.astype(np.float64)) + acc * dc0
        assert np.allclose(dc.cpu().numpy(), want, rtol=1e-6, atol=2e-6)


def test_small_planes_keep_the_threads_busy():
    # the same voxels in planes of 4 x 4 and of 64 x 64: a block per small plane took 12 times as long
    lib = _lib()

    def best(C, D, H, W):
        x = torch.zeros((C, D, H, W), dtype=torch.bfloat16, device="cuda")
        y = torch.zeros((C, (D + 1) // 2, (H + 1) // 2, (W + 1) // 2), dtype=torch.bfloat16, device="cuda")
        ms = []
        for _ in range(20):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            for _ in range(10):
                assert lib.fwi_nn_pool2_forward(_p(x), C, D, H, W, _p(y), _s()) == 0
            b.record()
            b.synchronize()
            ms.append(a.elapsed_time(b))
        return min(ms)

    assert best(64, 4096, 4, 4) < 4 * best(64, 16, 64, 64)
