"""Weight gradients on thin grids, where a voxel tile (8 x 16) holds few voxels and the tiles are
many: more slices than one grid dimension takes (a line of 3.2 million voxels), and a copy of the
gradient in whole tiles that is many times the gradient (it is made in turns). Against the sums
over the taps in FP64.

Tolerance: an accumulator adds at most 384 values per slice as on full grids (2.2e-6 of the
gradient there), and at most 8334 slices are added by eight warps each, a random walk of 2^-24
sqrt(1042) = 2e-6: 1e-5 as in the other weight-gradient tests."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from test_gpu_precond import _lib, _p, _s  # noqa: E402


def _reference(dy, x):
    """dw[co][ci][t], db[co] in FP64 on the device."""
    D, H, W = x.shape[1:]
    dy, pad = dy.double(), torch.nn.functional.pad(x.double(), (1, 1, 1, 1, 1, 1))
    flat = dy.reshape(dy.shape[0], -1)
    dw = [flat @ pad[:, a:a + D, b:b + H, c:c + W].reshape(x.shape[0], -1).T
          for a in range(3) for b in range(3) for c in range(3)]
    return torch.stack(dw, dim=2), flat.sum(1)


@pytest.mark.parametrize("cin,cout,shape", [(2, 3, (3_200_000, 1, 1)), (3, 2, (1, 1, 70_001)), (5, 6, (1500, 1, 4099)),
                                            (9, 50, (301, 2, 703)), (40, 3, (1, 900, 1))])
def test_weight_gradient_on_thin_grids(cin, cout, shape):
    lib = _lib()
    gen = torch.Generator(device="cuda").manual_seed(cin + 100 * cout)
    x = torch.randn((cin, *shape), generator=gen, device="cuda").to(torch.bfloat16)
    dy = torch.randn((cout, *shape), generator=gen, device="cuda")
    work = torch.empty(lib.fwi_nn_conv3d_backward_weight_work(cin, cout, *shape), dtype=torch.float32, device="cuda")
    got = []
    for _ in range(2):
        dw = torch.full((cout, cin, 27), 7.0, device="cuda")
        db = torch.full((cout,), 7.0, device="cuda")
        assert lib.fwi_nn_conv3d_backward_weight(_p(dy), _p(x), cin, cout, *shape, _p(dw), _p(db), _p(work), _s()) == 0
        got.append((dw, db))
    (dw, db), (dw2, db2) = got
    assert torch.equal(dw, dw2) and torch.equal(db, db2)
    rw, rb = _reference(dy, x)
    assert float((dw.double() - rw).norm() / rw.norm()) < 1e-5
    assert float((db.double() - rb).norm() / rb.norm()) < 1e-5
    assert bool((dw[rw == 0] == 0).all())  # taps that no voxel has
