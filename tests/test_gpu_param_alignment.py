"""A parameter matrix that begins anywhere in a buffer of floats is served.

The projection and its reverse stage the SH rows 16 bytes at a time where the
matrix lies on 16 bytes, else float by float: the same records and tangents, bit
by bit, and the same gradient up to the order of its float sums (1e-4 of each
row's largest entry).  Sizes with a ragged last warp, and every SH degree."""
import math

import pytest

from paper_2602_00395_gb300 import synth as S

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def offset_copy(t, off):
    buf = torch.zeros(t.numel() + 4, device="cuda")
    out = buf[off: off + t.numel()].view(t.shape)
    out.copy_(t)
    return out


@pytest.mark.parametrize("off", [1, 2, 3])
@pytest.mark.parametrize("n,deg,nu", [(5, 0, 0), (130, 1, 1), (333, 2, 2), (333, 3, 2)])
def test_matrix_at_any_float(n, deg, nu, off):
    from paper_2602_00395_gb300.engine import BatchEntry, BatchStep, TRStep
    W, H = 70, 45
    sc = S.make_scene(n, deg, seed=3, extent=0.8, log_scale_shift=math.log(2.0))
    target = S.noise_target(2, H, W, seed=4)
    e = TRStep(n, deg, 2, W, H, nu=nu)
    e.set_cameras([S.single_camera(W, H)] * 2)
    e.set_params(sc.params)
    e.set_target(target)
    e.ensure_capacity()
    got = []
    for x in (e.x, offset_copy(e.x, off)):
        assert (x.data_ptr() % 16 == 0) == (x is e.x)
        e.x = x
        e.project(2, probes=nu > 0)
        e.bin_sort()
        e.raster_fwd(2, probes=nu > 0)
        e.raster_bwd(2, probes=nu > 0)
        assert e.read_status() == 0
        got.append((e.rec.clone(), e.tan.clone(), e.image.clone(), e.grad.clone(), e.hz.clone() if nu else e.grad))
    (rec0, tan0, img0, g0, h0), (rec1, tan1, img1, g1, h1) = got
    assert torch.equal(rec0.view(torch.int32), rec1.view(torch.int32)) and torch.equal(img0, img1)
    assert torch.equal(tan0.view(torch.int32), tan1.view(torch.int32)) or nu == 0
    for a, b in ((g0, g1), (h0, h1)):
        assert bool(((a - b).abs() <= 1e-4 * a.abs().amax(1, keepdim=True)).all())
    # a request of a batch (a render: the update needs 16-byte rows as before)
    cam = e.cams[:96].contiguous()
    imgs = []
    for x in (offset_copy(e.x, 0), offset_copy(e.x, off)):
        b = BatchStep([BatchEntry(x, x, x, n, cam)], W, H, sh_degree=deg, nu=0, capacity=e.capacity, train=False)
        b.run()
        imgs.append(b.images().clone())
    assert torch.equal(*imgs)
