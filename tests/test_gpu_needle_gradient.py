"""The gradient of needles is held to recorded values.

The moments that the reverse blend sums over a splat's pixels cancel in the
projection's reverse pass, for a needle by about the square of its axis ratio, so
another order of those sums moves the gradients of its scale and rotation by many
roundings.  Here 96 needles (16 : 1 in variance), each alone in 32 x 32 pixels and
across two 8 x 8 pixel blocks, have sums that do not depend on the order of the
blocks; `data/needle_gradient.npy` holds their gradients (3 scale and 4 rotation
rows) as the scalar reverse blend of the library's first version computed them.
"""
import os

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

RECORDED = os.path.join(os.path.dirname(os.path.abspath(__file__)), "data", "needle_gradient.npy")
W, H = 384, 256


class Camera:
    viewmat = np.eye(4, dtype=np.float32)
    fx = fy = 256.0
    cx, cy, near, width, height = W / 2, H / 2, 0.2, W, H


def needles():
    """Parameters (uniform draws and sums of them only, so that every machine has
    the same bits) and a target image of rational steps."""
    r = np.random.RandomState(5)
    u = lambda lo, hi: r.randint(0, 1 << 20, 96) / float(1 << 20) * (hi - lo) + lo
    cell = np.arange(96)
    px, py = cell % 12 * 32 + 16 + u(-1, 1), cell // 12 * 32 + 12 + u(-0.4, 0.4)
    z = np.full(96, 4.0)
    rows = [(px - W / 2) / 64, (py - H / 2) / 64, z, u(-3.45, -3.35), u(-7, -6), u(-7, -6), u(-0.05, 0.05),
            u(-0.05, 0.05), u(0.1, 0.25) * np.where(cell % 2, 1, -1), np.ones(96), u(-0.5, 0.5),
            u(-1, 1), u(-1, 1), u(-1, 1)]
    y, x = np.mgrid[0:H, 0:W]
    target = np.stack([(x * k + y * m) % 64 / 128.0 for k, m in ((1, 3), (5, 2), (3, 7))])[None]
    return np.stack(rows).astype(np.float32), target.astype(np.float32)


def gradient(nu):
    from paper_2602_00395_gb300.engine import TRStep
    params, target = needles()
    e = TRStep(96, 0, 1, W, H, nu=nu)
    e.set_cameras([Camera()])
    e.set_params(params)
    e.set_target(target)
    e.ensure_capacity()
    e.project(1, probes=nu > 0)
    e.bin_sort()
    e.raster_fwd(1, probes=nu > 0)
    out = []
    for _ in range(2):
        e.raster_bwd(1, probes=nu > 0)
        out.append(e.grad[3:10, :96].cpu().numpy())
    assert e.read_status() == 0
    rec = e.rec.view(-1, 12)[:96].cpu().numpy()
    return out, rec


@pytest.mark.parametrize("nu", [0, 1, 2])
def test_gradient_of_needles_is_the_recorded_one(nu):
    """The rotation in the image plane (z and w) is where the moments cancel: half of
    its entries agree to two roundings (2^-22), which the projection's reverse pass
    may add of its own; sums in another order differ by many more."""
    (a, b), rec = gradient(nu)
    ext = rec[:, 11].copy().view(np.float16).reshape(-1, 2).astype(np.float64)
    lo, hi = rec[:, :2] - ext, rec[:, :2] + ext
    blocks = np.prod(np.floor((hi - 0.5) / 8) - np.floor((lo - 0.5 + 0.999) / 8) + 1, axis=1)
    assert blocks.max() <= 2
    assert np.array_equal(a, b)
    want = np.load(RECORDED)
    assert np.median((np.abs(a.astype(np.float64) - want) / np.abs(want))[5:7]) <= 2.0 ** -22
