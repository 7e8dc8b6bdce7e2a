"""The reverse blend at the sizes where its per-block walk can go wrong.

A warp walks one 8 x 8 pixel block: it stages the block's visible splats in
buffers of 32 and merges them four at a time.  So the lists here are short
(partial merges: 1, 3, 4, 5 splats), around the staging buffer (31, 32, 33, 65)
and longer than two buffers (130), on an image whose right and lower blocks are
partial or empty, with 0, 1 and 2 probes.  Against the FP64 oracle with the
tolerances of the parity tests (gradient 1e-4, z.Hz 1e-3, the oracle's
allowances); the objective is a plain sum, 1e-6.
"""
import math

import numpy as np
import pytest

import oracle as O
from paper_2602_00395_gb300 import synth as S

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("nu", [0, 1, 2])
@pytest.mark.parametrize("n", [1, 3, 4, 5, 31, 32, 33, 65, 130])
def test_short_lists_match_oracle(n, nu):
    from paper_2602_00395_gb300.engine import TRStep
    from test_gpu_parity import _group_close
    W, H, t = 41, 19, 3
    sc = S.make_scene(n, 1, seed=70 + n, extent=0.4, log_scale_shift=math.log(3.0))
    cams = [S.single_camera(W, H)]
    target = S.noise_target(1, H, W, seed=71)
    e = TRStep(n, 1, 1, W, H, nu=nu)
    e.set_cameras(cams)
    e.set_params(sc.params)
    e.set_target(target)
    e.ensure_capacity()
    probes = nu > 0
    e.project(t, probes=probes)
    e.bin_sort()
    e.raster_fwd(t, probes=probes)
    for _ in range(2):  # the second call finds its workspace as the first left it
        e.loss_val.zero_()
        e.raster_bwd(t, probes=probes)
    torch.cuda.synchronize()
    assert e.read_status() == 0
    ref = O.backward(O.params64(sc), 1, cams, target.astype(np.float64), seed=42, t=t, nu=nu, masses=True)
    assert abs(float(e.loss_val.item()) - ref["loss"]) <= 1e-6 * ref["loss"]
    _group_close(e.grad[:, :n].cpu().numpy(), ref["grad"], 1e-4, "grad", ref["grad_mass"], ref["grad_allow"],
                 rnd=ref["grad_round"])
    if nu:
        _group_close(e.hz[:, :n].cpu().numpy(), ref["hz"], 1e-3, "hz", ref["hz_mass"], ref["hz_sens"],
                     ref["hz_allow"], rnd=ref["hz_round"])


@pytest.mark.parametrize("n,off,room", [(1, 0, 0), (33, 0, 0), (33, 0, 1), (33, 0, 2), (33, 1, 0), (33, 2, 3), (33, 3, 1)])
def test_masks_at_any_address(n, off, room):
    """The masks are written as 32-bit words: whatever the buffer's address and
    size, the bytes around it stay, the bytes in whole words are what an aligned
    buffer holds, the others have every bit set, and the gradient is the one
    without masks up to the order of its float sums."""
    from paper_2602_00395_gb300.engine import TRStep
    W, H = 41, 19
    sc = S.make_scene(n, 1, seed=70 + n, extent=0.4, log_scale_shift=math.log(3.0))
    e = TRStep(n, 1, 1, W, H, nu=0)
    e.set_cameras([S.single_camera(W, H)])
    e.set_params(sc.params)
    e.set_target(S.noise_target(1, H, W, seed=71))
    e.ensure_capacity()
    e.project()
    e.bin_sort()
    P = int(e.n_pairs.item())
    e._alloc_pairs(P + room)
    e.bin_sort()
    e.raster_fwd()
    aligned = e.masks.clone()
    e.raster_bwd()
    grad = e.grad.clone()
    e.masks_valid = False
    e.raster_bwd()
    plain = e.grad.clone()
    around = torch.full((P + room + 32,), 0xA5, dtype=torch.uint8, device="cuda")
    e.masks = around[16 + off : 16 + off + P + room]
    e.raster_fwd()
    e.raster_bwd()
    torch.cuda.synchronize()
    assert e.read_status() == 0
    assert bool((around[: 16 + off] == 0xA5).all()) and bool((around[16 + off + P + room :] == 0xA5).all())
    at = torch.arange(16 + off, 16 + off + P + room, device="cuda")
    whole = (at // 4 * 4 >= 16 + off) & (at // 4 * 4 + 4 <= 16 + off + P + room) & (P + room >= 8)
    both = whole & (torch.arange(P + room, device="cuda") < (P + room) // 4 * 4)
    assert torch.equal(e.masks[both], aligned[both]) and bool((e.masks[~whole] == 0xFF).all())
    scale = float(plain.abs().max())
    assert scale > 0
    for g in (grad, e.grad):
        assert float((g - plain).abs().max()) <= 1e-5 * scale
