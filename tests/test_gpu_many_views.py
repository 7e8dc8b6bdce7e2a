"""The projection's reverse pass past the views whose colour cotangents it keeps.

Up to 8 views pass 2 of the projection reverse reads the clamped colour cotangents
from shared memory; from there on it reads the cotangent rows again (two probes'
interleaved) and takes the clamp decisions from bits kept up to view 21, and
recomputes them after that; rows of views from 64 on are cleared without a look at
what was read.  A third of the colours are clamped at zero.  Against the FP64
oracle with the tolerances of the parity tests; each call runs twice, so that the
second finds the rows as the first left them."""
import math

import numpy as np
import pytest

import oracle as O
from paper_2602_00395_gb300 import synth as S

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("nu", [0, 1, 2])
@pytest.mark.parametrize("V,deg", [(9, 3), (23, 1), (66, 0)])
def test_many_views_match_oracle(V, deg, nu):
    from paper_2602_00395_gb300.engine import TRStep
    from test_gpu_parity import _group_close
    n, W, H, t = 40, 33, 21, 2
    sc = S.make_scene(n, deg, seed=90 + V, extent=0.5, log_scale_shift=math.log(2.5))
    sc.params[S.ROW_SH: S.ROW_SH + 3, : n: 3] -= 2.5  # a third of the splats: below zero in some channels
    cams = S.camera_ring(V, W, H, 1.0)
    target = S.noise_target(V, H, W, seed=91)
    e = TRStep(n, deg, V, W, H, nu=nu)
    e.set_cameras(cams)
    e.set_params(sc.params)
    e.set_target(target)
    e.ensure_capacity()
    e.project(t, probes=nu > 0)
    clamped = e.rec.view(V, e.n_pad, 12)[:, :n, 6:9] == 0
    assert 0.1 < float(clamped.float().mean()) < 0.7
    e.bin_sort()
    e.raster_fwd(t, probes=nu > 0)
    for _ in range(2):
        e.loss_val.zero_()
        e.raster_bwd(t, probes=nu > 0)
    torch.cuda.synchronize()
    assert e.read_status() == 0
    ref = O.backward(O.params64(sc), deg, cams, target.astype(np.float64), seed=42, t=t, nu=nu, masses=True)
    assert abs(float(e.loss_val.item()) - ref["loss"]) <= 1e-6 * ref["loss"]
    _group_close(e.grad[:, :n].cpu().numpy(), ref["grad"], 1e-4, "grad", ref["grad_mass"], ref["grad_allow"],
                 rnd=ref["grad_round"])
    if nu:
        _group_close(e.hz[:, :n].cpu().numpy(), ref["hz"], 1e-3, "hz", ref["hz_mass"], ref["hz_sens"],
                     ref["hz_allow"], rnd=ref["hz_round"])
