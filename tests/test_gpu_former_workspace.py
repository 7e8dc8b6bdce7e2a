"""A step's or a batch's reverse workspace in memory that held one before: the
allocator hands it back with the former header, which calls its rows clear, while
another tensor has written over the rows.  The results are those of fresh memory."""
import numpy as np
import pytest

from paper_2602_00395_gb300 import synth as S

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

N, W, H, DEG = 700, 97, 75, 1


def _former(monkeypatch, nbytes):
    """torch.empty returns, for a byte buffer of this size, a former workspace; the
    list of those handed out."""
    real, out = torch.empty, []
    header = np.array([0x9D2C5680A3B1F4E7, 1 << 62], np.uint64).view(np.uint8)  # magic, floats said to be zero

    def empty(*size, **kw):
        t = real(*size, **kw)
        if kw.get("dtype") == torch.uint8 and t.numel() == nbytes:
            t[256:].view(torch.float32).fill_(3.0)
            t[:16].copy_(torch.from_numpy(header.copy()))
            out.append(t)
        return t

    monkeypatch.setattr(torch, "empty", empty)
    return out


@pytest.mark.parametrize("kind", ["step", "batch", "pooled batch"])
def test_rows_of_a_former_workspace_are_cleared(kind, monkeypatch):
    from paper_2602_00395_gb300 import gs3dtr as G
    from paper_2602_00395_gb300.engine import BatchEntry, BatchStep, TRConfig, TRStep
    sc = S.make_scene(N, DEG, seed=31, kind="cube", extent=1.0)
    cam, tg = S.camera_ring(1, W, H, 1.0, seed=7, ring_factor=3.0)[0], S.noise_target(1, H, W, seed=32)

    def step():
        e = TRStep(N, DEG, 1, W, H, nu=1, cfg=TRConfig(l=1))
        e.set_cameras([cam])
        e.set_params(sc.params)
        e.set_target(tg)
        e.ensure_capacity()
        if kind == "step":
            e.step(1, 1e-5)
            out = e.grad, e.hz
        else:
            b = BatchStep([BatchEntry(e.x, e.g_ema, e.d_ema, N, e.cams, target=e.target, t=1, eps=1e-5)], W, H,
                          sh_degree=DEG, nu=1, capacity=e.capacity, cfg=TRConfig(l=1),
                          pool={} if kind == "pooled batch" else None)
            b.run()
            out = b.grads[0], b.hzs[0]
        torch.cuda.synchronize()
        return [t[:, :N].clone() for t in out]

    fresh = step()
    former = _former(monkeypatch, G.gs_raster_bwd_workspace_size(S.pad_count(N), G.frame_struct(1, W, H), 1))
    again = step()
    assert former
    for a, b in zip(again, fresh):
        assert torch.isfinite(b).all()
        torch.testing.assert_close(a, b, rtol=0, atol=1e-3 * b.abs().max().item())  # order of the atomics: below 1e-4
