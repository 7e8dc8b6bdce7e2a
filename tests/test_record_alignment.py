"""Records and tangents off a 16-byte boundary are refused on the host (the kernels
store and read them 16 bytes at a time); no device is touched."""
import ctypes as C

import pytest


@pytest.fixture(scope="module")
def lib():
    from paper_2602_00395_gb300 import build, gs3dtr
    build.build()
    return gs3dtr.load()


@pytest.mark.parametrize("rec,tan,nu", [(8, 16, 0), (4, 16, 1), (16, 8, 1), (16, 12, 2)])
def test_misaligned_records_are_refused(lib, rec, tan, nu):
    from paper_2602_00395_gb300 import gs3dtr as G
    fr, x, v = G.frame_struct(1, 32, 32), G.gs_params(30, 32, 0, 0, 16), C.c_void_p(16)
    proj, pr = G.gs_projected(rec, tan), (C.byref(G.probe_struct(1, 1, nu)) if nu else None)
    srt, loss, ref = G.gs_sorted(16, 16, 16, 16, 100, None, None), G.gs_loss(0, 1e-3), C.byref
    item = (G.gs_batch_item * 1)(G.gs_batch_item(x, x, x, x, x, 16, 1, 1e-6, 0))
    calls = [lambda: lib.gs_project(ref(x), v, fr, pr, ref(proj), None, None),
             lambda: lib.gs_project_batch(item, 1, 32, fr, pr, ref(proj), None, None),
             lambda: lib.gs_raster_fwd(ref(proj), ref(srt), 32, fr, pr, v, v, v, v, None, None)]
    if rec != 16:
        calls += [lambda: lib.gs_raster_bwd(ref(x), v, fr, ref(proj), ref(srt), v, v, v, v, v, pr, loss, ref(x), ref(x),
                                            None, v, 1 << 40, None, None),
                  lambda: lib.gs_raster_bwd_batch(item, 1, 32, fr, ref(proj), ref(srt), v, v, v, v, v, pr, loss, None,
                                                  v, 1 << 40, None, None)]
    for call in calls:
        assert call() == G.GS_ERR_INVALID_ARG
        assert b"16-byte aligned" in lib.gs_last_error()
