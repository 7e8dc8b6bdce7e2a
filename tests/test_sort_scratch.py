"""The scratch of gs_bin_sort does not grow: the allocation-free entry holds a
fixed 32 MiB and refuses what needs more, so a larger need would refuse calls that
it served.  Bounds: what these frames needed with a histogram per tile."""
import os

import pytest

from paper_2602_00395_gb300 import gs3dtr as G

pytestmark = pytest.mark.skipif(not os.path.exists(G.LIB_PATH), reason="library not built")


@pytest.mark.parametrize("views,n,w,h,capacity,tile,most", [
    (2, 160000, 256, 1080, 900000, (32, 16), 32772864), (2000, 32, 1920, 16, 1380000, (16, 16), 27714560),
    (2000, 4, 64, 64, 100, (8, 8), 2500352), (1, 160000, 16, 1080, 900000, (8, 8), 23812608),
    (1, 4000, 1920, 256, 1380000, (8, 8), 22996992), (8, 4, 256, 256, 1380000, (32, 16), 22774784)])
def test_scratch_of_the_sort(views, n, w, h, capacity, tile, most):
    assert 0 < G.gs_bin_sort_workspace_size(n, G.frame_struct(views, w, h, *tile), capacity) <= most
