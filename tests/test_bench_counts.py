"""Counts that bench.py reports: kernels per step, visited pixels, and the traffic
of the captured tile shape only."""
import hashlib
import os
import types

import numpy as np
import pytest

import bench


def test_launched_kernels_per_step():
    # step counter, projection; the sort: record keys, 4 record passes of three
    # kernels, gather, scan of the blocks' sums, offsets, emit, 2 pair passes of
    # three, ranges, 3 of the tile order; forward; workspace check, reverse blend,
    # projection reverse; update
    sort = 1 + 4 * 3 + 3 + 1 + 2 * 3 + 1 + 3
    assert bench.launched_per_step(types.SimpleNamespace(Tx=120, Ty=68)) == 1 + 1 + sort + 1 + 3 + 1 == 34


def test_visited_pixels_counts_the_mask_bits():
    torch = pytest.importorskip("torch")
    m = torch.from_numpy(np.random.RandomState(0).randint(0, 256, 1003).astype(np.uint8))
    want = 64 * int(np.unpackbits(m[:1000].numpy()).sum())
    assert float(bench.visited_pixels(m)) == want


def test_traffic_is_reported_only_for_the_captured_tile(monkeypatch):
    sources = {rel: hashlib.sha256(open(os.path.join(bench.ROOT, rel), "rb").read()).hexdigest()
               for rel in bench.RASTER_BWD_TRAFFIC["sources"]}
    monkeypatch.setattr(bench, "RASTER_BWD_TRAFFIC", dict(bench.RASTER_BWD_TRAFFIC, sources=sources, tile=(16, 16)))
    assert bench.raster_bwd_traffic(1e6, 1000, 2, (16, 16)) == bench.raster_bwd_traffic(1e6, 1000, 2) > 0
    assert bench.raster_bwd_traffic(1e6, 1000, 2, (16, 32)) is None
