"""Tiles whose time windows are larger than the staging buffers: linked in parts of a
tile, or from global memory where a part of one cluster per thread is still too large.
Links are integers: they equal the oracle's."""
import numpy as np
import pytest

import oracle as orc
from gpu_util import run_gpu
from mlp_util import random_net

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def env():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2102_08862_gb300 import _build, tpcca
    _build.build()
    return tpcca, torch.device("cuda", 0)


def _rows(n_row, group, pads, seed, rows=5):
    """`rows` rows of n_row clusters (one more in every second row).  group > 0: in bursts of
    `group` within a time window of 12 bins, 40 bins apart; else -group of them per 12 bins,
    evenly."""
    rng = np.random.default_rng(seed)
    parts = []
    for r in range(10, 10 + rows):
        n = n_row + r % 2
        if group > 0:
            time = 40.0 * (np.arange(n) // group) + rng.integers(0, 9, n) * 0.75
        else:
            time = rng.uniform(0.0, 12.0 * n / -group, n)
        pad = 5.0 + rng.integers(0, 4 * pads, n) * 0.25
        time, pad = time.astype(np.float32), pad.astype(np.float32)
        order = np.lexsort((pad, time))
        parts.append((np.full(n, 3, np.uint16), np.full(n, r, np.uint16), pad[order], time[order]))
    return [np.concatenate(p) for p in zip(*parts)]


# evenly spread windows that fit in halves, quarters and not at all; bursts that fit only
# inside a burst; a burst as large as the windows of tile 512 and 768, and of tile 1024
CASES = [(3000, -300, 20), (2500, -600, 30), (2600, -900, 40), (2300, -1100, 60), (1600, 700, 40), (1300, 1023, 60),
         (1300, 1024, 60), (2300, 2047, 60), (2300, 2048, 60)]


@pytest.mark.parametrize("n_row,group,pads", CASES)
def test_links_of_tiles_in_parts(env, n_row, group, pads):
    tpcca, dev = env
    frame = _rows(n_row, group, pads, n_row + abs(group))
    ref = orc.track(*frame)
    # (the persistent launch's barriers do not wait for tiles of larger windows than these)
    persistent = [dict(persistent=1)] if abs(group) <= 700 else []
    for kw in [dict(nb_tile=512), {}, dict(nb_tile=1024), dict(row_cap=700)] + persistent:
        tr = tpcca.TimeFrameTracker(len(frame[0]), **kw)
        try:
            g = run_gpu(tr, torch, dev, *frame)
        finally:
            tr.close()
        for name in ("down", "up", "mup"):
            assert np.array_equal(g[name], ref[name]), (kw, name)


@pytest.mark.parametrize("n_row,group", [(1100, -300), (1100, -600), (1060, 1024)])
def test_pruned_links_of_tiles_in_parts(env, n_row, group):
    tpcca, dev = env
    frame = _rows(n_row, group, 60, n_row + abs(group), rows=3)
    blob = tpcca.pack_blob(*random_net(6, feature_scale=True))
    ref = orc.track(*frame, mlp=blob, tau=0.5)
    keep = ~ref["band"]
    assert ref["stats"][2] > 0 and keep.mean() > 0.8
    for tile in (512, 768):
        tr = tpcca.TimeFrameTracker(len(frame[0]), mode=tpcca.TPC_MODE_PRUNED, tau=0.5, nb_tile=tile)
        try:
            tr.load_mlp(blob)
            g = run_gpu(tr, torch, dev, *frame)
            rescored = tr.pruned_clusters()
        finally:
            tr.close()
        assert rescored == ref["stats"][0]
        for name in ("down", "up"):
            assert np.array_equal(g[name][keep], ref[name][keep]), (tile, name)


@pytest.mark.parametrize("group", [-500, -700])
def test_tiles_without_room_for_parts(env, group):
    """One sector whose every row holds clusters, rows of two tiles and one cluster: the
    parts find one free place, or need three; the other tiles stay whole."""
    tpcca, dev = env
    dense = _rows(1537, group, 60, 9)
    one = [np.array(r, dtype=a.dtype) for r, a in zip(zip(*[(0, r, 30.0, 5.0) for r in range(152) if not 10 <= r < 15]),
                                                        dense)]
    frame = [np.concatenate([a, b]) for a, b in zip(dense, one)]
    frame[0][:] = 0
    order = np.lexsort((frame[2], frame[3], frame[1]))
    frame = [a[order] for a in frame]
    ref = orc.track(*frame)
    for kw in ({}, dict(persistent=1)):
        tr = tpcca.TimeFrameTracker(len(frame[0]), n_sectors=1, **kw)
        try:
            g = run_gpu(tr, torch, dev, *frame)
        finally:
            tr.close()
        for name in ("down", "up", "mup"):
            assert np.array_equal(g[name], ref[name]), (kw, name)
