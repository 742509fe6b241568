"""Neighbour finding at the edges of its staging: rows around the tile sizes, time
windows around the 32 entries that a candidate mask holds and around the staged
window's capacity, equal costs everywhere (times and pads on a coarse grid, so that
ties decide), negative times.  Links are integers: they equal the oracle's."""
import numpy as np
import pytest

import oracle as orc
from gpu_util import run_gpu
from mlp_util import random_net

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

ROWS = range(10, 15)


@pytest.fixture(scope="module")
def env():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2102_08862_gb300 import _build, tpcca
    _build.build()
    return tpcca, torch.device("cuda", 0)


def _rows(n_row, group, seed):
    """Five rows of n_row clusters (one more in every second row) in groups of `group`
    that share a time window of 12 bins, 40 bins apart, starting before time 0."""
    rng = np.random.default_rng(seed)
    parts = []
    for r in ROWS:
        n = n_row + r % 2
        k = np.arange(n) // group
        time = 40.0 * k - 100.0 + rng.integers(0, 9, n) * 0.75
        pad = 40.0 + rng.integers(0, 33, n) * 0.25
        order = np.lexsort((pad, time))
        parts.append((np.full(n, 3), np.full(n, r), pad[order], time[order]))
    return [np.concatenate(p).astype(t) for p, t in zip(zip(*parts), (np.uint16, np.uint16, np.float32, np.float32))]


CASES = [(1, 1), (31, 31), (127, 16), (129, 30), (511, 31), (513, 32), (600, 33), (768, 64), (769, 7), (1023, 1023),
         (1025, 1100), (2049, 40)]


@pytest.mark.parametrize("n_row,group", CASES)
def test_links_at_tile_and_window_edges(env, n_row, group):
    tpcca, dev = env
    frame = _rows(n_row, group, n_row + group)
    ref = orc.track(*frame)
    for tile in (512, 768, 1024):
        tr = tpcca.TimeFrameTracker(len(frame[0]), nb_tile=tile)
        try:
            g = run_gpu(tr, torch, dev, *frame)
        finally:
            tr.close()
        for name in ("down", "up", "mup"):
            assert np.array_equal(g[name], ref[name]), (tile, name)


@pytest.mark.parametrize("n_row,group", [(31, 31), (129, 5), (600, 9), (513, 33), (300, 60)])
@pytest.mark.parametrize("tile", [512, 1024])
def test_pruned_links_at_window_edges(env, n_row, group, tile):
    """Ambiguous clusters by mask, by pair (windows over 32 entries) and by list (over
    32 pairs, a full region): every choice outside the score band is the oracle's."""
    tpcca, dev = env
    frame = _rows(n_row, group, 7 * n_row + group)
    blob = tpcca.pack_blob(*random_net(6, feature_scale=True))
    ref = orc.track(*frame, mlp=blob, tau=0.5)
    tr = tpcca.TimeFrameTracker(len(frame[0]), mode=tpcca.TPC_MODE_PRUNED, tau=0.5, nb_tile=tile)
    try:
        tr.load_mlp(blob)
        g = run_gpu(tr, torch, dev, *frame)
        rescored = tr.pruned_clusters()
    finally:
        tr.close()
    keep = ~ref["band"]
    assert rescored == ref["stats"][0] and ref["stats"][2] > 0  # every ambiguous cluster, some choices changed
    assert keep.mean() > 0.9
    for name in ("down", "up"):
        assert np.array_equal(g[name][keep], ref[name][keep]), name
