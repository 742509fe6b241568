"""Ingest tables on sparse frames: sizes around the 8 clusters of a thread, the 256 of a
warp and the 32768 of the start list's tile, empty rows and sectors at either end, and a
batched call with empty instances.  Links and cluster -> track equal the oracle's."""
import numpy as np
import pytest

import oracle as orc
import tpcsynth as ts
from gpu_util import run_gpu

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def env():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2102_08862_gb300 import _build, tpcca
    _build.build()
    return tpcca, torch.device("cuda", 0)


@pytest.fixture(scope="module")
def frame():
    f = ts.generate(ts.continuous(0.05, 11))
    return f.sector, f.row, f.pad, f.time


def _check(g, ref):
    for name in ("down", "up", "mup"):
        assert np.array_equal(g[name], ref[name]), name
    assert g["n_tracks"] == ref["n_tracks"]
    assert np.array_equal(g["cluster_track"], ref["cluster_track"])


@pytest.mark.parametrize("n", [1, 7, 8, 9, 255, 256, 257, 2047, 2049, 32767, 32768, 32769, 70001])
@pytest.mark.parametrize("last", [False, True])
def test_first_and_last_clusters_of_a_frame(env, frame, n, last):
    """The first n clusters (sectors from 0 on) or the last n (up to sector 35)."""
    tpcca, dev = env
    part = [a[-n:] if last else a[:n] for a in frame]
    tr = tpcca.TimeFrameTracker(len(frame[0]))
    try:
        _check(run_gpu(tr, torch, dev, *part), orc.track(*part))
    finally:
        tr.close()


@pytest.mark.parametrize("keep", ["middle sector", "two far sectors", "no outer rows", "rows in blocks"])
def test_empty_rows_and_sectors(env, frame, keep):
    tpcca, dev = env
    s, r = frame[0], frame[1]
    m = {"middle sector": s == 17, "two far sectors": (s == 2) | (s == 33), "no outer rows": (r > 20) & (r < 130),
         "rows in blocks": r % 40 < 30}[keep]
    part = [a[m] for a in frame]
    tr = tpcca.TimeFrameTracker(len(frame[0]))
    try:
        _check(run_gpu(tr, torch, dev, *part), orc.track(*part))
    finally:
        tr.close()


def test_batch_with_empty_instances(env, frame):
    tpcca, dev = env
    m = frame[0] < 3
    part = [a[m] for a in frame]
    ids = np.array([4, 57, 98], np.uint16)[part[0]]
    tr = tpcca.TimeFrameTracker(len(ids), n_sectors=100)
    try:
        _check(run_gpu(tr, torch, dev, ids, *part[1:]), orc.track(*part))
    finally:
        tr.close()
