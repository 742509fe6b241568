"""Ingest of unsorted input: the order of the clusters inside a (sector, row) at the
sizes where the sort changes kernel, with spread, crowded, equal and signed-zero
times.  The order is exact: numpy's stable sort by (sector, row, time, pad)."""
import numpy as np
import pytest

from gpu_util import as_dev

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def env():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2102_08862_gb300 import _build, tpcca
    _build.build()
    return tpcca, torch.device("cuda", 0)


def _times(kind, n, rng):
    if kind == "spread":
        return rng.uniform(-200.0, 3000.0, n)
    if kind == "one burst":  # most clusters in a thousandth of the span
        return np.where(rng.random(n) < 0.9, rng.uniform(100.0, 103.0, n), rng.uniform(0.0, 3000.0, n))
    if kind == "equal":
        return np.full(n, 17.25)
    return rng.choice([-0.0, 0.0, 1.0], n)


def _frame(sizes, kind, seed):
    """One (sector, row) of each size, other rows empty, in random order."""
    rng = np.random.default_rng(seed)
    key = np.concatenate([np.full(m, 40 + 411 * q) for q, m in enumerate(sizes)])
    n = key.size
    time = _times(kind, n, rng)
    pad = rng.integers(0, 40, n) * 0.5 if kind != "equal" else rng.choice([-0.0, 0.0, 2.0], n)
    p = rng.permutation(n)
    return ((key // 152).astype(np.uint16)[p], (key % 152).astype(np.uint16)[p], pad.astype(np.float32)[p],
            time.astype(np.float32)[p])


@pytest.mark.parametrize("kind", ["spread", "one burst", "equal", "zeros"])
@pytest.mark.parametrize("sizes", [[1], [2, 64, 65, 66, 1], [2047, 2048, 2049], [8191, 8192, 8193, 3], [16384, 700]])
def test_order_of_unsorted_clusters(env, sizes, kind):
    tpcca, dev = env
    sector, row, pad, time = _frame(sizes, kind, sum(sizes))
    tr = tpcca.TimeFrameTracker(len(sector))
    try:
        res = tr.track(*as_dev(torch, dev, sector, row, pad, time), sorted_input=False)
        order = tr.debug_links()["order"].cpu().numpy()
        assert res.cluster_track.shape[0] == len(sector)
    finally:
        tr.close()
    key = sector.astype(np.int64) * 152 + row
    assert np.array_equal(order, np.lexsort((pad, time, key)))


def test_row_beyond_the_sort_is_refused(env):
    tpcca, dev = env
    frame = _frame([16385, 5], "spread", 1)
    tr = tpcca.TimeFrameTracker(len(frame[0]))
    try:
        with pytest.raises(tpcca.TpcError) as e:
            tr.track(*as_dev(torch, dev, *frame), sorted_input=False)
        assert e.value.code == tpcca.TPC_ERR_CAPACITY
    finally:
        tr.close()
