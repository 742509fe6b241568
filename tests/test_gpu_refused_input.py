"""Input that a call refuses while its kernels run on: every store stays inside the
caller's arrays, whatever an earlier frame left in the handle, and the next frame is
tracked as ever."""
import numpy as np
import pytest

import oracle as orc
import tpcsynth as ts
from gpu_util import as_dev, run_gpu
from mlp_util import random_net

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

GUARD = 4096  # entries around cluster_track that no call may write
MARK = -77


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


def _guarded_call(tpcca, dev, tr, arrays, sorted_input):
    """One call with cluster_track between guards; (return code, cluster_track, first clusters)."""
    import ctypes
    d = as_dev(torch, dev, *arrays)
    n = d[0].numel()
    buf = torch.full((n + 2 * GUARD,), MARK, dtype=torch.int32, device=dev)
    cnt = ctypes.c_uint32(0)
    cl, out, _, cap = tr.structs(*d, sorted_input=sorted_input, host_count=cnt)
    out.cluster_track = buf.data_ptr() + 4 * GUARD
    rc = tpcca.tpc_track_timeframe(tr.handle, cl, out, torch.cuda.current_stream(dev).cuda_stream)
    torch.cuda.synchronize()
    guard = torch.cat([buf[:GUARD], buf[GUARD + n:]])
    assert bool((guard == MARK).all()), "a store outside cluster_track"
    m = min(cnt.value, cap)
    return rc, buf[GUARD:GUARD + n].cpu().numpy(), tr._out["first_cluster"][:m].cpu().numpy(), cnt.value


def _check_next_frame(tr, dev, frame):
    ref = orc.track(*frame)
    g = run_gpu(tr, torch, dev, *frame)
    for name in ("down", "up", "mup"):
        assert np.array_equal(g[name], ref[name]), name
    assert np.array_equal(g["cluster_track"], ref["cluster_track"])


def _crowd(keys, sizes, seed):
    """Unsorted clusters, sizes[q] of them in (sector, row) keys[q]."""
    rng = np.random.default_rng(seed)
    key = np.repeat(keys, sizes)
    n = key.size
    p = rng.permutation(n)
    return ((key // 152).astype(np.uint16)[p], (key % 152).astype(np.uint16)[p],
            rng.uniform(0.0, 60.0, n).astype(np.float32), rng.uniform(0.0, 3000.0, n).astype(np.float32))


@pytest.mark.parametrize("keys,sizes,code", [
    ([40, 451], [16385, 5], "TPC_ERR_CAPACITY"),
    ([40, 41, 42, 43], [20000, 17000, 16384, 30000], "TPC_ERR_CAPACITY"),  # neighbouring rows
    ([40, 40 * 152 + 7], [500, 17000], "TPC_ERR_INPUT")])                  # sector 40
@pytest.mark.parametrize("follow", [0, 2])
def test_rows_beyond_the_sort(env, frame, keys, sizes, code, follow):
    """More unsorted clusters of a (sector, row) than the sort holds, on a handle that has
    tracked a larger unsorted frame of other rows."""
    tpcca, dev = env
    larger = [np.concatenate([a] * 6)[::-1] for a in frame]
    larger[2] = larger[2] + np.repeat(np.arange(6, dtype=np.float32) * 2.0, len(frame[0]))
    assert len(larger[0]) > sum(sizes)
    tr = tpcca.TimeFrameTracker(len(larger[0]), follow=follow)
    try:
        tr.track(*as_dev(torch, dev, *larger), sorted_input=False)
        bad = _crowd(keys, sizes, 5)
        rc, ct, first, count = _guarded_call(tpcca, dev, tr, bad, False)
        assert rc == getattr(tpcca, code)
        assert ct.min() >= -1 and ct.max() < max(count, 1)  # every entry written
        assert first.size == 0 or (first.min() >= 0 and first.max() < len(bad[0]))
        if follow == 0:
            _check_next_frame(tr, dev, frame)
    finally:
        tr.close()


def _chain_heads(frame, count):
    """First clusters of `count` tracks from the middle of a sorted frame."""
    first = np.sort(orc.track(*frame)["tracks"]["first_cluster"])
    first = first[(first > len(frame[0]) // 4) & (first < 3 * len(frame[0]) // 4)]
    return first[:: max(1, len(first) // count)][:count]


ENTRIES = {"handle": {}, "batched": dict(n_sectors=100), "persistent": dict(persistent=1), "followed": dict(follow=2)}


@pytest.mark.parametrize("entry", list(ENTRIES))
@pytest.mark.parametrize("field,value", [("sector", 200), ("sector", 65535), ("row", 180), ("row", 65535)])
def test_chain_head_outside_the_detector(env, frame, entry, field, value):
    """A sector or row that does not exist, on clusters that head a chain in the middle of
    a sorted frame: the chain's links belong to the rows where the clusters lie."""
    tpcca, dev = env
    heads = _chain_heads(frame, 6)
    assert len(heads) == 6
    bad = [a.copy() for a in frame]
    bad[("sector", "row").index(field)][heads] = value
    tr = tpcca.TimeFrameTracker(len(frame[0]), **ENTRIES[entry])
    try:
        tr.track(*as_dev(torch, dev, *frame))
        rc, ct, first, count = _guarded_call(tpcca, dev, tr, bad, True)
        assert rc == tpcca.TPC_ERR_INPUT
        assert ct.min() >= -1 and ct.max() < max(count, 1)
        assert first.size == 0 or (first.min() >= 0 and first.max() < len(frame[0]))
        if entry != "followed":
            _check_next_frame(tr, dev, frame)
    finally:
        tr.close()


@pytest.mark.parametrize("entry", ["handle", "persistent", "followed"])
@pytest.mark.parametrize("bad", [1, 300, "all"])
@pytest.mark.parametrize("sorted_input", [True, False])
def test_frame_that_begins_outside_the_detector(env, frame, entry, bad, sorted_input):
    """The first clusters, or all of them, in a sector that does not exist, on a handle
    that has tracked a larger frame: they are in no row of the detector and link to nothing."""
    tpcca, dev = env
    larger = [np.concatenate([a] * 2)[::-1] for a in frame]
    larger[2] = larger[2] + np.repeat(np.arange(2, dtype=np.float32) * 2.0, len(frame[0]))
    n = len(frame[0])
    b = [a.copy() for a in frame]
    b[0][:n if bad == "all" else bad] = 40
    tr = tpcca.TimeFrameTracker(len(larger[0]), **ENTRIES[entry])
    try:
        tr.track(*as_dev(torch, dev, *larger), sorted_input=False)
        rc, ct, first, count = _guarded_call(tpcca, dev, tr, b, sorted_input)
        assert rc == tpcca.TPC_ERR_INPUT
        assert ct.min() >= -1 and ct.max() < max(count, 1)  # every entry written
        assert bad != "all" or count == 0
        assert first.size == 0 or (first.min() >= 0 and first.max() < n)
        if entry != "followed":
            _check_next_frame(tr, dev, frame)
    finally:
        tr.close()


@pytest.mark.parametrize("bad", [1, 300, "all"])
def test_noalloc_frame_that_begins_outside_the_detector(env, frame, bad):
    tpcca, dev = env
    import ctypes
    n = len(frame[0])
    b = [a.copy() for a in frame]
    b[0][:n if bad == "all" else bad] = 40
    tr = tpcca.TimeFrameTracker(n)  # (its output tensors)
    try:
        for arrays, code in ((frame, 0), (b, tpcca.TPC_ERR_INPUT), (frame, 0)):
            cnt = ctypes.c_uint32(0)
            d = as_dev(torch, dev, *arrays)
            cl, out, _, _ = tr.structs(*d, host_count=cnt)
            assert tpcca.tpc_track_timeframe_noalloc(None, cl, out, 0) == code
        ref = orc.track(*frame)
        assert np.array_equal(tr._out["cluster_track"][:n].cpu().numpy(), ref["cluster_track"])
    finally:
        tr.close()


@pytest.mark.parametrize("n_sectors", [36, 100])
@pytest.mark.parametrize("field", ["sector", "row"])
def test_listed_cluster_outside_the_detector(env, frame, field, n_sectors):
    """Pruned mode, every window beyond the staging buffers, so that ambiguous clusters go
    through the list; some of them have a sector or a row that does not exist."""
    tpcca, dev = env
    blob = tpcca.pack_blob(*random_net(6, feature_scale=True))
    tr = tpcca.TimeFrameTracker(len(frame[0]), mode=tpcca.TPC_MODE_PRUNED, tau=0.5, row_cap=1, n_sectors=n_sectors)
    try:
        tr.load_mlp(blob)
        tri = tr.extract(*as_dev(torch, dev, *frame))[2].cpu().numpy()
        amb = np.unique(tri[:, 0])
        amb = amb[len(amb) // 4:][:: max(1, len(amb) // 30)][:20]
        assert len(amb) >= 10
        bad = [a.copy() for a in frame]
        bad[("sector", "row").index(field)][amb] = 65535
        tr.track(*as_dev(torch, dev, *frame))
        assert tr.pruned_split()[1] > 0
        rc, ct, first, count = _guarded_call(tpcca, dev, tr, bad, True)
        assert rc == tpcca.TPC_ERR_INPUT
        assert tr.pruned_split()[1] > 0
        assert ct.min() >= -1 and ct.max() < max(count, 1)
        ref = orc.track(*frame, mlp=blob, tau=0.5)
        g = run_gpu(tr, torch, dev, *frame)
        keep = ~ref["band"]
        for name in ("down", "up"):
            assert np.array_equal(g[name][keep], ref[name][keep]), name
    finally:
        tr.close()
