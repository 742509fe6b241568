"""Rows beyond the 16-bit link index: links up to a row's 65535th cluster are kept, a link
past it is reported."""
import numpy as np
import pytest

import oracle as orc
from gpu_util import as_dev, run_gpu

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

N_ROW = 70000


def _frame(index):
    """A straight track over rows 50..61 whose cluster of row 55 is that row's cluster
    `index` of N_ROW; the others of the row lie on another pad, 2.7 bins apart."""
    other = -60000.0 + 2.7 * np.arange(N_ROW - 1)
    t_track = other[index - 1] + 1.25
    parts = []
    for r in range(50, 62):
        time = np.array([t_track], np.float32)
        pad = np.array([60.0], np.float32)
        if r == 55:
            time = np.concatenate([other, time]).astype(np.float32)
            pad = np.concatenate([np.full(N_ROW - 1, 2.0), pad]).astype(np.float32)
        order = np.lexsort((pad, time))
        parts.append((np.full(len(time), 3, np.uint16), np.full(len(time), r, np.uint16), pad[order], time[order]))
    return [np.concatenate(p) for p in zip(*parts)]


@pytest.mark.parametrize("index,kept", [(100, True), (65534, True), (65535, False), (69998, False)])
@pytest.mark.parametrize("persistent", [0, 1])
def test_link_to_a_late_cluster_of_a_long_row(index, kept, persistent):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2102_08862_gb300 import _build, tpcca
    _build.build()
    dev = torch.device("cuda", 0)
    frame = _frame(index)
    ref = orc.track(*frame)
    assert ref["n_tracks"] == 1 and ref["tracks"]["nhits"][0] == 10  # (the outer two rows head no pair)
    tr = tpcca.TimeFrameTracker(len(frame[0]), persistent=persistent)
    try:
        if kept:
            g = run_gpu(tr, torch, dev, *frame)
            assert np.array_equal(g["cluster_track"], ref["cluster_track"])
        else:
            with pytest.raises(tpcca.TpcError) as e:
                tr.track(*as_dev(torch, dev, *frame))
            assert e.value.code == tpcca.TPC_ERR_CAPACITY
    finally:
        tr.close()
