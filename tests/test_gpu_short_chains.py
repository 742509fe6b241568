"""Frames of many short chains: more 256-track groups of the fit than the frame's size
suggests.  Links, records and assignment equal the oracle's."""
import numpy as np
import pytest

import oracle as orc
import tpcsynth as ts
from gpu_util import compare_tracks, run_gpu

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("ms", [0.02, 0.1, 0.6])
def test_chains_of_a_few_rows(ms):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2102_08862_gb300 import _build, tpcca
    _build.build()
    dev = torch.device("cuda", 0)
    f = ts.generate(ts.continuous(ms, 5))
    m = f.row % 6 < 5
    frame = [a[m] for a in (f.sector, f.row, f.pad, f.time)]
    o = orc.track(*frame, orc.params(n_min=3))
    assert o["n_tracks"] * 20 > len(frame[0]) and o["tracks"]["nhits"].max() <= 5
    tr = tpcca.TimeFrameTracker(len(frame[0]), n_min=3)
    try:
        g = run_gpu(tr, torch, dev, *frame, capacity=o["n_tracks"])
    finally:
        tr.close()
    for name in ("down", "up", "mup"):
        assert np.array_equal(g[name], o[name]), name
    compare_tracks(g, o)
