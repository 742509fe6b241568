"""A captured call and the classifier: the graph holds part of the weights (the scorer's
standardisation and output layer are kernel parameters), so new weights need a new one."""
import numpy as np
import pytest

import tpcsynth as ts
from gpu_util import as_dev
from mlp_util import random_net

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("engine", [0, 1])
def test_replay_after_loading_other_weights(engine):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2102_08862_gb300 import _build, tpcca
    _build.build()
    dev = torch.device("cuda", 0)
    f = ts.generate(ts.c2())
    m = f.sector < 2
    ins = as_dev(torch, dev, f.sector[m], f.row[m], f.pad[m], f.time[m])
    n = int(m.sum())
    nets = [random_net(6, feature_scale=True), random_net(17, feature_scale=True)]
    nets[1] = (nets[1][0] + 0.3, nets[1][1] * 1.5, nets[1][2])
    blobs = [tpcca.pack_blob(*net) for net in nets]
    tr = tpcca.TimeFrameTracker(n, mode=tpcca.TPC_MODE_PRUNED, tau=0.5, mlp_engine=engine)
    try:
        direct, replay = [], []
        for blob in blobs:
            tr.load_mlp(blob)
            direct.append(tr.track(*ins).cluster_track.cpu().numpy().copy())
        for blob in blobs + blobs[:1]:
            tr.load_mlp(blob)
            for _ in range(2):  # captured, then replayed
                tr._out["cluster_track"].fill_(-7)
                tr.track_graph(*ins)
                torch.cuda.synchronize()
            replay.append(tr._out["cluster_track"][:n].cpu().numpy().copy())
    finally:
        tr.close()
    assert not np.array_equal(direct[0], direct[1])
    for got, want in zip(replay, direct + direct[:1]):
        assert np.array_equal(got, want)
