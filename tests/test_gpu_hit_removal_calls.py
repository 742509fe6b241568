"""Hit removal without a tracking call before it, and one call after another: every call
leaves the handle's counter as it found it."""
import numpy as np
import pytest

from gpu_util import as_dev

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def test_removal_on_a_fresh_handle_and_again():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2102_08862_gb300 import _build, tpcca
    _build.build()
    dev = torch.device("cuda", 0)
    rng = np.random.default_rng(2)
    tr = tpcca.TimeFrameTracker(200_000)
    try:
        assert tpcca.tpc_tf_status(tr.handle, 0) == tpcca.TPC_OK
        for n in (200_000, 1, 0, 2048, 2049, 40_000, 40_000):
            frame = (rng.integers(0, 36, n).astype(np.uint16), rng.integers(0, 152, n).astype(np.uint16),
                     rng.random(n, np.float32), rng.random(n, np.float32))
            track = np.where(rng.random(n) < 0.7, rng.integers(0, 1000, n), -1).astype(np.int32)
            out = tr.remove_unassigned(*as_dev(torch, dev, *frame), torch.from_numpy(track).to(dev))
            keep = track >= 0
            for name, a in zip(("sector", "row", "pad", "time", "track"), frame + (track,)):
                got = out[name].cpu().numpy()
                assert np.array_equal(got.view(a.dtype), a[keep]), (n, name)
    finally:
        tr.close()
