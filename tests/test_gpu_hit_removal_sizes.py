"""Hit removal at the edges of its 2048-cluster tiles and of a warp's 32, with nothing,
everything and a random part kept, and with an assignment array that is 4-byte aligned
only: byte for byte numpy's selection."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("n", [1, 31, 33, 2047, 2048, 2049, 6144, 70001])
@pytest.mark.parametrize("kept", [0.0, 0.5, 1.0])
def test_selection_at_tile_edges(n, kept):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2102_08862_gb300 import tpcca
    rng = np.random.default_rng(n)
    fields = [rng.integers(0, 36, n).astype(np.int16), rng.integers(0, 152, n).astype(np.int16),
              rng.random(n, np.float32), rng.random(n, np.float32)]
    track = np.where(rng.random(n) < kept, rng.integers(0, 1000, n), -1).astype(np.int32)
    dev = [torch.from_numpy(a).cuda() for a in fields]
    tr = tpcca.TimeFrameTracker(n)
    try:
        for shift in (0, 1):
            owner = torch.full((n + 1,), 7, dtype=torch.int32, device="cuda")[shift:shift + n]
            owner.copy_(torch.from_numpy(track))
            out = tr.remove_unassigned(*dev, owner)
            m = track >= 0
            for name, want in zip(("sector", "row", "pad", "time", "track"), fields + [track]):
                assert np.array_equal(out[name].cpu().numpy(), want[m]), (name, shift)
    finally:
        tr.close()
