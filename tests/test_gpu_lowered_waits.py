"""Tracking calls whose look-back and grid-barrier waits may give up after a poll or two:
such a call reports TPC_ERR_TIMEOUT and stores nothing outside the caller's arrays, one
that did not have to wait is right, and with the default limit back the next one is."""
import ctypes

import numpy as np
import pytest

import tpcsynth as ts
from gpu_util import as_dev

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

GUARD, MARK = 4096, -77


@pytest.mark.parametrize("settings", [{}, dict(follow=1), dict(follow=2), dict(fit_variant=1), dict(persistent=1)],
                         ids=["plain", "joins", "links", "warp fit", "persistent"])
@pytest.mark.parametrize("limit", [1, 3])
def test_calls_with_a_lowered_limit(settings, limit):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2102_08862_gb300 import _build, tpcca
    _build.build()
    dev = torch.device("cuda", 0)
    f = ts.generate(ts.c2())
    m = f.sector < 3
    ins = as_dev(torch, dev, f.sector[m], f.row[m], f.pad[m], f.time[m])
    n = int(m.sum())
    buf = torch.full((n + 2 * GUARD,), MARK, dtype=torch.int32, device=dev)
    tr = tpcca.TimeFrameTracker(n, **settings)
    try:
        cnt = ctypes.c_uint32(0)
        cl, out, _, _ = tr.structs(*ins, host_count=cnt)
        out.cluster_track = buf.data_ptr() + 4 * GUARD

        def call():
            rc = tpcca.tpc_track_timeframe(tr.handle, cl, out, torch.cuda.current_stream(dev).cuda_stream)
            torch.cuda.synchronize()
            assert bool((torch.cat([buf[:GUARD], buf[GUARD + n:]]) == MARK).all())
            return rc, cnt.value, buf[GUARD:GUARD + n].cpu().numpy()

        rc, count, want = call()
        assert rc == tpcca.TPC_OK and count > 1000
        assert tpcca.tpc_tf_set_spin_limit(tr.handle, limit) == tpcca.TPC_OK
        for _ in range(10):
            rc, got_count, got = call()
            assert rc in (tpcca.TPC_OK, tpcca.TPC_ERR_TIMEOUT)
            if rc == tpcca.TPC_OK:
                assert got_count == count and np.array_equal(got, want)
        assert tpcca.tpc_tf_set_spin_limit(tr.handle, 0) == tpcca.TPC_OK
        rc, got_count, got = call()
        assert rc == tpcca.TPC_OK and got_count == count and np.array_equal(got, want)
    finally:
        tr.close()
