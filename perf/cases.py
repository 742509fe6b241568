"""The workloads whose speed this repository answers for, as a user's program calls them.

A case is one call of the public Python API (paper_2102_08862_gb300.tpcca) on one kind of input:

* ``frame``  a time frame on the device through tpc_track_timeframe (plain or learned-pruned, sorted or shuffled
             clusters, with or without track following and cross-sector links), waiting for the number of tracks;
* ``batch``  many independent (sector x time frame) instances in one call, replayed from a CUDA graph;
* ``host``   a frame in page-locked host buffers through tpc_track_timeframe_host, copies included;
* ``score``  the link classifier on a dense block of feature rows;
* ``train``  one gradient of the classifier's trainer;
* ``remove`` hit removal: the clusters attached to a track, compacted.

Frames come from the seeded generator ``tpcsynth`` that the tests and the benchmark use (helices, pile-up and noise of a
50 kHz continuous readout, about 8.88e4 clusters per sector and millisecond).  A frame is as long as it takes to hold
exactly ``clusters`` clusters, and the output arrays are a program's own, allocated once and zero where no track is."""
from __future__ import annotations

import ctypes
import json
import math
import os

import numpy as np
import torch

import tpcsynth
from paper_2102_08862_gb300 import tpcca

_ROOT = os.path.dirname(os.path.dirname(os.path.abspath(tpcca.__file__)))
_WEIGHTS = os.path.join(_ROOT, "paper_2102_08862_gb300", "weights", "link_classifier")
_FLOATS = ("params", "cov", "t_ref", "x", "chi2")
_WHOLE = ("ndf", "nhits", "first_cluster", "sector", "row_first", "row_last", "status")


def listed():
    frame = {"kind": "frame", "sector": -1, "mode": "plain", "follow": 0, "sorted": True}
    return [
        # the smallest frame in use: one collision seen by one sector; launches and latency count
        {**frame, "name": "one_collision", "clusters": 7600, "sector": 0},
        # a short online frame of the whole detector (0.3 ms)
        {**frame, "name": "frame_0.3ms", "clusters": 959_003},
        # an ordinary frame of the whole detector (2 ms)
        {**frame, "name": "frame_2ms", "clusters": 6_171_551},
        # clusters in arrival order instead of the clusteriser's: sorted by the call itself
        {**frame, "name": "frame_2ms_shuffled", "clusters": 6_171_551, "sorted": False},
        # one sector of a full frame, as a shard of a frame split over several workers, with the learned classifier
        {**frame, "name": "sector_10ms_pruned", "clusters": 887_777, "sector": 5, "mode": "pruned"},
        # the benchmark's workload: a full 10 ms frame with the learned classifier
        {**frame, "name": "frame_10ms_pruned", "clusters": 31_960_037, "mode": "pruned"},
        # the complete tracker on 5 ms: following, joins and links across sector boundaries
        {**frame, "name": "frame_5ms_links", "clusters": 16_765_809, "follow": 2},
        # many dense instances of unlike size in one replayed call, with the learned classifier
        {"name": "batch_pruned", "kind": "batch", "instances": 48, "largest": 400_000, "mode": "pruned"},
        # a 5 ms frame in a readout host's page-locked memory: copies in and out are part of the call
        {"name": "host_5ms_pruned", "kind": "host", "clusters": 16_765_809, "mode": "pruned"},
        # the classifier alone on a large block of candidate pairs
        {"name": "score_5M", "kind": "score", "rows": 5_200_000},
        # one gradient of the classifier's training at its batch size
        {"name": "train_8k", "kind": "train", "rows": 8192},
        # the compression step after tracking
        {"name": "remove_5ms", "kind": "remove", "clusters": 16_765_809},
    ]


def _log(rng, lo, hi):
    return int(math.exp(rng.uniform(math.log(lo), math.log(hi))))


def draw(rng):
    kind = rng.choice(["frame"] * 7 + ["batch", "host", "score", "train", "remove"])
    mode = rng.choice(["plain", "pruned"])
    if kind == "frame":
        follow = rng.choice([0, 0, 0, 1, 2])
        in_order = rng.random() < 0.75
        sector = rng.choice([-1, -1, rng.randrange(36)])
        if sector >= 0:
            follow = min(follow, 1)
            n = _log(rng, 20_000, 1_000_000)
        else:
            n = _log(rng, 300_000, 9_000_000 if follow or not in_order else 29_000_000)
        return {"kind": kind, "clusters": n, "sector": sector, "mode": mode, "follow": follow, "sorted": in_order}
    if kind == "batch":
        return {"kind": kind, "instances": rng.randrange(7, 60), "largest": _log(rng, 30_000, 400_000), "mode": mode}
    if kind == "host":
        return {"kind": kind, "clusters": _log(rng, 600_000, 14_000_000), "mode": mode}
    if kind == "remove":
        return {"kind": kind, "clusters": _log(rng, 600_000, 16_000_000)}
    if kind == "score":
        return {"kind": kind, "rows": _log(rng, 1000, 5_200_000) | 1}
    return {"kind": kind, "rows": rng.randrange(257, 8192) | 1}


# ------------------------------------------------------------------ inputs
def _cut(f, n, one_collision):
    """(sector, row, pad, time) on the device of exactly n clusters of a frame with more: its first n in time, or, of one
    collision, its noise and as many whole tracks as it takes."""
    arrays = [torch.from_numpy(a).cuda() for a in (f.sector.view(np.int16), f.row.view(np.int16), f.pad, f.time)]
    rank = torch.from_numpy(f.label).cuda() if one_collision else arrays[3]
    last = torch.kthvalue(rank, n).values
    keep = rank < last
    ties = torch.nonzero(rank == last).squeeze(1)
    keep[ties[:n - int(keep.sum())]] = True
    return [a[keep] for a in arrays]


def _continuous(n, sector, seed, rate_khz=50.0):
    """The first n clusters of a continuous readout of one sector, or of all with sector -1."""
    ms = n / (tpcsynth.CLUSTERS_PER_SECTOR_MS_50KHZ * (36 if sector < 0 else 1) * rate_khz / 50.0)
    longer = 1.1 + 0.25 / math.sqrt(ms * rate_khz)
    while True:
        cfg = tpcsynth.continuous(ms * longer, seed)
        cfg.sector_only = sector
        cfg.rate_khz = rate_khz
        f = tpcsynth.generate(cfg)
        if f.n >= n:
            return _cut(f, n, False)
        longer *= 1.3


def _frame_arrays(case, seed):
    """(sector, row, pad, time) of a frame on the device, sorted or in a random order."""
    n = case["clusters"]
    if n < 10_000:
        cfg = tpcsynth.c1(seed + 1)
        cfg.n_tracks = 260
        arrays = _cut(tpcsynth.generate(cfg), n, True)
    else:
        arrays = _continuous(n, case.get("sector", -1), seed + 1)
    if not case.get("sorted", True):
        gen = torch.Generator(device="cuda")
        gen.manual_seed(seed)
        order = torch.randperm(n, device="cuda", generator=gen)
        arrays = [a[order] for a in arrays]
    return arrays


def _batch_sizes(case):
    """Cluster counts of the instances, evenly spread over their logarithm from 1e4, in an order of no meaning."""
    m = case["instances"]
    sizes = [int(1e4 * (case["largest"] / 1e4) ** (k / max(1, m - 1))) for k in range(m)]
    return [sizes[(k * 29) % m] if math.gcd(29, m) == 1 else sizes[k] for k in range(m)]


def _batch_arrays(case, seed):
    """The instances one after another, the sector field holding the instance's number."""
    lengths = np.random.default_rng(seed).uniform(0.2, 10.0, case["instances"])
    parts = []
    for k, n in enumerate(_batch_sizes(case)):
        rate = 50.0 * n / (tpcsynth.CLUSTERS_PER_SECTOR_MS_50KHZ * lengths[k])
        arrays = _continuous(n, k % 36, seed * 1009 + k + 1, rate)
        arrays[0] = torch.full_like(arrays[0], k)
        parts.append(arrays)
    return [torch.cat(p) for p in zip(*parts)]


def _classifier():
    with open(_WEIGHTS + ".bin", "rb") as f:
        blob = f.read()
    with open(_WEIGHTS + ".json") as f:
        return blob, float(json.load(f)["tau"])


def _tracker(n, mode, **settings):
    blob, tau = _classifier()
    if mode == "plain":
        return tpcca.TimeFrameTracker(n, **settings)
    tracker = tpcca.TimeFrameTracker(n, mode=tpcca.TPC_MODE_PRUNED, tau=tau, **settings)
    tracker.load_mlp(blob)
    return tracker


def _features(rows, seed):
    """Feature rows with the classifier's own means and spreads."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    mean, inv_std, _ = tpcca.unpack_blob(_classifier()[0])
    z = torch.randn(rows, tpcca.MLP_IN, device="cuda", generator=gen)
    return z / torch.from_numpy(inv_std).cuda() + torch.from_numpy(mean).cuda()


def _training_rows(case, seed):
    """A pool of feature rows with labels, and the indices of one shuffled batch."""
    rows = case["rows"]
    pool = 16 * rows
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed + 1)
    feat = _features(pool, seed)
    label = (torch.rand(pool, device="cuda", generator=gen) < 0.36).to(torch.uint8)
    index = torch.randperm(pool, device="cuda", generator=gen)[:rows].to(torch.int32)
    return feat, label, index


def _capacity(n):
    """Track records a program provides for n clusters (a track takes about 70)."""
    return n // 48 + 64


def prepare(case, seed):
    kind = case["kind"]
    if kind == "score":
        tracker = _tracker(1024, "plain")
        tracker.load_mlp(_classifier()[0])
        return {"kind": kind, "tracker": tracker, "feat": _features(case["rows"], seed)}
    if kind == "train":
        feat, label, index = _training_rows(case, seed)
        trainer = tpcca.Trainer(_classifier()[0], max_batch=case["rows"])
        return {"kind": kind, "trainer": trainer, "feat": feat, "label": label, "index": index}
    clusters = _batch_arrays(case, seed) if kind == "batch" else _frame_arrays(case, seed)
    n = clusters[0].numel()
    settings = {"n_sectors": case["instances"]} if kind == "batch" else {"follow": case.get("follow", 0)}
    tracker = _tracker(n, case.get("mode", "plain"), **settings)
    pinned = kind == "host"
    if pinned:
        clusters = [a.cpu().pin_memory() for a in clusters]
    cap = _capacity(n)
    out = {"cluster_track": (n, torch.int32), "params": ((cap, 5), torch.float32), "cov": ((cap, 15), torch.float32)}
    out.update({k: (cap, torch.float32) for k in ("t_ref", "x", "chi2")})
    out.update({k: (cap, torch.int32) for k in ("ndf", "nhits", "first_cluster")})
    out.update({k: (cap, torch.int16) for k in ("sector", "row_first", "row_last")})
    out["status"] = (cap, torch.uint8)
    if tracker.cfg.follow == 2:
        out["next_track"] = (cap, torch.int32)
    where = {"pin_memory": True} if pinned else {"device": "cuda"}
    out = {k: torch.zeros(shape, dtype=dtype, **where) for k, (shape, dtype) in out.items()}
    count = torch.zeros(1, dtype=torch.int32, **where)  # written by the device, or by the call on a host buffer
    cl = tpcca.tpc_clusters(n=n, flags=tpcca.TPC_INPUT_SORTED if case.get("sorted", True) else 0,
                            **{k: a.data_ptr() for k, a in zip(("sector", "row", "pad", "time"), clusters)})
    tr = tpcca.tpc_tracks(track_capacity=cap, n_tracks=count.data_ptr(), **{k: v.data_ptr() for k, v in out.items()})
    host_count = tpcca.c_u32(0)
    if kind in ("frame", "remove"):  # a call with this pointer waits for its result
        tr.n_tracks_host = ctypes.addressof(host_count)
    state = {"kind": kind, "tracker": tracker, "clusters": clusters, "cl": cl, "tr": tr, "out": out, "count": count,
             "host_count": host_count}
    if kind == "remove":
        _check(tpcca.tpc_track_timeframe(tracker.handle, cl, tr, _stream()))
        kept = {k: torch.zeros_like(a) for k, a in zip(("sector", "row", "pad", "time"), clusters)}
        kept["track"] = torch.zeros_like(out["cluster_track"])
        return {**state, "kept": kept}
    return state


def _stream():
    return torch.cuda.current_stream().cuda_stream


def _check(code):
    if code != tpcca.TPC_OK:
        raise RuntimeError(tpcca.tpc_last_error())


# ------------------------------------------------------------------ one pass
def run(state):
    kind = state["kind"]
    if kind == "score":
        return {"logit": state["tracker"].score(state["feat"])}
    if kind == "train":
        grad, loss = state["trainer"].gradient(state["feat"], state["label"], state["index"])
        return {"grad": grad, "loss": loss}
    handle, cl, tr = state["tracker"].handle, state["cl"], state["tr"]
    if kind == "frame":
        _check(tpcca.tpc_track_timeframe(handle, cl, tr, _stream()))
        return {**state["out"], "n_tracks": state["host_count"].value}
    if kind == "batch":
        _check(tpcca.tpc_track_timeframe_graph(handle, cl, tr, _stream()))
        return {**state["out"], "n_tracks": state["count"]}
    if kind == "host":
        _check(tpcca.tpc_track_timeframe_host(handle, cl, tr, _stream()))
        return {**state["out"], "n_tracks": state["count"]}
    kept = state["kept"]
    _check(tpcca.load().tpc_tf_remove_unassigned(
        handle, ctypes.byref(cl), state["out"]["cluster_track"].data_ptr(), kept["sector"].data_ptr(),
        kept["row"].data_ptr(), kept["pad"].data_ptr(), kept["time"].data_ptr(), kept["track"].data_ptr(),
        state["count"].data_ptr(), _stream()))
    return {**kept, "count": state["count"]}


def work(case):
    kind = case["kind"]
    if kind == "score":  # 12 features in, a logit out; 12-64-64-1
        return {"bytes": 52.0 * case["rows"], "flops": 2.0 * (12 * 64 + 64 * 64 + 64) * case["rows"]}
    if kind == "train":  # forward and twice that backward; the gathered rows, the gradient
        return {"bytes": 53.0 * case["rows"] + 4.0 * tpcca.MLP_NPARAM,
                "flops": 6.0 * (12 * 64 + 64 * 64 + 64) * case["rows"]}
    n = sum(_batch_sizes(case)) if kind == "batch" else case["clusters"]
    if kind == "remove":  # 16 B of every cluster's track id and fields in, 16 B of the nine tenths kept out
        return {"bytes": (4.0 + 0.9 * 28.0) * n, "flops": 0.0}
    # clusters in (12 B) and their track ids out (4 B), a record of 111 B for a track of 65 clusters; a Kalman step
    # costs about 200 operations
    return {"bytes": 16.0 * n + 111.0 * n / 72.0, "flops": 200.0 * 0.9 * n}


# ------------------------------------------------------------------ the same in 64 bits
def exact(case, seed):
    kind = case["kind"]
    if kind == "score":
        return {"logit": _exact_logits(_features(case["rows"], seed))}
    if kind == "train":
        grad, loss = _exact_gradient(*_training_rows(case, seed))
        return {"grad": grad, "loss": loss}
    # the classifier's choices and the follower's hang on thresholds of 32-bit values: which clusters make a track is
    # part of the result there, and a 64-bit evaluation gives other tracks; hit removal computes nothing
    if kind == "remove" or case["mode"] != "plain" or case.get("follow"):
        return None
    arrays = _batch_arrays(case, seed) if kind == "batch" else _frame_arrays(case, seed)
    n = arrays[0].numel()
    if n > 8_000_000:  # beyond about 20 seconds
        return None
    out = {}
    for name, value in _exact_tracks(*arrays).items():
        out[name] = torch.zeros(_capacity(n), *value.shape[1:], dtype=torch.float64, device="cuda")
        out[name][:value.shape[0]] = value
    return {**out, "cluster_track": None, "n_tracks": None, **{k: None for k in _WHOLE}}


def _exact_logits(feat):
    """The network at 64 bits on its 16-bit operands: standardised inputs, weights and first hidden layer are rounded to
    bfloat16 (that is the network's definition), everything else is double."""
    mean, inv_std, theta = (torch.from_numpy(a).cuda() for a in tpcca.unpack_blob(_classifier()[0]))
    w1, b1, w2, b2, w3, b3 = _parameters(theta)
    half = lambda v: v.to(torch.bfloat16).double()  # noqa: E731
    out = []
    for part in feat.split(1 << 20):
        x = half((part - mean) * inv_std)
        h1 = half(torch.relu(x @ half(w1).T + b1.double()).float())
        h2 = torch.relu(h1 @ half(w2).T + b2.double())
        out.append(h2 @ half(w3) + b3.double())
    return torch.cat(out)


def _parameters(theta):
    parts, at = [], 0
    for _, shape in tpcca.MLP_PARAM_SHAPES:
        size = math.prod(shape)
        parts.append(theta[at:at + size].reshape(shape))
        at += size
    return parts


def _exact_gradient(feat, label, index):
    mean, inv_std, theta = (torch.from_numpy(a).cuda() for a in tpcca.unpack_blob(_classifier()[0]))
    theta = theta.double().requires_grad_(True)
    w1, b1, w2, b2, w3, b3 = _parameters(theta)
    rows = index.long()
    x = (feat[rows].double() - mean.double()) * inv_std.double()
    logit = torch.relu(torch.relu(x @ w1.T + b1) @ w2.T + b2) @ w3 + b3
    loss = torch.nn.functional.binary_cross_entropy_with_logits(logit, label[rows].double())
    loss.backward()
    return theta.grad, float(loss.detach())


_ROWS = 152
_DX = 160.0 / 151.0
_WY, _WT, _COST = 1280000, 384, 147456000000
_BZ, _CM_PER_BIN = 0.00149896229, 0.516


def _ragged(first, count):
    """(owner, element) of the ranges [first, first + count), one after another."""
    owner = torch.repeat_interleave(torch.arange(count.numel(), device=count.device), count)
    start = torch.cumsum(count, 0) - count
    return owner, torch.arange(owner.numel(), device=count.device) - start[owner] + first[owner]


def _candidates(t, y, key, order_key, span, i, step):
    """For the clusters i: those of the row `step` away inside both windows, as (position in i, cluster), in order."""
    lo = torch.searchsorted(order_key, (key[i] + step) * span + t[i] - _WT)
    hi = torch.searchsorted(order_key, (key[i] + step) * span + t[i] + _WT, right=True)
    owner, c = _ragged(lo, hi - lo)
    near = (y[c] - y[i[owner]]).abs() <= _WY
    return owner[near], c[near]


def _links(t, y, key, row):
    """Best straight neighbour pair of every cluster of rows 1..150, then the claims of rows 0 and 151."""
    n = t.numel()
    dev = t.device
    t = t - t.min() + _WT + 1
    span = int(t.max()) + _WT + 2
    order_key = key * span + t
    down = torch.full((n,), -1, dtype=torch.int64, device=dev)
    up = down.clone()
    best_cost = down.clone()
    middle = torch.nonzero((row > 0) & (row < _ROWS - 1)).squeeze(1)
    for i in middle.split(1 << 21):
        oj, cj = _candidates(t, y, key, order_key, span, i, -1)
        ok, ck = _candidates(t, y, key, order_key, span, i, 1)
        nk = torch.bincount(ok, minlength=i.numel())
        first_k = torch.cumsum(nk, 0) - nk
        pj, pk = _ragged(first_k[oj], nk[oj])
        o, j, k = oj[pj], cj[pj], ck[pk]
        dy = y[j] + y[k] - 2 * y[i[o]]
        dz = 5160 * (t[j] + t[k] - 2 * t[i[o]])
        cost = dy * dy + dz * dz
        keep = cost <= _COST
        o, j, k, cost = o[keep], j[keep], k[keep], cost[keep]
        for rank in range(3):  # smallest cost, then j, then k
            value = (cost, j, k)[rank]
            low = torch.full((i.numel(),), 1 << 62, dtype=torch.int64, device=dev).scatter_reduce(0, o, value, "amin")
            sel = value == low[o]
            o, j, k, cost = o[sel], j[sel], k[sel], cost[sel]
        down[i[o]], up[i[o]], best_cost[i[o]] = j, k, cost
    for edge, mine, link in ((1, up, down), (_ROWS - 2, down, up)):
        claim = torch.nonzero((row == edge) & (link >= 0)).squeeze(1)
        target, cost = link[claim], best_cost[claim]
        low = torch.full((n,), 1 << 62, dtype=torch.int64, device=dev).scatter_reduce(0, target, cost, "amin")
        sel = cost == low[target]
        claim, target = claim[sel], target[sel]
        first = torch.full((n,), 1 << 62, dtype=torch.int64, device=dev).scatter_reduce(0, target, claim, "amin")
        has = first < (1 << 62)
        mine[has] = first[has]
    return down, up


def _exact_tracks(sector, row, pad, time, n_min=10):
    key = sector.long() * _ROWS + row.long()
    order = torch.arange(key.numel(), device=key.device)
    for value in (pad, time, key):  # (sector, row, time, pad, input index)
        order = order[torch.sort(value[order], stable=True).indices]
    key, row, pad, time = key[order], row[order], pad[order], time[order]
    row = row.long()
    n, dev = key.numel(), key.device
    npads = 66 + (144 * row + 151) // 302
    pitch = 4000 + (4000 * row + 151) // 302
    t_q = torch.round(time.double() * 64).long()
    y_q = (torch.round(pad.double() * 64).long() - 32 * (npads - 1)) * pitch
    down, up = _links(t_q, y_q, key, row)
    at = torch.arange(n, device=dev)
    mutual_up = torch.where((up >= 0) & (down[up.clamp_min(0)] == at), up, -1)
    mutual_down = (down >= 0) & (up[down.clamp_min(0)] == at)
    start = torch.nonzero((mutual_up >= 0) & ~mutual_down).squeeze(1)
    chain = torch.full((_ROWS, start.numel()), -1, dtype=torch.int64, device=dev)
    c = start
    for s in range(_ROWS):
        chain[s] = c
        c = torch.where(c >= 0, mutual_up[c.clamp_min(0)], -1)
    length = (chain >= 0).sum(0)
    chain, length = chain[:, length >= n_min], length[length >= n_min]
    y = (pad.double() - 0.5 * (npads - 1).double()) * pitch.double() * 1e-4
    return _kalman(chain, length, row, y, time)


def _kalman(chain, length, row, y, time):
    m = length.numel()
    dev = chain.device
    col = torch.arange(m, device=dev)
    first, mid, last = chain[0], chain[length // 2, col], chain[length - 1, col]
    t_ref = time[first]
    zeta = lambda c: _CM_PER_BIN * (time[c].double() - t_ref.double())  # noqa: E731
    r0 = row[first]
    ax, bx = _DX * (row[mid] - r0).double(), _DX * (row[last] - r0).double()
    ay, by = y[mid] - y[first], y[last] - y[first]
    d01, d02, d12 = torch.hypot(ax, ay), torch.hypot(bx, by), torch.hypot(bx - ax, by - ay)
    curv = 2.0 * (ax * by - bx * ay) / (d01 * d02 * d12)
    u = 0.5 * curv * d02
    straight = u.abs() >= 0.999
    sin0 = torch.where(straight, by / d02, by / d02 * torch.sqrt((1 - u * u).clamp_min(0)) - bx / d02 * u)
    straight = straight | (sin0.abs() >= 0.999)
    curv, u = torch.where(straight, 0.0, curv), torch.where(straight, 0.0, u)
    sin0 = torch.where(straight, by / d02, sin0)
    p = torch.stack([y[first], torch.zeros_like(y[first]), sin0, zeta(last) / (d02 * _arc(u)), -curv / _BZ], 1)
    vy, vz = 0.06 ** 2, 0.0516 ** 2
    cov = torch.diag(torch.tensor([vy, vz, 0.01, 0.01, 0.01], dtype=torch.float64, device=dev)).repeat(m, 1, 1)
    chi2 = torch.zeros(m, dtype=torch.float64, device=dev)
    used = torch.ones(m, dtype=torch.int64, device=dev)
    active = torch.ones(m, dtype=torch.bool, device=dev)
    for s in range(1, int(length.max()) if m else 0):
        c = chain[s].clamp_min(0)
        curv = -_BZ * p[:, 4]
        s1, s2 = p[:, 2], p[:, 2] + curv * _DX
        active = active & (length > s) & (s1.abs() < 0.999) & (s2.abs() < 0.999)
        a = torch.nonzero(active).squeeze(1)
        if not a.numel():
            break
        q, f = _transport(p[a], s2[a])
        v = f @ cov[a] @ f.transpose(1, 2)
        res = torch.stack([y[c[a]] - q[:, 0], _CM_PER_BIN * (time[c[a]].double() - t_ref[a].double()) - q[:, 1]], 1)
        gate = v[:, :2, :2] + torch.diag(torch.tensor([vy, vz], dtype=torch.float64, device=dev))
        inv = torch.linalg.inv(gate)
        gain = v[:, :, :2] @ inv
        p[a] = q + (gain @ res.unsqueeze(2)).squeeze(2)
        v = v - gain @ v[:, :2, :]
        cov[a] = 0.5 * (v + v.transpose(1, 2))
        chi2[a] += (res.unsqueeze(1) @ inv @ res.unsqueeze(2)).reshape(-1)
        used[a] += 1
    i, j = torch.tril_indices(5, 5, device=dev)
    x = 85.0 + _DX * (r0 + used - 1).double()
    return {"params": p, "cov": cov[:, i, j], "t_ref": t_ref.double(), "x": x, "chi2": chi2}


def _arc(u):
    """asin(u) / u."""
    return torch.where(u.abs() < 1e-4, 1 + u * u / 6, torch.asin(u) / torch.where(u == 0, 1.0, u))


def _transport(p, s2):
    """State one row outward and the Jacobian of that step."""
    s1, t = p[:, 2], p[:, 3]
    curv = -_BZ * p[:, 4]
    c1, c2 = torch.sqrt(1 - s1 * s1), torch.sqrt(1 - s2 * s2)
    dy = _DX * (s1 + s2) / (c1 + c2)
    chord = torch.sqrt(_DX * _DX + dy * dy)
    u = 0.5 * curv * chord
    arc = chord * _arc(u)
    d = c1 + c2
    y_s = _DX * (2 * d + (s1 + s2) * (s1 / c1 + s2 / c2)) / (d * d)
    y_c = _DX * _DX * (d + (s1 + s2) * s2 / c2) / (d * d)
    g = 1.0 / torch.sqrt(1 - u * u)
    # d(asin(u)/u)/du, by its series where u is small
    arc_d = torch.where(u.abs() < 1e-2, u / 3 + 0.3 * u ** 3 + 15 / 56 * u ** 5,
                        (u * g - torch.asin(u)) / torch.where(u == 0, 1.0, u * u))
    f = torch.eye(5, dtype=torch.float64, device=p.device).repeat(p.shape[0], 1, 1)
    f[:, 0, 2], f[:, 0, 4] = y_s, -_BZ * y_c
    f[:, 1, 2] = t * g * dy / chord * y_s
    f[:, 1, 3] = arc
    f[:, 1, 4] = -_BZ * t * (g * dy / chord * y_c + 0.5 * chord * chord * arc_d)
    f[:, 2, 4] = -_BZ * _DX
    q = p.clone()
    q[:, 0] += dy
    q[:, 1] += t * arc
    q[:, 2] = s2
    return q, f
