"""The two ways the gradient keeps its forward states, and the two register splits of its reverse
pass: tracks of LEN_BUCKETS - 1 = 511 hits and more (here: outgoing tracks whose clusters are listed
several times) keep checkpoints with every track of their 32, all others store every step; a call
with more than 128 x 128 x 3 clusters a multiprocessor takes the other register split.  The per-track
records must not depend on either, and the gradient of the long tracks must match FP64 central
differences."""
import numpy as np
import pytest
import torch

from paper_1712_09434_gb300 import capi, synth
from tests import _gpu

pytestmark = pytest.mark.gpu

REC = 26


def _tracks(n_tracks=60, seed=21):
    ev = synth.make_event(synth.full_event(seed=seed, n_tracks=n_tracks))
    ctx = _gpu.make_context(ev.n_clusters, 1)
    g = _gpu.run(ctx, _gpu.clusters_of(ev))
    ctx.close()
    hits = [g["trk_hits"][a:b] for a, b in zip(g["trk_off"][:-1], g["trk_off"][1:])]
    return ev, [h for i, h in enumerate(hits) if g["chi2"][i] < 4 * max(int(g["ndf"][i]), 1) and len(h) > 40]


def _refit(ev, tracks, theta, raw, pad_clusters=0):
    """Sum of chi2, gradient and per-track records; pad_clusters more clusters in the last bin."""
    off = ev.bin_off.astype(np.int64).copy()
    off[-1] += pad_clusters
    z = np.zeros(pad_clusters, np.int16)
    cl = capi.Clusters.from_numpy(np.concatenate([ev.pad_fp, z]), np.concatenate([ev.time_fp, z.view(np.uint16)]), off, 1)
    nt, nh = len(tracks), sum(len(t) for t in tracks)
    ctx = capi.Context(max_clusters=max(cl.n_clusters, nh, 10 * nt), max_events=1)
    tr = capi.Tracks(cl.n_clusters, 1, nt, nh)
    to = np.cumsum([0] + [len(t) for t in tracks]).astype(np.int32)
    tr.trk_off[:] = torch.from_numpy(to).cuda()
    tr.trk_hits[:] = torch.from_numpy(np.concatenate(tracks).astype(np.int32)).cuda()
    tr.n_tracks.fill_(nt)
    s = torch.zeros(1, dtype=torch.float64, device="cuda")
    g = torch.zeros(73, dtype=torch.float64, device="cuda")
    ctx.tpc_refit_grad(cl, tr, torch.tensor(theta, device="cuda"), s, g, None, None, int(raw))
    assert ctx.tpc_sync_status() == 0
    rec = torch.empty(nt * REC, dtype=torch.int32, device="cuda")
    ctx.tpc_debug_copy(11, rec)
    out = float(s.item()), g.cpu().numpy(), rec.cpu().numpy().reshape(nt, REC)
    ctx.close()
    return (*out, to)


def _theta():
    th = synth.theta_nominal()
    rng = np.random.default_rng(4)
    th[0] += 2.0 ** -11
    th[1:37] += rng.normal(0, 0.02, 36)
    return th


@pytest.mark.parametrize("raw", [False, True])
def test_records_do_not_depend_on_how_states_are_kept(raw):
    ev, tracks = _tracks()
    assert len(tracks) > 35
    th = _theta()
    base = _refit(ev, tracks, th, raw)[2]
    # two long tracks: the first 32 of the length order keep checkpoints, the rest stores states
    a, b = sorted(tracks, key=len)[-2:]
    long_ = [np.repeat(a, 5)[:511], np.repeat(b, 6)]
    assert len(long_[0]) == 511 and len(long_[1]) > 511
    mixed = _refit(ev, long_ + tracks, th, raw)[2]
    np.testing.assert_array_equal(mixed[2:], base)
    # 510 hits: the longest class whose states are stored
    short = _refit(ev, [np.repeat(a, 5)[:510]] + tracks, th, raw)[2]
    np.testing.assert_array_equal(short[1:], base)
    # the other register split of the reverse pass
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    many = _refit(ev, tracks, th, raw, pad_clusters=128 * 128 * 3 * sms + 128)[2]
    np.testing.assert_array_equal(many, base)



@pytest.mark.parametrize("n", [608, 609, 1300, 4864, 9729, 155649])
def test_records_do_not_depend_on_the_spread_over_warps(n):
    # 152 x 128 threads are spread: 32 threads a track up to 608 tracks, one from 9,729 on; more
    # tracks than threads are taken from the queue
    ev, tracks = _tracks()
    tracks = [t[-20:] for t in tracks]
    th = _theta()
    base = _refit(ev, tracks, th, True)[2]
    many = _refit(ev, [tracks[i % len(tracks)] for i in range(n)], th, True)[2]
    np.testing.assert_array_equal(many, base[np.arange(n) % len(tracks)])
