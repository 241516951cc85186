"""Selection, merge and track output against the oracle where one, two or four blocks share a
sector (the choice depends on the number of sectors and events), and on geometries whose row
range needs one word of kept hits, exactly five, and more than a warp's five slots a lane."""
import numpy as np
import pytest
import torch

from oracle import oracle as O
from paper_1712_09434_gb300 import capi

pytestmark = pytest.mark.gpu


def _event(rng, ns, nr, per_sector, noise):
    """Straight crossing tracks and noise in every sector, sorted in the library's layout."""
    pts = []
    for k in range(ns):
        n = per_sector
        y0, sy = rng.uniform(-1800, 1800, n), rng.uniform(-12, 12, n)
        z0, sz = rng.uniform(2000, 12000, n), rng.uniform(-20, 20, n)
        r0 = rng.integers(0, max(nr - 20, 1), n)
        for t in range(n):
            r = np.arange(r0[t], min(nr, r0[t] + rng.integers(12, nr + 1)))
            y = np.round(y0[t] + sy[t] * r + rng.normal(0, 4, r.size))
            z = np.round(z0[t] + sz[t] * r + rng.normal(0, 4, r.size))
            keep = (np.abs(y) < 1900) & (z >= 0)
            pts.append(np.stack([np.full(r.size, k), r, y, z], 1)[keep])
        m = noise
        pts.append(np.stack([np.full(m, k), rng.integers(0, nr, m), rng.integers(-1900, 1900, m),
                             rng.integers(0, 15000, m)], 1))
    p = np.unique(np.concatenate(pts).astype(np.int64), axis=0)
    off = np.searchsorted(p[:, 0] * nr + p[:, 1], np.arange(ns * nr + 1)).astype(np.int32)
    return p[:, 2].astype(np.int16), p[:, 3].astype(np.uint16), off


def _oracle(pad, tim, off, og, nr):
    """O.track_event with the geometry's number of rows."""
    up, down = O.links(pad, tim, off, og)
    up2, down2 = O.clean(up, down)
    start, length = O.chains(up2, down2)
    hits, n = O.follow(pad, tim, off, start, length, up2, og)
    seg, segn, _ = O.select(len(pad), hits, n, start, n_rows=nr)
    return O.assemble(len(pad), seg, segn, O.merge(pad, tim, off, seg, segn, og), n_rows=nr)


@pytest.mark.parametrize("ns,nr,events,per_sector", [
    (2, 200, 1, 60),      # 2 sectors: four blocks each; ranges beyond 160 rows
    (4, 161, 1, 50),      # one row past five slots a lane
    (36, 160, 1, 25),     # four blocks, exactly five words
    (36, 31, 3, 30),      # 108 sectors: two or four blocks; one word
    (36, 64, 5, 12),      # 180 sectors
    (36, 33, 12, 8),      # 432 sectors: one block from the queue
    (2, 159, 1, 0),       # no candidate at all
])
def test_selection_groups_match_the_oracle(ns, nr, events, per_sector):
    rng = np.random.default_rng(100 * ns + nr)
    x_last = 85.0 + 162.0 / 158.0 * (nr - 1)
    geo = capi.tpc_geometry(ns, nr, 85.0, x_last, 10.0, 250.0, 1.0 / 128.0)
    og = O.geometry(n_sectors=ns, n_rows=nr, x_last=x_last)
    evs = [_event(rng, ns, nr, per_sector, 20 * nr // 10) for _ in range(events)]
    n = np.cumsum([0] + [len(e[0]) for e in evs])
    off = np.concatenate([e[2][:-1] + n[i] for i, e in enumerate(evs)] + [n[-1:]]).astype(np.int32)
    cl = capi.Clusters.from_numpy(np.concatenate([e[0] for e in evs]), np.concatenate([e[1] for e in evs]), off, events)
    ctx = capi.Context(geometry=geo, max_clusters=cl.n_clusters, max_events=events)
    tr = capi.Tracks(cl.n_clusters, events, cl.n_clusters // 10 + 16, cl.n_clusters)
    ctx.tpc_track_event(cl, tr)
    assert ctx.tpc_sync_status() == 0
    g = tr.to_host()
    base = 0
    for i, e in enumerate(evs):
        o_off, o_hits, o_label = _oracle(*e, og, nr)
        nt = len(o_off) - 1
        assert g["ev_trk_off"][i + 1] - g["ev_trk_off"][i] == nt
        if per_sector:
            assert nt > per_sector
        t0 = g["ev_trk_off"][i]
        np.testing.assert_array_equal(g["trk_off"][t0:t0 + nt + 1] - g["trk_off"][t0], o_off)
        a, b = g["trk_off"][t0], g["trk_off"][t0 + nt]
        np.testing.assert_array_equal(g["trk_hits"][a:b] - n[i], o_hits)
        lab = g["label"][n[i]:n[i + 1]]
        np.testing.assert_array_equal(np.where(lab >= 0, lab - base, -1), o_label)
        base += nt
    assert base == g["n_tracks"]
    ctx.close()
    torch.cuda.synchronize()
