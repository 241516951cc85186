"""The following against the oracle in both of its word sizes (the 32-bit filter needs ymax <= 16383
and zmax <= 32767 LSB) at the ends of the coordinate ranges: drift length near 0 and near its
maximum, times beyond the drift range (up to the last 16-bit value), the acceptance edge, steep
slopes, with and without the skip-row rule; and in both mappings (eight lanes a task up to 2^20
clusters of a call, a thread a task beyond), on these tracks and on the edge constructions."""
import numpy as np
import pytest

import torch

from oracle import oracle as O
from paper_1712_09434_gb300 import capi
from tests._constructed import edge_events

pytestmark = pytest.mark.gpu

NS, NR = 4, 159


def _lines(rng, n, y_lo, y_hi, z_lo, z_hi, slope_z, drop, z_top):
    """Straight tracks with small scatter whose middle lies in the given range, 10 % noise around."""
    pts = []
    for k in range(NS):
        for _ in range(n):
            a = rng.integers(0, 120)
            r = np.arange(a, min(NR, a + rng.integers(15, 159)))
            sy, sz = rng.uniform(-14, 14), rng.uniform(-slope_z, slope_z)
            mid = r[len(r) // 2]
            y = rng.uniform(y_lo, y_hi) + sy * (r - mid) + rng.normal(0, 6, r.size)
            z = rng.uniform(z_lo, z_hi) + sz * (r - mid) + rng.normal(0, 6, r.size)
            keep = (np.abs(y) < 32000) & (z >= 0) & (z <= z_top) & (rng.random(r.size) >= drop)
            pts.append(np.stack([np.full(r.size, k), r, np.round(y), np.round(z)], 1)[keep])
        m = 15 * n
        pts.append(np.stack([np.full(m, k), rng.integers(0, NR, m), rng.integers(int(y_lo) - 500, int(y_hi) + 500, m),
                             np.clip(rng.integers(int(z_lo) - 500, int(z_hi) + 500, m), 0, z_top)], 1))
    p = np.unique(np.concatenate(pts).astype(np.int64), axis=0)
    off = np.searchsorted(p[:, 0] * NR + p[:, 1], np.arange(NS * NR + 1)).astype(np.int32)
    return p[:, 2].astype(np.int16), p[:, 3].astype(np.uint16), off


def _noise(rng, ns, n):
    """A second event without tracks, of n clusters spread over all rows."""
    b = rng.integers(0, ns * NR, n)
    p = np.unique(np.stack([b, rng.integers(-1300, 1300, n), rng.integers(0, 32000, n)], 1), axis=0)
    off = np.searchsorted(p[:, 0], np.arange(ns * NR + 1)).astype(np.int32)
    return p[:, 1].astype(np.int16), p[:, 2].astype(np.uint16), off


def _check(pad, tim, off, ns, geo, og, rules, many):
    """Candidates and tracks of the event against the oracle; many: with a noise event of 2^20 clusters
    behind it."""
    o = O.track_event(pad, tim, off, g=og, keep_stages=True, rules=rules)
    nc, nt = len(o["cand_n"]), len(o["trk_off"]) - 1
    assert nc > 10
    n_ev = 1
    if many:
        q = _noise(np.random.default_rng(9), ns, (1 << 20) + 40000)
        assert len(q[0]) > 1 << 20
        off = np.concatenate([off[:-1], q[2] + off[-1]]).astype(np.int32)
        pad, tim, n_ev = np.concatenate([pad, q[0]]), np.concatenate([tim, q[1]]), 2
    cl = capi.Clusters.from_numpy(pad, tim, off, n_ev)
    ctx = capi.Context(geometry=geo, max_clusters=cl.n_clusters, max_events=n_ev)
    ctx.tpc_set_rules(rules)
    tr = capi.Tracks(cl.n_clusters, n_ev, cl.n_clusters // 10 + 16, cl.n_clusters)
    ctx.tpc_track_event(cl, tr)
    assert ctx.tpc_sync_status() == 0

    def get(what, n):
        b = torch.empty(n, dtype=torch.int32, device="cuda")
        ctx.tpc_debug_copy(what, b)
        return b.cpu().numpy()

    total = int(get(2, 1)[0])
    assert total == nc or (many and total > nc)
    np.testing.assert_array_equal(get(5, nc), o["cand_n"])
    slots, rows = get(6, nc * NR).reshape(nc, NR), get(7, nc)
    for t in range(nc):
        s = slots[t, rows[t] & 0xffff:(rows[t] >> 16) + 1]
        np.testing.assert_array_equal(s[s >= 0], o["cand_hits"][t][:o["cand_n"][t]])
    g = tr.to_host()
    assert g["ev_trk_off"][1] == nt
    np.testing.assert_array_equal(g["trk_off"][:nt + 1], o["trk_off"])
    np.testing.assert_array_equal(g["trk_hits"][:o["trk_off"][-1]], o["trk_hits"])
    ctx.close()


@pytest.mark.parametrize("lsb,zmax_cm", [(1.0 / 128, 250.0), (1.0 / 256, 250.0), (1.0 / 128, 255.9)])
@pytest.mark.parametrize("rules", [0, 1])
@pytest.mark.parametrize("y,z,slope_z", [
    ((-1500, 1500), (0, 900), 12),            # start of the drift range
    ((-1500, 1500), (31000, 32767), 12),      # its end in the first geometry, and beyond
    ((-1500, 1500), (48000, 50500), 30),      # far beyond: around the last value a 32-bit filter reads
    ((-1500, 1500), (62000, 65535), 60),      # the last 16-bit times
    ((1700, 3400), (5000, 9000), 300),        # the acceptance edge, steep in z
    ((-31000, -29000), (5000, 9000), 12),     # pad coordinates far outside the acceptance
])
def test_following_words_match_the_oracle(lsb, zmax_cm, rules, y, z, slope_z):
    rng = np.random.default_rng(int(abs(y[0]) + z[0]) + rules)
    pad, tim, off = _lines(rng, 12, *y, *z, slope_z, 0.06 if rules else 0.02, 65535)
    geo = capi.tpc_geometry(NS, NR, 85.0, 247.0, 10.0, zmax_cm, lsb)
    og = O.geometry(n_sectors=NS, n_rows=NR, z_max=zmax_cm, lsb=lsb)
    _check(pad, tim, off, NS, geo, og, rules, False)
    if rules == 0:
        _check(pad, tim, off, NS, geo, og, rules, True)


@pytest.mark.parametrize("many", [False, True])
def test_edge_events_in_both_mappings(many):
    for pad, tim, off, _ in edge_events():
        _check(pad, tim, off, 36, capi.default_geometry(), O.geometry(), 0, many)
