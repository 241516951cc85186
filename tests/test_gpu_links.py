"""Neighbour links against the oracle where a bin is shared by 1, 2 and 16 warps, at the ends of the
coordinate ranges, and with windows that hold more candidates than the kernel's list."""
import numpy as np
import pytest
import torch

from oracle import oracle as O
from paper_1712_09434_gb300 import capi

pytestmark = pytest.mark.gpu

NS, NR = 2, 6


def _rows(rng, per_bin, y_lo, y_hi, z_lo, z_hi):
    pts = []
    for b in range(NS * NR):
        n = int(per_bin * rng.uniform(0.3, 1.7))
        pts.append(np.stack([np.full(n, b), rng.integers(y_lo, y_hi + 1, n), rng.integers(z_lo, z_hi + 1, n)], 1))
    p = np.unique(np.concatenate(pts).astype(np.int64), axis=0)
    off = np.searchsorted(p[:, 0], np.arange(NS * NR + 1)).astype(np.int32)
    return p[:, 1].astype(np.int16), p[:, 2].astype(np.uint16), off


@pytest.mark.parametrize("rules", [0, 1])
@pytest.mark.parametrize("per_bin,y,z", [
    (5, (-400, 400), (0, 900)),               # nearly empty rows: one warp a bin, skipped rows
    (33, (-800, 800), (0, 2000)),             # one warp, a second group of one cluster
    (70, (-32768, -31000), (63000, 65535)),   # two warps; the last 16-bit times, the lowest pads
    (70, (31000, 32767), (0, 1500)),          # the highest pads, times from 0
    (70, (-300, 300), (31900, 32600)),        # across the last slab boundary
    (300, (-500, 500), (5000, 6000)),         # windows of well over a list of 12 candidates
    (1500, (-4000, 4000), (0, 32000)),        # 16 warps a bin (the most)
])
def test_links_match_the_oracle(rules, per_bin, y, z):
    rng = np.random.default_rng(per_bin + abs(y[0]))
    pad, tim, off = _rows(rng, per_bin, *y, *z)
    geo = capi.tpc_geometry(NS, NR, 85.0, 90.0, 10.0, 250.0, 1.0 / 128.0)
    up, down = O.links(pad, tim, off, O.geometry(n_sectors=NS, n_rows=NR, x_last=90.0), rules)
    cl = capi.Clusters.from_numpy(pad, tim, off, 1)
    n = cl.n_clusters
    ctx = capi.Context(geometry=geo, max_clusters=n, max_events=1)
    ctx.tpc_set_rules(rules)
    tr = capi.Tracks(n, 1, n + 16, n + 16)
    ctx.tpc_track_event(cl, tr)
    assert ctx.tpc_sync_status() == 0
    got = [torch.empty(n, dtype=torch.int32, device="cuda") for _ in range(2)]
    ctx.tpc_debug_copy(0, got[0])
    ctx.tpc_debug_copy(1, got[1])
    np.testing.assert_array_equal(got[0].cpu().numpy(), up)
    np.testing.assert_array_equal(got[1].cpu().numpy(), down)
    assert (up >= 0).sum() > 0 or per_bin < 10
    if rules == 0:
        status = torch.empty(1, dtype=torch.int32, device="cuda")
        assert capi.tpc_links_noalloc(geo, cl, got[0], got[1], status) == 0
        np.testing.assert_array_equal(got[0].cpu().numpy(), up)
        np.testing.assert_array_equal(got[1].cpu().numpy(), down)
        assert int(status.item()) == 0
    ctx.close()
