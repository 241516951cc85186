"""TPC-ITS matching where every track is inside the window of every ITS track, with fewer and with
more pairs than the pair list of the matching holds: all pairs have the same chi2, so both sides
choose index 0 and exactly one match remains, and a pair made better must win."""
import numpy as np
import pytest
import torch

from paper_1712_09434_gb300 import capi

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 33, 700, 6000])      # 6000^2 pairs: well over the list of ~0.65 M
def test_all_pairs_inside_the_window(n):
    n_cl = 5 * n + 10
    off = np.full(36 * 159 + 1, n_cl, np.int32)
    off[0] = 0                                           # every cluster in sector 0, row 0
    cl = capi.Clusters.from_numpy(np.zeros(n_cl, np.int16), np.zeros(n_cl, np.uint16), off, 1)
    ctx = capi.Context(max_clusters=max(n_cl, 30000), max_events=1)
    tr = capi.Tracks(n_cl, 1, n, n_cl)
    tl, q = 0.25, 0.01
    par = np.tile(np.array([0.0, 85.0 * tl, 0.0, tl, q], np.float32), (n, 1))
    cov = np.zeros((n, 15), np.float32)
    cov[:, [0, 2, 5, 9, 14]] = (1e-2, 1e-2, 1e-4, 1e-4, 1e-3)
    f = lambda a: torch.from_numpy(a).cuda()
    tr.par[:] = f(par).view(-1)
    tr.cov[:] = f(cov).view(-1)
    tr.xref.fill_(85.0)
    tr.ndf.fill_(100)
    tr.trk_off[:] = torch.arange(n + 1, dtype=torch.int32, device="cuda")
    tr.trk_hits[:n] = torch.arange(n, dtype=torch.int32, device="cuda")
    tr.n_tracks.fill_(n)
    its = np.zeros((n, 8), np.float32)
    its[:] = (np.deg2rad(10.0), 0.0, tl + 0.001, q, 1e-3, 0.01, 1e-3, 1e-3)
    mt = torch.empty(n, dtype=torch.int32, device="cuda")
    mi = torch.empty(n, dtype=torch.int32, device="cuda")
    anchor = torch.empty((n, 8), dtype=torch.float32, device="cuda")
    ctx.tpc_its_match(cl, tr, f(its), mt, mi, anchor)
    assert ctx.tpc_sync_status() == 0
    want = np.full(n, -1)
    want[0] = 0
    np.testing.assert_array_equal(mt.cpu().numpy(), want)
    np.testing.assert_array_equal(mi.cpu().numpy(), want)
    its[n - 1, 2] = tl                                   # the last ITS track fits better: all tracks
    ctx.tpc_its_match(cl, tr, f(its), mt, mi, anchor)    # choose it, and it chooses track 0
    assert ctx.tpc_sync_status() == 0
    m = mt.cpu().numpy()
    assert m[0] == n - 1 and np.all(m[1:] == -1)
    assert mi.cpu().numpy()[n - 1] == 0
    ctx.close()
