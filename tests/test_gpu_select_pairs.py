"""Selection, merge and track output against the oracle where two blocks share a sector: 72 and 216
sectors in a call (two and six events), on row ranges of one word, of five, and beyond 160 rows; and
a launch with a grid of its own, which takes one block a sector whatever the sizes."""
import numpy as np
import pytest
import torch

from oracle import oracle as O
from paper_1712_09434_gb300 import capi, tune
from tests.test_gpu_select import _event, _oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nr,events,per_sector,shape", [
    (31, 2, 30, (0, 0, 0)), (160, 2, 25, (0, 0, 0)), (200, 2, 20, (0, 0, 0)), (64, 6, 12, (0, 0, 0)),
    (161, 6, 10, (0, 0, 0)), (200, 2, 20, (512, 0, 0)), (200, 2, 20, (1024, 1, 0))])
def test_selection_with_two_blocks_a_sector_matches_the_oracle(nr, events, per_sector, shape):
    ns = 36
    rng = np.random.default_rng(10 * nr + events)
    x_last = 85.0 + 162.0 / 158.0 * (nr - 1)
    geo = capi.tpc_geometry(ns, nr, 85.0, x_last, 10.0, 250.0, 1.0 / 128.0)
    og = O.geometry(n_sectors=ns, n_rows=nr, x_last=x_last)
    evs = [_event(rng, ns, nr, per_sector, 2 * nr) for _ in range(events)]
    n = np.cumsum([0] + [len(e[0]) for e in evs])
    off = np.concatenate([e[2][:-1] + n[i] for i, e in enumerate(evs)] + [n[-1:]]).astype(np.int32)
    cl = capi.Clusters.from_numpy(np.concatenate([e[0] for e in evs]), np.concatenate([e[1] for e in evs]), off, events)
    ctx = capi.Context(geometry=geo, max_clusters=cl.n_clusters, max_events=events)
    ctx.tpc_set_tuning(tune.to_struct({"select": shape}))
    tr = capi.Tracks(cl.n_clusters, events, cl.n_clusters // 10 + 16, cl.n_clusters)
    ctx.tpc_track_event(cl, tr)
    assert ctx.tpc_sync_status() == 0
    g = tr.to_host()
    base = 0
    for i, e in enumerate(evs):
        o_off, o_hits, o_label = _oracle(*e, og, nr)
        nt = len(o_off) - 1
        t0 = g["ev_trk_off"][i]
        assert g["ev_trk_off"][i + 1] - t0 == nt > per_sector
        np.testing.assert_array_equal(g["trk_off"][t0:t0 + nt + 1] - g["trk_off"][t0], o_off)
        np.testing.assert_array_equal(g["trk_hits"][g["trk_off"][t0]:g["trk_off"][t0 + nt]] - n[i], o_hits)
        lab = g["label"][n[i]:n[i + 1]]
        np.testing.assert_array_equal(np.where(lab >= 0, lab - base, -1), o_label)
        base += nt
    ctx.close()
    torch.cuda.synchronize()
