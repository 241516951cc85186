"""Gradient of many tracks too long for the length order (511 hits and more, which keep checkpoints):
the per-track records must not depend on how many there are, whether they are spread over the warps,
taken by block index, or handed out by the queue (here: few small blocks)."""
import numpy as np
import pytest
import torch

from paper_1712_09434_gb300 import capi, tune
from tests.test_gpu_refit_forms import REC, _refit, _theta, _tracks

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,shape", [(33, (0, 0, 0)), (609, (0, 0, 0)), (1300, (0, 0, 0)), (4865, (0, 0, 0)),
                                     (9729, (0, 0, 0)), (9729, (64, 1, 0)), (1300, (32, 1, 1))])
def test_records_of_long_tracks_do_not_depend_on_their_number(n, shape):
    ev, tracks = _tracks()
    few = [np.repeat(t, -(-511 // len(t)))[:511 + 16 * i] for i, t in enumerate(sorted(tracks, key=len)[-5:])]
    assert min(len(t) for t in few) >= 511
    th = _theta()
    base = _refit(ev, few, th, True)[2]
    tracks = [few[i % 5] for i in range(n)]
    hits = np.concatenate(tracks).astype(np.int32)
    off = np.cumsum([0] + [len(t) for t in tracks]).astype(np.int32)
    cl = capi.Clusters.from_numpy(ev.pad_fp, ev.time_fp, ev.bin_off, 1)
    ctx = capi.Context(max_clusters=len(hits), max_events=1)
    ctx.tpc_set_tuning(tune.to_struct({"refit_grad": shape}))
    tr = capi.Tracks(cl.n_clusters, 1, n, len(hits))
    tr.trk_off[:] = torch.from_numpy(off).cuda()
    tr.trk_hits[:] = torch.from_numpy(hits).cuda()
    tr.n_tracks.fill_(n)
    s = torch.zeros(1, dtype=torch.float64, device="cuda")
    g = torch.zeros(73, dtype=torch.float64, device="cuda")
    ctx.tpc_refit_grad(cl, tr, torch.tensor(th, device="cuda"), s, g, None, None, 1)
    assert ctx.tpc_sync_status() == 0
    rec = torch.empty(n * REC, dtype=torch.int32, device="cuda")
    ctx.tpc_debug_copy(11, rec)
    np.testing.assert_array_equal(rec.cpu().numpy().reshape(n, REC), base[np.arange(n) % 5])
    ctx.close()
