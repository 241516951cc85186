"""Calls on a stream that does not wait for the default stream (torch's pool gives non-blocking
streams), while the default stream still has work queued: a context that was made or grown just before
must give the same results as an idle one.  The device memory that the workspace is taken from is
filled beforehand, so that nothing starts at zero by chance."""
import numpy as np
import pytest
import torch

from paper_1712_09434_gb300 import capi, synth
from tests import _gpu

pytestmark = pytest.mark.gpu


def _queue_work(ms=40):
    """Some tens of milliseconds of copies on the default stream."""
    x = torch.ones(1 << 28, device="cuda")
    for _ in range(4 * ms):
        x.mul_(1.0)
    return x


def _fill_free_memory(n_bytes):
    x = torch.full((n_bytes,), 0x5b, dtype=torch.uint8, device="cuda")
    torch.cuda.synchronize()
    del x
    torch.cuda.empty_cache()


def _outputs(ev):
    return (capi.Tracks(ev.n_clusters, 1, ev.n_clusters // 10 + 16, ev.n_clusters),
            torch.zeros(1, dtype=torch.float64, device="cuda"), torch.zeros(73, dtype=torch.float64, device="cuda"))


def _step(ctx, cl, out, th, stream=None):
    tr, s, g = out
    ctx.tpc_track_event(cl, tr, stream=stream)
    ctx.tpc_refit_grad(cl, tr, th, s, g, stream=stream)


@pytest.mark.parametrize("grown", [False, True])
def test_first_call_of_a_workspace_on_a_stream_that_does_not_wait(grown):
    ev = synth.make_event(synth.full_event(seed=31, n_tracks=300))
    cl = _gpu.clusters_of(ev)
    th = torch.tensor(synth.theta_nominal(), device="cuda")
    ref, got = _outputs(ev), _outputs(ev)
    ctx = _gpu.make_context(ev.n_clusters, 1)
    _step(ctx, cl, ref, th)
    assert ctx.tpc_sync_status() == 0
    ctx.close()
    _fill_free_memory(2 << 30)
    ctx = _gpu.make_context(1000, 1) if grown else capi.Context()
    side = torch.cuda.Stream()
    torch.cuda.synchronize()
    busy = _queue_work()
    ctx.reserve(ev.n_clusters, 1)
    for _ in range(2):
        _step(ctx, cl, got, th, stream=side)
    assert ctx.tpc_sync_status(stream=side) == 0
    torch.cuda.synchronize()
    a, b = ref[0].to_host(), got[0].to_host()
    assert a["n_tracks"] == b["n_tracks"] > 250
    for k in ("trk_off", "trk_hits", "label", "par", "cov", "chi2", "ndf"):
        np.testing.assert_array_equal(a[k], b[k], err_msg=k)
    assert ref[1].item() == got[1].item()
    np.testing.assert_array_equal(ref[2].cpu().numpy(), got[2].cpu().numpy())
    ctx.close()
    del busy


def test_an_error_on_a_stream_that_does_not_wait_is_not_lost():
    ev = synth.make_event(synth.full_event(seed=31, n_tracks=300))
    off = ev.bin_off.copy()
    off[-1] -= 1                       # the offsets do not end at the number of clusters
    cl = capi.Clusters.from_numpy(ev.pad_fp, ev.time_fp, off, 1)
    tr = _outputs(ev)[0]
    warm = _gpu.make_context(ev.n_clusters, 1)         # kernels loaded: loading them waits for the device
    warm.tpc_track_event(_gpu.clusters_of(ev), tr)
    assert warm.tpc_sync_status() == 0
    ctx = capi.Context()
    side = torch.cuda.Stream()
    torch.cuda.synchronize()
    busy = _queue_work()
    ctx.reserve(ev.n_clusters, 1)
    ctx.tpc_track_event(cl, tr, stream=side)
    assert ctx.tpc_sync_status(stream=side) == capi.TPC_ERR_BOUNDS
    assert ctx.tpc_sync_status(stream=side) == capi.TPC_OK       # read and cleared
    torch.cuda.synchronize()
    ctx.close()
    del busy
