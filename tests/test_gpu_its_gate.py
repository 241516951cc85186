"""TPC-ITS matching with errors far smaller than a fit gives (the caller's variances have no lower
bound): candidate pairs on both sides of the chi2 gate, one ITS track a window, against the oracle.  A
pair may only be left out by the FP64 chi2, however small its errors are against FP32 rounding."""
import numpy as np
import pytest
import torch

from oracle import oracle as O
from paper_1712_09434_gb300 import capi

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sigma", [1e-7, 1e-6, 1e-5, 1e-4])
def test_pairs_near_the_gate_with_small_errors(sigma):
    rng = np.random.default_rng(int(-np.log10(sigma)))
    # windows apart in azimuth (0.1 rad), tan lambda (0.1) and z (2 cm)
    sn, tl, z = np.meshgrid(np.sin(np.arange(-0.5, 0.51, 0.25)), np.arange(-0.9, 0.91, 0.3), np.arange(-240, 241, 8.0),
                            indexing="ij")
    n = sn.size
    sn, tl, z = (a.ravel() for a in (sn, tl, z))
    par = np.stack([85.0 * sn / np.sqrt(1 - sn * sn), z, sn, tl, rng.uniform(-1.0, 1.0, n)], 1).astype(np.float32)
    par[:, 4] = np.where(np.abs(par[:, 4]) < 0.2, 0.2, par[:, 4])
    at_vertex = lambda: np.array([O.propagate(85.0, p.astype(np.float64), 0.0)[1] for p in par])
    v = at_vertex()
    par[:, 0] -= v[:, 0]
    par[:, 1] -= v[:, 1] - z
    v = at_vertex()
    assert np.all(np.abs(v[:, 0]) < 1e-3) and np.all(np.abs(v[:, 1] - z) < 0.1)
    cov = np.zeros((n, 15), np.float32)
    cov[:, 0] = cov[:, 2] = 1e-2
    # 9.5 to 10.5 errors apart in sin phi, tan lambda or q/pT (gate: 10)
    d = rng.uniform(9.5, 10.5, n) * rng.choice([-1.0, 1.0], n)
    which = rng.integers(0, 3, n)
    phi = np.deg2rad(10.0) + np.arcsin(v[:, 2])
    its = np.stack([phi + sigma * d * (which == 0), v[:, 1], v[:, 3] + sigma * d * (which == 1),
                    v[:, 4] * (1 + sigma * d * (which == 2)), np.full(n, sigma), np.full(n, 0.01), np.full(n, sigma),
                    sigma * np.abs(v[:, 4])], 1).astype(np.float32)
    fit = dict(par=par.astype(np.float64), cov=cov.astype(np.float64), xref=np.full(n, 85.0), ndf=np.full(n, 100))
    want_t, want_i, _ = O.its_match(fit, np.zeros(n, np.int32), its.astype(np.float64))
    if sigma > 1e-7:                     # (below, the FP32 inputs themselves are further apart than the errors)
        assert 0.2 * n < (want_t >= 0).sum() < 0.8 * n
    n_cl = 5 * n + 10
    off = np.full(36 * 159 + 1, n_cl, np.int32)
    off[0] = 0                           # every cluster in sector 0, row 0
    cl = capi.Clusters.from_numpy(np.zeros(n_cl, np.int16), np.zeros(n_cl, np.uint16), off, 1)
    ctx = capi.Context(max_clusters=max(n_cl, 30000), max_events=1)
    tr = capi.Tracks(n_cl, 1, n, n_cl)
    f = lambda a: torch.from_numpy(a).cuda()
    tr.par[:] = f(par).view(-1)
    tr.cov[:] = f(cov).view(-1)
    tr.xref.fill_(85.0)
    tr.ndf.fill_(100)
    tr.trk_off[:] = torch.arange(n + 1, dtype=torch.int32, device="cuda")
    tr.trk_hits[:n] = torch.arange(n, dtype=torch.int32, device="cuda")
    tr.n_tracks.fill_(n)
    mt = torch.empty(n, dtype=torch.int32, device="cuda")
    mi = torch.empty(n, dtype=torch.int32, device="cuda")
    ctx.tpc_its_match(cl, tr, f(its), mt, mi)
    assert ctx.tpc_sync_status() == 0
    np.testing.assert_array_equal(mt.cpu().numpy(), want_t)
    np.testing.assert_array_equal(mi.cpu().numpy(), want_i)
    ctx.close()
