"""Performance cases: the calls a user of the library makes, over the sizes they are made at.

Every case names one call (`call`) and the shape of its input; `prepare` makes the input on the GPU
from the seed, `run` makes the call once through the binding (paper_1712_09434_gb300.capi), `work`
counts the bytes and operations the call cannot do without, and `exact` gives the result in 64 bits
where a plain calculation can.

Inputs are simulated events like those of paper_1712_09434_gb300.synth (charged helices from the
origin in a 0.5 T field, one smeared cluster per pad row crossed, uniform noise, fixed-point
quantisation), made with torch on the device so that a 64-event batch takes a moment instead of
half a minute.
"""
from __future__ import annotations

import math
from types import SimpleNamespace

import numpy as np
import torch

from paper_1712_09434_gb300 import capi, synth

NB = synth.N_SECTORS * synth.N_ROWS
HITS_PER_TRACK = 155.0          # mean clusters of a generated track (measured on the central event)
DEAD_ROWS = ((60, 61), (100, 111))


def listed():
    return [
        # One sector of an online readout chain, or a test beam: the smallest call, launch latency.
        {"name": "event-sector", "call": "event", "tracks": 200, "noise": 0.10, "loopers": 0.0, "sector": True,
         "rules": 0, "dead": False},
        # An ordinary whole event, tracked on its own as it arrives.
        {"name": "event-full", "call": "event", "tracks": 5000, "noise": 0.15, "loopers": 0.0, "sector": False,
         "rules": 0, "dead": False},
        # A central Pb-Pb event: low-pT loopers, much noise.
        {"name": "event-central", "call": "event", "tracks": 20000, "noise": 0.30, "loopers": 0.10, "sector": False,
         "rules": 0, "dead": False},
        # The same multiplicity on a detector with dead pad rows and 5 % lost clusters, with the
        # rules for missing clusters switched on.
        {"name": "event-inefficient", "call": "event", "tracks": 20000, "noise": 0.30, "loopers": 0.10,
         "sector": False, "rules": 3, "dead": True},
        # A small batch of uneven events (a time bin of the online farm), tracking only.
        {"name": "batch-12", "call": "batch", "events": 12, "low": 100, "high": 4000, "noise": 0.20, "loopers": 0.10},
        # The throughput workload: 64 events of 100 to 20,000 tracks, tracking, refit and adjoint in
        # one graph launch.
        {"name": "step-64", "call": "step", "events": 64, "low": 100, "high": 20000, "noise": 0.20, "loopers": 0.10},
        # One gradient of the calibration loop on a central event: raw errors, references at the vertex.
        {"name": "grad-central", "call": "refit", "tracks": 20000, "noise": 0.30, "anchors": True, "raw": True,
         "backward": True},
        # The objective alone (a line search, a quality figure) on an ordinary event, fixed errors.
        {"name": "objective-full", "call": "refit", "tracks": 5000, "noise": 0.15, "anchors": False, "raw": False,
         "backward": False},
        # TPC-ITS matching of a central event for the drift calibration.
        {"name": "its-central", "call": "its", "tracks": 20000, "noise": 0.30, "loopers": 0.10},
        # Looper-leg pairing of a looper-rich event.
        {"name": "loopers-rich", "call": "loopers", "tracks": 3000, "noise": 0.10, "loopers": 0.30},
        # Continuous readout: collisions at 5 per drift length, cut into slices, tracked and joined.
        {"name": "frame-24", "call": "frame", "events": 24, "low": 100, "high": 8000, "noise": 0.20, "loopers": 0.10,
         "slice_len": 32000},
        # Neighbour links without a context or workspace (callers that cannot allocate).
        {"name": "links-full", "call": "links", "tracks": 5000, "noise": 0.15, "loopers": 0.0},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the same ranges, sizes spread over their logarithm."""
    call = rng.choice(["event", "event", "event", "batch", "batch", "step", "refit", "refit", "refit", "its", "loopers",
                       "frame", "links"])
    noise = round(rng.uniform(0.02, 0.35), 3)
    loopers = round(rng.choice([0.0, rng.uniform(0.02, 0.30)]), 3)
    if call == "event":
        sector = rng.random() < 0.25
        dead = rng.random() < 0.3
        return {"call": call, "tracks": _log_int(rng, 30, 700 if sector else 20000), "noise": noise,
                "loopers": loopers, "sector": sector, "rules": rng.choice([1, 2, 3]) if dead else 0, "dead": dead}
    if call == "batch" or call == "step":
        low = _log_int(rng, 50, 300)
        return {"call": call, "events": _log_int(rng, 2, 60), "low": low, "high": _log_int(rng, 2 * low, 18000),
                "noise": min(noise, 0.2), "loopers": min(loopers, 0.1)}
    if call == "refit":
        return {"call": call, "tracks": _log_int(rng, 30, 20000), "noise": noise, "anchors": rng.random() < 0.5,
                "raw": rng.random() < 0.5, "backward": rng.random() < 0.7}
    if call == "its":
        return {"call": call, "tracks": _log_int(rng, 100, 20000), "noise": noise, "loopers": loopers}
    if call == "loopers":
        return {"call": call, "tracks": _log_int(rng, 300, 20000), "noise": noise,
                "loopers": round(rng.uniform(0.05, 0.35), 3)}
    if call == "frame":
        low = _log_int(rng, 50, 200)
        return {"call": call, "events": _log_int(rng, 2, 28), "low": low, "high": _log_int(rng, 2 * low, 8000),
                "noise": min(noise, 0.2), "loopers": min(loopers, 0.1), "slice_len": rng.randint(8000, 32000)}
    return {"call": call, "tracks": _log_int(rng, 30, 5000), "noise": min(noise, 0.15), "loopers": 0.0}


# ---- the simulated input ----------------------------------------------------------------------

def _multiplicities(case):
    """Track counts of a batch, log-uniform between low and high (the quantiles, so that the total
    does not depend on the seed)."""
    n = case["events"]
    u = (np.arange(n) + 0.5) / n
    return np.floor(np.exp(math.log(case["low"]) + u * math.log(case["high"] / case["low"]))).astype(np.int64)


def _particles(rng, mult, looper_frac, single_sector):
    """Kinematics of all particles of the events (numpy; a few hundred thousand numbers)."""
    ev = np.repeat(np.arange(len(mult)), mult)
    n = ev.size
    loop = np.concatenate([np.arange(m) >= m - int(round(looper_frac * m)) for m in mult])
    pt = np.where(loop, rng.uniform(0.05, 0.15, n), 0.1 + rng.exponential(0.6, n))
    eta = rng.uniform(-0.9, 0.9, n)
    if single_sector:
        eta = np.abs(eta)
    phi0 = rng.uniform(0.0, math.radians(2 * synth.HALF_ANGLE_DEG) if single_sector else 2 * math.pi, n)
    q = rng.choice(np.array([-1.0, 1.0]), n)
    return SimpleNamespace(ev=ev, trk_pt=pt, trk_eta=eta, trk_phi0=phi0, trk_q=q)


def _signals(p, dev, gen, single_sector, theta):
    """Smeared clusters of all particles: (particle, sector, row, y, drift, path length, sin phi)."""
    f = lambda a: torch.as_tensor(a, device=dev, dtype=torch.float64)
    phi0, C, tl = f(p.trk_phi0), f(synth.KB * p.trk_q / p.trk_pt), torch.sinh(f(p.trk_eta))
    aC = C.abs()
    turn = 2 * math.pi / aC
    v_out, v_in = synth.R_OUT * aC / 2, synth.X_FIRST * aC / 2
    s_exit = torch.where(v_out < 1, 2 * torch.asin(v_out.clamp(max=1.0)) / aC, turn)
    s_end = torch.minimum(torch.minimum(s_exit, synth.Z_MAX / tl.abs().clamp(min=1e-300)), turn)
    s_in = torch.where(v_in < 1, 2 * torch.asin(v_in.clamp(max=1.0)) / aC, torch.zeros_like(aC))
    s_last = torch.minimum(s_end, turn - s_in)
    w = math.radians(2 * synth.HALF_ANGLE_DEG)
    pa, pb = phi0 + C * s_in / 2, phi0 + C * s_last / 2     # position angles: they fix the sectors
    j_lo = torch.floor(torch.minimum(pa, pb) / w) - 1
    span = (torch.floor(torch.maximum(pa, pb) / w) + 2 - j_lo).clamp(max=18)
    live = (v_in < 1) & (s_last > s_in)
    j = torch.arange(18, device=dev)
    pair = (live[:, None] & (j[None, :] < span[:, None])).nonzero()
    trk = pair[:, 0]
    ks = torch.remainder(j_lo[trk] + pair[:, 1], 18).long()
    if single_sector:
        trk, ks = trk[ks == 0], ks[ks == 0]
    sec = ks + torch.where(tl[trk] >= 0, 0, 18)
    row_x = f(synth.ROW_X)
    th = None if theta is None else f(theta)
    got = []
    for c0 in range(0, trk.numel(), 65536):
        t, k = trk[c0:c0 + 65536], sec[c0:c0 + 65536]
        al = ((k % 18).double() + 0.5) * w
        Ct, a0 = C[t][:, None], (phi0[t] - al)[:, None]
        v = torch.sin(a0) + Ct * row_x[None, :]
        inside = v.abs() <= 1.0
        b = torch.asin(v.clamp(-1.0, 1.0))
        for branch in (0, 1):
            d = torch.remainder((b if branch == 0 else math.pi - b) - a0, 2 * math.pi)
            s = torch.where(Ct < 0, d - 2 * math.pi, d) / Ct
            hit = (inside & (s > 0) & (s < s_end[t][:, None])).nonzero()
            pi, ri = hit[:, 0], hit[:, 1]
            got.append((t[pi], k[pi], ri, s[pi, ri]))
        del v, b, d, s, inside
    t, k, r, s = (torch.cat([g[i] for g in got]) for i in range(4))
    ph, Ct, al, xr = phi0[t], C[t], ((k % 18).double() + 0.5) * w, row_x[r]

    def local(s):
        psi = ph + Ct * s - al
        return (torch.sin(psi) - torch.sin(ph - al)) / Ct, (torch.cos(ph - al) - torch.cos(psi)) / Ct, psi

    if th is not None:     # the pad row collects the charge whose raw position lies on its plane
        ak = th[37 + k]
        for _ in range(6):
            xl, yl, psi = local(s)
            rho = torch.hypot(xl, yl)
            raw = xl * (rho + 85.0 * ak / 162.0) / (1.0 + ak / 162.0) / rho
            cp = torch.cos(psi)
            s = s - ((raw - xr) / torch.where(cp.abs() > 1e-3, cp, torch.full_like(cp, 1e-3))).clamp(-1.0, 1.0)
    xl, yl, psi = local(s)
    z = s * tl[t]
    side = torch.where(k < 18, 1.0, -1.0).double()
    y = yl
    drift = synth.Z_MAX - side * z
    if th is not None:
        rho = torch.hypot(xl, yl)
        y = yl * (rho + 85.0 * ak / 162.0) / (1.0 + ak / 162.0) / rho
        drift = (synth.Z_MAX - side * (z - th[1 + k])) / th[0]
    keep = (y.abs() <= xr * synth.TAN_HALF) & (z.abs() <= synth.Z_MAX) & torch.where(side > 0, z >= 0, z < 0)
    keep &= (xl - xr).abs() < 2.0
    y = y + 0.1 * torch.randn(y.shape, generator=gen, device=dev, dtype=torch.float64)
    drift = drift + 0.1 * torch.randn(y.shape, generator=gen, device=dev, dtype=torch.float64)
    keep &= (drift >= 0.0) & (drift <= synth.Z_MAX)
    snp = torch.sin(psi)
    return [a[keep] for a in (t, k, r, y, drift, s, snp)]


def _quantise(y, drift):
    half_away = lambda v: torch.sign(v) * torch.floor(v.abs() + 0.5)
    pad = half_away(y / synth.LSB).long()
    tim = half_away(drift / synth.LSB).long().clamp(0, synth.Z_MAX_LSB)
    return pad, tim


def _clusters(case, seed, mult, dev, single_sector=False, dead=False, theta=None, frame=None):
    """Clusters of the events in the library's layout, and what generated them."""
    rng = np.random.default_rng(seed)
    gen = torch.Generator(device=dev)
    gen.manual_seed(seed)
    p = _particles(rng, mult, case.get("loopers", 0.0), single_sector)
    t, k, r, y, d, s, snp = _signals(p, dev, gen, single_sector, theta)
    ev_of = torch.as_tensor(p.ev, device=dev)
    uni = lambda n: torch.rand(n, generator=gen, device=dev, dtype=torch.float64)
    if dead:
        alive = uni(t.numel()) >= 0.05
        for r0, r1 in DEAD_ROWS:
            alive &= (r < r0) | (r > r1)
        t, k, r, y, d, s, snp = (a[alive] for a in (t, k, r, y, d, s, snp))
    ev = ev_of[t]
    n_noise = (torch.bincount(ev, minlength=len(mult)) * case["noise"]).round().long()
    nev = torch.repeat_interleave(torch.arange(len(mult), device=dev), n_noise)
    nn = nev.numel()
    nk = torch.zeros(nn, dtype=torch.long, device=dev) if single_sector else (uni(nn) * synth.N_SECTORS).long()
    nr = (uni(nn) * synth.N_ROWS).long()
    if dead:
        for r0, r1 in DEAD_ROWS:
            nr = torch.where((nr >= r0) & (nr <= r1), nr - 20, nr)
    row_x = torch.as_tensor(synth.ROW_X, device=dev)
    ny = (2 * uni(nn) - 1) * row_x[nr] * synth.TAN_HALF
    nd = uni(nn) * synth.Z_MAX
    pad, tim = _quantise(torch.cat([y, ny]), torch.cat([d, nd]))
    ev, k, r = torch.cat([ev, nev]), torch.cat([k, nk]), torch.cat([r, nr])
    mc = torch.cat([t, torch.full_like(nev, -1)])
    fill = torch.zeros(nn, dtype=torch.float64, device=dev)
    s, snp = torch.cat([s, fill]), torch.cat([snp, fill])
    n_ev = len(mult)
    if frame is not None:       # collisions at Poisson times, 5 per drift length, cut into slices
        gaps = rng.exponential(synth.DRIFT_LSB / 5.0, n_ev)
        gaps[0] = 0.0
        t0 = torch.as_tensor(np.floor(np.cumsum(gaps)).astype(np.int64), device=dev)
        tau = tim + t0[ev]
        ev = tau // frame
        tim = tau - ev * frame
        n_ev = int(ev.max()) + 1
    b = (ev * synth.N_SECTORS + k) * synth.N_ROWS + r
    key, o = torch.sort((b << 32) | ((pad + 32768) << 16) | tim, stable=True)
    off = torch.searchsorted(key >> 32, torch.arange(n_ev * NB + 1, device=dev)).to(torch.int32)
    u16 = torch.where(tim >= 32768, tim - 65536, tim)
    cl = capi.Clusters(pad[o].to(torch.int16), u16[o].to(torch.int16), off, n_ev)
    return cl, SimpleNamespace(p=p, mc=mc[o], s=s[o], snp=snp[o], sector=k[o], row=r[o], bins=b[o])


def _theta(rng):
    th = np.empty(73)
    th[0] = 1.0 + 0.003 * rng.uniform(-1.0, 1.0)
    th[1:37] = rng.normal(0.0, 0.05, 36)
    th[37:73] = rng.normal(0.0, 0.1, 36)
    return th


def _given_tracks(truth, dev):
    """Hit lists of the generated particles as a tracking call would return them: the outgoing leg
    up to the slope where the following stops, hits in path order, at least 10 of them, tracks in
    the order of their first hit."""
    Cabs = np.abs(synth.KB / truth.p.trk_pt)
    half_turn = torch.as_tensor(math.pi / Cabs, device=dev)
    use = ((truth.mc >= 0) & (truth.snp.abs() < 0.92)).nonzero()[:, 0]
    use = use[truth.s[use] < half_turn[truth.mc[use]]]
    use = use[torch.argsort(truth.s[use], stable=True)]
    use = use[torch.argsort(truth.mc[use], stable=True)]
    trk = truth.mc[use]
    n = torch.bincount(trk, minlength=len(Cabs))
    use = use[n[trk] >= 10]
    trk, n = torch.unique_consecutive(truth.mc[use], return_counts=True)
    start = torch.cumsum(n, 0) - n
    o = torch.argsort(use[start])
    trk, n, start = trk[o], n[o], start[o]
    off = torch.cat([torch.zeros(1, dtype=torch.long, device=dev), torch.cumsum(n, 0)])
    hits = use[torch.repeat_interleave(start - off[:-1], n) + torch.arange(int(off[-1]), device=dev)]
    return off, hits, trk


def _references(truth, off, hits, trk, rng, dev):
    """Reference measurements at the vertex of the tracks an inner tracker would match: first hit
    within the first 8 rows, 30 hits or more, well inside the local parametrisation."""
    p = truth.p
    j = trk.cpu().numpy()
    n = np.diff(off.cpu().numpy())
    first = hits[off[:-1]]
    row, sec = truth.row[first].cpu().numpy(), truth.sector[first].cpu().numpy()
    snp = np.sin(p.trk_phi0[j] - synth.sector_alpha(sec))
    ok = (row <= 8) & (n >= 30) & (np.abs(snp) < 0.9)
    g = rng.normal(0.0, 1.0, (j.size, 3))
    q = p.trk_q[j] / p.trk_pt[j]
    sq = synth.REF_SIGMA_QPT_REL * np.abs(q)
    a = np.stack([np.full(j.size, synth.REF_SIGMA_V), synth.REF_SIGMA_Z0 * g[:, 0],
                  np.full(j.size, synth.REF_SIGMA_Z0), np.sinh(p.trk_eta[j]) + synth.REF_SIGMA_TL * g[:, 1],
                  np.full(j.size, synth.REF_SIGMA_TL), q + sq * g[:, 2], sq, np.zeros(j.size)], axis=1)
    return torch.as_tensor((a * ok[:, None]).astype(np.float32), device=dev)


def _refit_input(case, seed, dev):
    """Clusters distorted by a calibration, the tracks, weights and references of one refit call."""
    rng = np.random.default_rng([seed, 7])
    cl, truth = _clusters(case, seed, np.array([case["tracks"]]), dev, theta=_theta(rng))
    off, hits, trk = _given_tracks(truth, dev)
    # the calibration leaves out some tracks (a cut on the quality of the nominal fit)
    weight = torch.as_tensor((rng.random(off.numel() - 1) > 0.05).astype(np.float32), device=dev)
    anchor = _references(truth, off, hits, trk, rng, dev) if case["anchors"] else None
    theta = torch.as_tensor(synth.theta_nominal(), dtype=torch.float64, device=dev)
    theta[0] += 2.0 ** -12           # a point on the way, exactly representable in 32 bits
    theta[1:37] += torch.as_tensor(np.round(rng.normal(0.0, 0.01, 36) * 4096) / 4096, device=dev)
    theta[37:] += torch.as_tensor(np.round(rng.normal(0.0, 0.02, 36) * 4096) / 4096, device=dev)
    return cl, truth, off, hits, weight, anchor, theta


# ---- the cases' state and calls ----------------------------------------------------------------

def _room(case):
    """Clusters that the output buffers of a case hold: a program keeps buffers for its largest event."""
    n = float(_multiplicities(case).sum() if "events" in case else case["tracks"])
    return int((200 * n + 1000 * math.sqrt(n) + 1024) * (1.0 + case["noise"]))


def _tracks(n, n_events):
    """Output buffers; values past the last track are not written by the library and start at 0."""
    t = capi.Tracks(n, n_events, n // 32 + 256, n)
    for name in ("label", "trk_off", "trk_hits", "ev_trk_off", "par", "xref", "cov", "chi2", "ndf", "n_tracks"):
        getattr(t, name).zero_()
    return t


def _context(cl):
    return capi.Context(max_clusters=cl.n_clusters, max_events=cl.n_events)


def prepare(case, seed):
    dev = torch.device("cuda")
    call = case["call"]
    st = SimpleNamespace(call=call)
    if call == "refit":
        st.cl, _, off, hits, st.weight, st.anchor, st.theta = _refit_input(case, seed, dev)
        st.tr = capi.Tracks(st.cl.n_clusters, 1, off.numel(), hits.numel())
        st.tr.trk_off[:off.numel()] = off.to(torch.int32)
        st.tr.trk_hits[:] = hits.to(torch.int32)
        st.tr.n_tracks.fill_(off.numel() - 1)
        st.model = capi.TPC_ERRORS_RAW if case["raw"] else capi.TPC_ERRORS_FIXED
        st.sum = torch.zeros(1, dtype=torch.float64, device=dev)
        st.grad = torch.zeros(73, dtype=torch.float64, device=dev) if case["backward"] else None
        st.ctx = _context(st.cl)
    elif call in ("event", "its", "loopers", "links"):
        st.cl, truth = _clusters(case, seed, np.array([case["tracks"]]), dev,
                                 single_sector=case.get("sector", False), dead=case.get("dead", False))
        n = _room(case)
        if call == "links":
            st.geom = capi.default_geometry()
            st.up = torch.zeros(n, dtype=torch.int32, device=dev)
            st.down = torch.zeros(n, dtype=torch.int32, device=dev)
            st.status = torch.zeros(1, dtype=torch.int32, device=dev)
            return st
        st.ctx = _context(st.cl)
        st.ctx.tpc_set_rules(case.get("rules", 0))
        st.tr = _tracks(n, 1)
        if call != "event":            # the matching steps take the fitted tracks of a tracking call
            st.ctx.tpc_track_event(st.cl, st.tr)
            zeros = lambda m, dt: torch.zeros(m, dtype=dt, device=dev)
            if call == "its":
                its, _ = synth.its_tracks(truth.p, seed=seed % 100003)
                st.its = torch.as_tensor(its.astype(np.float32), device=dev)
                st.match_trk = zeros(st.tr.cap_tracks, torch.int32)
                st.match_its = zeros(case["tracks"] * 11 // 10 + 64, torch.int32)
                st.anchor = zeros((st.tr.cap_tracks, 8), torch.float32)
            else:
                st.pair, st.leg = zeros(st.tr.cap_tracks, torch.int32), zeros(st.tr.cap_tracks, torch.int32)
    else:
        frame = case["slice_len"] if call == "frame" else None
        st.cl, _ = _clusters(case, seed, _multiplicities(case), dev, frame=frame)
        st.ctx = _context(st.cl)
        n = _room(case)
        st.tr = _tracks(n, case["events"] if frame is None else 2 * case["events"] * synth.DRIFT_LSB // frame + 8)
        if call == "frame":
            st.slice_len = frame
            st.fr = _tracks(n, 1)
        elif call == "step":
            st.theta = torch.as_tensor(synth.theta_nominal(), dtype=torch.float64, device=dev)
            st.sum = torch.zeros(1, dtype=torch.float64, device=dev)
            st.grad = torch.zeros(73, dtype=torch.float64, device=dev)
    return st


def _result(t):
    return {"label": t.label, "trk_off": t.trk_off, "trk_hits": t.trk_hits, "ev_trk_off": t.ev_trk_off, "par": t.par,
            "xref": t.xref, "cov": t.cov, "chi2": t.chi2, "ndf": t.ndf, "n_tracks": t.n_tracks}


def run(st):
    if st.call == "event":
        st.ctx.tpc_track_event(st.cl, st.tr)
        return _result(st.tr)
    if st.call == "batch":
        st.ctx.tpc_track_batch(st.cl, st.tr)
        return _result(st.tr)
    if st.call == "step":
        st.ctx.tpc_track_refit_batch(st.cl, st.tr, st.theta, st.sum, st.grad)
        return dict(_result(st.tr), sum_chi2=st.sum, grad=st.grad)
    if st.call == "refit":
        st.ctx.tpc_refit_grad(st.cl, st.tr, st.theta, st.sum, st.grad, st.weight, st.anchor, st.model)
        return {"sum_chi2": st.sum, "grad": st.grad}
    if st.call == "its":
        st.ctx.tpc_its_match(st.cl, st.tr, st.its, st.match_trk, st.match_its, st.anchor)
        return {"match_trk": st.match_trk, "match_its": st.match_its, "anchor": st.anchor}
    if st.call == "loopers":
        st.ctx.tpc_looper_pairs(st.cl, st.tr, st.pair, st.leg)
        return {"pair": st.pair, "leg": st.leg}
    if st.call == "frame":
        st.ctx.tpc_track_batch(st.cl, st.tr)
        st.ctx.tpc_merge_slices(st.cl, st.tr, st.slice_len, st.fr)
        f = st.fr
        return dict(_result(st.tr), frame={"label": f.label, "trk_off": f.trk_off, "trk_hits": f.trk_hits,
                                           "ev_trk_off": f.ev_trk_off, "n_tracks": f.n_tracks})
    capi.check(capi.tpc_links_noalloc(st.geom, st.cl, st.up, st.down, st.status), "tpc_links_noalloc")
    return {"up": st.up, "down": st.down, "status": st.status}


# ---- what a call cannot do without -------------------------------------------------------------

FLOP_REFIT = 434.0              # FP32 operations per hit of the square-root filter (counted)
FLOP_FORWARD = 461.0            # ... of the covariance-form filter
FLOP_ADJOINT = 850.0            # ... of its adjoint step


def work(case):
    call = case["call"]
    if call in ("batch", "step", "frame"):
        n_trk, bins = float(_multiplicities(case).sum()), case["events"] * NB
    else:
        n_trk, bins = float(case["tracks"]), NB
    hits = HITS_PER_TRACK * n_trk
    n = hits * (1.0 + case["noise"])                  # clusters
    event_in = 4 * n + 4 * bins                       # pad, time, bin offsets
    result = 4 * n + 4 * hits + 100 * n_trk           # labels, hit lists, fitted tracks
    if call == "links":
        return {"bytes": event_in + 8 * n, "flops": 0.0}
    if call == "refit":
        per_hit = FLOP_FORWARD + (FLOP_ADJOINT if case["backward"] else 0.0)
        # the hit lists, the cluster of every hit (coordinates; sector and row through the bins)
        return {"bytes": 8 * hits + 4 * bins + (40 if case["anchors"] else 8) * n_trk, "flops": per_hit * hits}
    if call == "its":        # state and covariance in; the matches and references out
        return {"bytes": 96 * n_trk + 32 * n_trk + 40 * n_trk, "flops": 0.0}
    if call == "loopers":
        return {"bytes": 32 * n_trk + 8 * n_trk, "flops": 0.0}
    w = {"bytes": event_in + result, "flops": FLOP_REFIT * hits}
    if call == "step":
        w["flops"] += (FLOP_FORWARD + FLOP_ADJOINT) * hits
    if call == "frame":
        w["bytes"] += 4 * n + 8 * hits
    return w


# ---- the refit in 64 bits ------------------------------------------------------------------------

def _asinc(u):
    small = u.abs() < 0.05
    v = torch.where(small, torch.full_like(u, 0.5), u)
    u2 = u * u
    ser = 1 + u2 * (1 / 6 + u2 * (3 / 40 + u2 * (5 / 112 + u2 * (35 / 1152 + u2 * (63 / 2816 + u2 * (231 / 13312))))))
    return torch.where(small, ser, torch.asin(v.clamp(-1, 1)) / v)


def _fill(n, dev, entries):
    """Batched 5x5 identity with the given (i, j): value entries."""
    one, zero = torch.ones(n, dtype=torch.float64, device=dev), torch.zeros(n, dtype=torch.float64, device=dev)
    rows = [torch.stack([entries.get((i, j), one if i == j else zero) for j in range(5)], -1) for i in range(5)]
    return torch.stack(rows, -2)


def _propagate(p, P, dx):
    """Exact helix step by dx: state, covariance, and whether it stays in the local parametrisation."""
    sn, tl, q = p[:, 2], p[:, 3], p[:, 4]
    s2 = sn + synth.KB * q * dx
    ok = (s2.abs() < 0.999) & (sn.abs() < 0.999)
    a, b = torch.where(ok, sn, 0 * sn), torch.where(ok, s2, 0 * sn)
    c1, c2 = torch.sqrt(1 - a * a), torch.sqrt(1 - b * b)
    T = (a + b) / (c1 + c2)
    sW = torch.sqrt(1 + T * T)
    L = dx * sW
    arc = L * _asinc(0.5 * synth.KB * q * L)
    h, g = 0.5 * (1 / c1 + 1 / c2), 0.5 / c2 * synth.KB * dx * dx
    F = _fill(p.shape[0], p.device, {(0, 2): dx * (1 + T * T) * h, (0, 4): (1 + T * T) * g, (1, 2): tl * dx * T * sW * h,
                                     (1, 3): arc, (1, 4): tl * T * sW * g, (2, 4): synth.KB * dx})
    pn = torch.stack([p[:, 0] + dx * T, p[:, 1] + tl * arc, b, tl, q], -1)
    return pn, F @ P @ F.transpose(1, 2), ok


def _update(p, P, idx, meas, var):
    """Scalar measurement of component idx: the updated state and covariance and its chi2."""
    u = P[:, :, idx]
    S = u[:, idx] + var
    r = meas - p[:, idx]
    return p + u * (r / S)[:, None], P - u[:, :, None] * u[:, None, :] / S[:, None, None], r * r / S


def _chi2_chunk(th, off, n, sec, row, yraw, drift, anchor, raw):
    """chi2 of a chunk of tracks under theta (0 for a failed fit); differentiable in theta."""
    dev, m, nmax = th.device, off.numel(), int(n.max())
    row_x = torch.as_tensor(synth.ROW_X, device=dev)
    w = math.radians(2 * synth.HALF_ANGLE_DEG)

    def hit(i):              # hit i of every track: sector, calibrated (x, y, z), variances
        j = off + i
        k, x, y, D = sec[j], row_x[row[j]], yraw[j], drift[j]
        side = torch.where(k < 18, 1.0, -1.0).double()
        rho = torch.hypot(x, y)
        corr = th[37 + k] * (rho - synth.X_FIRST) / ((synth.X_LAST - synth.X_FIRST) * rho)
        vy = 0.01 * ((1 + corr) ** 2 if raw else torch.ones_like(corr))
        vz = 0.01 * (th[0] ** 2 if raw else 1.0) * torch.ones_like(corr)
        return k, x * (1 + corr), y * (1 + corr), side * (synth.Z_MAX - th[0] * D) + th[1 + k], vy, vz

    with torch.no_grad():    # the seed: circle through the nominal first, middle and last hit
        def nominal(i, ke):
            j = off + i
            da = (sec[j] % 18 - ke % 18).double() * w
            x, y = row_x[row[j]], yraw[j]
            z = torch.where(sec[j] < 18, 1.0, -1.0).double() * (synth.Z_MAX - drift[j])
            return x * torch.cos(da) - y * torch.sin(da), x * torch.sin(da) + y * torch.cos(da), z
        ke = sec[off + n - 1]
        ax, ay, az = nominal(0, ke)
        bx, by, _ = nominal((n - 1) // 2, ke)
        ex, ey, ez = nominal(n - 1, ke)
        cross = (bx - ax) * (ey - by) - (by - ay) * (ex - bx)
        lae = torch.hypot(ex - ax, ey - ay)
        kappa = 2 * cross / (torch.hypot(bx - ax, by - ay) * torch.hypot(ex - bx, ey - by) * lae)
        u = 0.5 * kappa * lae
        sn = ((ey - ay) * torch.sqrt((1 - u * u).clamp(min=0)) + (ex - ax) * u) / lae
        ok = (u.abs() < 1) & (sn.abs() < 0.999) & (n >= 3)
        sn = torch.where(ok, sn, 0 * sn)
        seed = (sn, (ez - az) / (lae * _asinc(u)), kappa / synth.KB)
    frame, x, y, z, _, _ = hit(n - 1)
    p = torch.stack([y, z, *seed], -1)
    P = torch.diag(torch.tensor([1.0, 1.0, 0.01, 0.01, 1.0], dtype=torch.float64, device=dev)).expand(m, 5, 5)
    chi2 = torch.zeros(m, dtype=torch.float64, device=dev)
    for q in range(nmax):
        on = (q < n) & ok
        k, hx, hy, hz, vy, vz = hit((n - 1 - q).clamp(min=0))
        da = (k % 18 - frame % 18).double() * w
        ca, sa = torch.cos(da), torch.sin(da)
        s0 = p[:, 2]
        c0 = torch.sqrt(1 - s0 * s0)
        c1 = c0 * ca + s0 * sa
        fits = c1 > 0.01
        c1 = torch.where(fits, c1, torch.ones_like(c1))
        J = _fill(m, dev, {(0, 0): c0 / c1, (1, 0): -p[:, 3] * sa / c1, (2, 0): -synth.KB * p[:, 4] * sa, (2, 2): c1 / c0})
        x1 = x * ca + p[:, 0] * sa
        p1 = torch.stack([-x * sa + p[:, 0] * ca, p[:, 1], s0 * ca - c0 * sa, p[:, 3], p[:, 4]], -1)
        p1 = torch.where((fits & on)[:, None], p1, p)
        x1 = torch.where(fits & on, x1, x)
        dx = torch.where(on & fits, hx - x1, torch.zeros_like(x1))
        p2, P2, inside = _propagate(p1, J @ P @ J.transpose(1, 2), dx)
        p3, P3, ca2 = _update(p2, P2, 0, hy, vy)
        p3, P3, cb2 = _update(p3, P3, 1, hz, vz)
        good = on & fits & inside
        p, P = torch.where(good[:, None], p3, p), torch.where(good[:, None, None], P3, P)
        chi2 = chi2 + torch.where(good, ca2 + cb2, torch.zeros_like(ca2))
        x = torch.where(good, hx, x)
        frame = torch.where(good, k, frame)
        ok = ok & (good | (q >= n))
    if anchor is not None:
        use = ok & (anchor[:, [0, 2, 4, 6]] > 0).any(1)
        p1, P1, inside = _propagate(p, P, torch.where(use, -x, torch.zeros_like(x)))
        ok = ok & (inside | ~use)
        zero = torch.zeros_like(x)
        for idx, meas, sig in ((0, zero, anchor[:, 0]), (1, zero, anchor[:, 0]), (1, anchor[:, 1], anchor[:, 2]),
                               (3, anchor[:, 3], anchor[:, 4]), (4, anchor[:, 5], anchor[:, 6])):
            on = use & ok & (sig > 0)
            p2, P2, c = _update(p1, P1, idx, meas, torch.where(sig > 0, sig, torch.ones_like(sig)) ** 2)
            p1, P1 = torch.where(on[:, None], p2, p1), torch.where(on[:, None, None], P2, P1)
            chi2 = chi2 + torch.where(on, c, torch.zeros_like(c))
    return torch.where(ok, chi2, torch.zeros_like(chi2))


def _refit_64(cl, truth, off, hits, weight, anchor, theta, raw, backward, chunk=6144):
    n = off[1:] - off[:-1]
    u16 = cl.time_fp.long() & 0xffff
    sec, row = truth.sector[hits], truth.row[hits]
    y, drift = cl.pad_fp[hits].double() * synth.LSB, u16[hits].double() * synth.LSB
    order = torch.argsort(n)
    total = torch.zeros(1, dtype=torch.float64, device=theta.device)
    grad = torch.zeros_like(theta)
    for c0 in range(0, order.numel(), chunk):
        t = order[c0:c0 + chunk]
        th = theta.clone().requires_grad_(backward)
        with torch.set_grad_enabled(backward):
            c2 = _chi2_chunk(th, off[t], n[t], sec, row, y, drift, None if anchor is None else anchor[t].double(), raw)
            f = (c2 * weight[t].double()).sum()
        if backward:
            f.backward()
            grad += th.grad
        total += f.detach()
    return total, grad


def exact(case, seed):
    """The refit calls in 64 bits, by autograd through a plain Kalman filter; the other calls decide
    in integers, or fit the tracks that they find themselves."""
    if case["call"] != "refit":
        return None
    cl, truth, off, hits, weight, anchor, theta = _refit_input(case, seed, torch.device("cuda"))
    total, grad = _refit_64(cl, truth, off, hits, weight, anchor, theta, case["raw"], case["backward"])
    return {"sum_chi2": total, "grad": grad if case["backward"] else None}
