"""Performance cases of the Kalman-filter track fitter.

Each case is one call that a reconstruction program makes: the fit of an event
or a batch of tracks (double or mixed precision, device or host data, with or
without the method variants), or the gradient of the fit for detector
alignment.  Inputs are simulated here from the seed alone: single charged
particles through a telescope of planes, multiple scattering drawn at every
plane, Gaussian hits, truth-smeared seeds.

``listed`` and ``draw`` give the cases, ``prepare`` what the program holds
before the call, ``run`` the call, ``work`` the bytes and operations the call
cannot do without, ``exact`` the same results from plain torch in 64 bits.

Fields of a case:
  call       "ex" (kf_fit_ex), "static" (kf_fit_static), "host" (kf_fit_host),
             "chi2_grad" (kf_chi2_grad), "autograd" (fit_autograd, forward and
             backward)
  precision  0 double, 1 mixed
  schedule   -1: the shape kf_autotune picked for this batch (tuned once per
             shape, as the handle caches it); None: the library's default;
             else a kf_schedule
  tracks, planes, gap (mm between planes), x0 (x/X0 of a plane), sigma (mm),
  pmin, pmax (GeV, log-uniform)
  ragged     each track crosses only its first U{5..planes} planes
  holes      probability that a crossed plane has no measurement
  tilt       planes tilted by up to this angle (rad); 0: all perpendicular to x
  field      "z" (2 T along z) or "general" (2 T in a general direction) or
             "map" (a falling 2 T field given as a grid map)
  corr       seed covariances with correlations, hit covariances too
  states     smoothed parameters on every state are wanted
  eloss, bf  energy loss; backward-filter smoother
"""
import math

import numpy as np
import torch

import paper_2105_01796_gb300 as kf

KAPPA = 2.99792458e-4   # GeV / (T mm)
C_LIGHT = 299.792458    # mm / ns
MASS = 0.1056583755     # muon, GeV
H_MAX, N_ITER = 50.0, 3
SILICON = (0.49848, 173.0e-9, 21.82, 4.4355, 0.2015, 2.8716, 0.1492, 3.2546, 0.14)
BF_SCALE = 1.0e4

_BASE = dict(call="ex", precision=0, schedule=None, tracks=1000, planes=10, gap=30.0, x0=0.005, sigma=0.05,
             pmin=1.0, pmax=10.0, ragged=False, holes=0.0, tilt=0.0, field="z", corr=False, states=False,
             eloss=False, bf=False)


def _case(name=None, **kw):
    c = dict(_BASE, **kw)
    return dict(c, name=name) if name else c


def listed():
    return [
        # one small event in a loop that must never allocate (a trigger):
        # latency of the calls and of a single warp per unit
        _case("trigger_97", call="static", tracks=97),
        # one event of the telescope with the launch shape tuned once
        _case("event_1k_fp64", schedule=-1, tracks=1000),
        # one event in mixed precision as a first-time user calls it
        _case("event_3k_mixed", precision=1, tracks=3001, planes=13, gap=27.0, x0=0.01),
        # the bulk reconstruction batch of the benchmark, mixed and double
        _case("batch_100k_mixed", precision=1, schedule=-1, tracks=100_000, planes=30, gap=25.0, x0=0.01,
              sigma=0.03, pmin=0.5, pmax=100.0),
        _case("batch_100k_fp64", tracks=100_000, planes=30, gap=25.0, x0=0.01, sigma=0.03, pmin=0.5, pmax=100.0),
        # a large sample of tracks of uneven length with missing hits
        _case("uneven_1m_mixed", precision=1, schedule=-1, tracks=1_000_000, planes=30, gap=25.0, x0=0.01,
              pmin=1.0, pmax=50.0, ragged=True, holes=0.05),
        # a real detector: tilted planes, a field along no axis, correlated
        # seeds and hits, uneven tracks, residuals wanted on every surface
        _case("tilted_20k_states", schedule=2, tracks=20_011, planes=24, gap=31.0, x0=0.01, pmin=0.5, pmax=50.0,
              ragged=True, holes=0.05, tilt=0.15, field="general", corr=True, states=True),
        # host arrays in, host arrays out
        _case("host_60k_fp64", call="host", tracks=60_000, planes=15, gap=30.0),
        # dense material: mean energy loss with the baseline smoother
        _case("eloss_50k", tracks=50_000, planes=20, gap=30.0, x0=0.02, pmin=0.5, pmax=20.0, eloss=True),
        # every method variant: field map, energy loss, backward filter
        _case("variants_map_30k", tracks=30_000, planes=30, gap=25.0, x0=0.01, sigma=0.03, pmin=0.5, pmax=100.0,
              field="map", eloss=True, bf=True),
        # detector alignment: the chi2 gradient over a large sample, and the
        # differentiable fit of one event inside a training step
        _case("align_chi2_100k", call="chi2_grad", tracks=100_000, planes=20),
        _case("align_autograd_2k", call="autograd", tracks=2_000, planes=20),
    ]


def _log_int(rng, lo, hi):
    n = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
    return min(hi, max(lo, n | (rng.random() < 0.5)))


def draw(rng):
    kind = rng.choice(["static", "event", "mixed", "mixed", "fp64", "fp64", "general", "host", "eloss", "map",
                       "chi2_grad", "autograd"])
    planes = rng.randint(5, 30)
    c = dict(planes=planes, gap=round(rng.uniform(15.0, min(60.0, 900.0 / planes)), 1),
             x0=round(rng.uniform(0.002, 0.02), 4), sigma=round(rng.uniform(0.02, 0.06), 3),
             pmin=round(rng.uniform(0.5, 1.5), 2), pmax=round(rng.uniform(8.0, 100.0), 1))
    ragged = planes >= 8 and rng.random() < 0.5
    holes = round(rng.uniform(0.01, 0.08), 3) if rng.random() < 0.5 else 0.0
    if kind == "static":
        return _case(call="static", precision=rng.randint(0, 1), tracks=_log_int(rng, 32, 4000), holes=holes, **c)
    if kind == "event":
        return _case(schedule=-1, tracks=_log_int(rng, 200, 5000), holes=holes, ragged=ragged, **c)
    if kind == "mixed":
        return _case(precision=1, schedule=rng.choice([None, -1, 2]), tracks=_log_int(rng, 1000, 500_000),
                     ragged=ragged, holes=holes, field=rng.choice(["z", "z", "general"]),
                     tilt=rng.choice([0.0, 0.1]), corr=rng.random() < 0.5, **c)
    if kind == "fp64":
        return _case(schedule=rng.choice([None, 0, 2]), tracks=_log_int(rng, 1000, 150_000), ragged=ragged,
                     holes=holes, corr=rng.random() < 0.5, **c)
    if kind == "general":
        return _case(precision=rng.randint(0, 1), schedule=rng.choice([None, 2]), tracks=_log_int(rng, 1000, 60_000),
                     ragged=ragged, holes=holes, tilt=round(rng.uniform(0.02, 0.15), 3), field="general", corr=True,
                     states=True, **c)
    if kind == "host":
        return _case(call="host", tracks=_log_int(rng, 1000, 80_000), ragged=ragged, holes=holes, **c)
    if kind == "eloss":
        return _case(tracks=_log_int(rng, 1000, 60_000), ragged=ragged, holes=holes, eloss=True, **c)
    if kind == "map":
        c["gap"] = min(c["gap"], round(800.0 / planes, 1))
        return _case(tracks=_log_int(rng, 1000, 30_000), ragged=ragged, holes=holes, field="map",
                     eloss=rng.random() < 0.5, bf=rng.random() < 0.5, **c)
    if kind == "chi2_grad":
        return _case(call="chi2_grad", tracks=_log_int(rng, 500, 100_000), holes=holes, **dict(c, planes=min(planes, 20)))
    return _case(call="autograd", tracks=_log_int(rng, 500, 20_000), holes=holes, **dict(c, planes=min(planes, 20)))


# --------------------------------------------------------------------------
# the method in plain torch, 64 bits: used to simulate the truth and by exact()
# --------------------------------------------------------------------------

def _dev():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _dot(a, b):
    return (a * b).sum(1)


def _bound_to_free(c, R, x):
    """Position and unit direction of bound parameters x [T,6], and the
    columns d/d(loc0, loc1, phi, theta, q/p) of both."""
    sp, cp, st, ct = torch.sin(x[:, 2]), torch.cos(x[:, 2]), torch.sin(x[:, 3]), torch.cos(x[:, 3])
    r = c + R[:, :, 0] * x[:, 0:1] + R[:, :, 1] * x[:, 1:2]
    T = torch.stack([cp * st, sp * st, ct], 1)
    z = torch.zeros_like(T)
    o = torch.zeros_like(sp)
    gr = torch.stack([R[:, :, 0], R[:, :, 1], z, z, z], 2)
    gT = torch.stack([z, z, torch.stack([-sp * st, cp * st, o], 1), torch.stack([cp * ct, sp * ct, -st], 1), z], 2)
    return r, T, gr, gT


def _field(fld, r):
    """Field at r [T,3]: a constant, or the trilinear map clamped to its grid."""
    if fld["map"] is None:
        return fld["b"].expand_as(r)
    b, n = fld["map"], fld["n"]
    u = torch.minimum(torch.clamp((r - fld["origin"]) / fld["spacing"], min=0.0), n - 1.0)
    i = torch.minimum(torch.floor(u), n - 2.0)
    w, i = u - i, i.long()
    out = 0.0
    for dl in (0, 1):
        for dj in (0, 1):
            for di in (0, 1):
                wt = ((w[:, 0] if di else 1 - w[:, 0]) * (w[:, 1] if dj else 1 - w[:, 1])
                      * (w[:, 2] if dl else 1 - w[:, 2]))
                out = out + wt[:, None] * b[i[:, 2] + dl, i[:, 1] + dj, i[:, 0] + di]
    return out


def _rkn(fld, r, T, t, lam, h, gr=None, gT=None, gt=None):
    """One Runge-Kutta-Nystrom step of length h [T], with the derivative of
    the step (stage fields held fixed) applied to the columns."""
    lk = (lam * KAPPA)[:, None]
    H = h[:, None]
    cr = torch.linalg.cross
    B1 = _field(fld, r)
    x1 = cr(T, B1)
    B2 = _field(fld, r + 0.5 * H * T + H * H / 8.0 * lk * x1)
    x2 = cr(T + 0.5 * H * lk * x1, B2)
    x3 = cr(T + 0.5 * H * lk * x2, B2)
    B4 = _field(fld, r + H * T + 0.5 * H * H * lk * x3)
    x4 = cr(T + H * lk * x3, B4)
    g = torch.sqrt(1.0 + MASS * MASS * lam * lam)
    if gr is not None:
        q = torch.zeros(5, dtype=r.dtype, device=r.device)
        q[4] = KAPPA
        L, H3 = lk[:, :, None], H[:, :, None]
        c5 = lambda v, B: cr(v, B[:, :, None].expand_as(v), dim=1)  # noqa: E731
        d1 = L * c5(gT, B1) + q * x1[:, :, None]
        d2 = L * c5(gT + 0.5 * H3 * d1, B2) + q * x2[:, :, None]
        d3 = L * c5(gT + 0.5 * H3 * d2, B2) + q * x3[:, :, None]
        d4 = L * c5(gT + H3 * d3, B4) + q * x4[:, :, None]
        gr = gr + H3 * gT + H3 * H3 / 6.0 * (d1 + d2 + d3)
        gT = gT + H3 / 6.0 * (d1 + 2.0 * d2 + 2.0 * d3 + d4)
        e4 = torch.zeros(5, dtype=r.dtype, device=r.device)
        e4[4] = 1.0
        gt = gt + (h * MASS * MASS * lam / (C_LIGHT * g))[:, None] * e4
    r = r + H * T + H * H / 6.0 * lk * (x1 + x2 + x3)
    T = T + H / 6.0 * lk * (x1 + 2.0 * x2 + 2.0 * x3 + x4)
    return r, T, t + h * g / C_LIGHT, gr, gT, gt


def _propagate(fld, r, T, t, lam, c, n, gr=None, gT=None, gt=None):
    """To the plane (c, n): equal steps of at most H_MAX over the straight-line
    distance, then N_ITER corrections."""
    s0 = _dot(n, c - r) / _dot(n, T)
    nsub = torch.clamp(torch.ceil(s0.detach().abs() / H_MAX), min=1.0)
    most = min(64, int(nsub.max()))
    h = s0 / nsub
    for k in range(most):
        hk = h if k == 0 else torch.where(nsub > k, h, torch.zeros_like(h))
        r, T, t, gr, gT, gt = _rkn(fld, r, T, t, lam, hk, gr, gT, gt)
    for _ in range(N_ITER):
        r, T, t, gr, gT, gt = _rkn(fld, r, T, t, lam, _dot(n, c - r) / _dot(n, T), gr, gT, gt)
    return r, T, t, gr, gT, gt


def _transport(fld, ca, Ra, x, cb, Rb):
    """Prediction [T,6], Jacobian [T,6,6], sin(theta) and incidence cosine."""
    r, T, gr, gT = _bound_to_free(ca, Ra, x)
    n, lam = Rb[:, :, 2], x[:, 4]
    gt = torch.zeros_like(x[:, :5])
    r, T, t, gr, gT, gt = _propagate(fld, r, T, x[:, 5], lam, cb, n, gr, gT, gt)
    nT = _dot(n, T)
    w = -(n[:, :, None] * gr).sum(1) / nT[:, None]
    AT = (lam * KAPPA)[:, None] * torch.linalg.cross(T, _field(fld, r))
    gr = gr + T[:, :, None] * w[:, None, :]
    gT = gT + AT[:, :, None] * w[:, None, :]
    gt = gt + (torch.sqrt(1.0 + MASS * MASS * lam * lam) / C_LIGHT)[:, None] * w
    phi = torch.atan2(T[:, 1], T[:, 0])
    theta = torch.atan2(torch.sqrt(T[:, 0] ** 2 + T[:, 1] ** 2), T[:, 2])
    sp, cp, st, ct = torch.sin(phi), torch.cos(phi), torch.sin(theta), torch.cos(theta)
    d = r - cb
    xp = torch.stack([_dot(d, Rb[:, :, 0]), _dot(d, Rb[:, :, 1]), phi, theta, lam, t], 1)
    rows = [(Rb[:, :, 0:1] * gr).sum(1), (Rb[:, :, 1:2] * gr).sum(1),
            (-sp / st)[:, None] * gT[:, 0] + (cp / st)[:, None] * gT[:, 1],
            (cp * ct)[:, None] * gT[:, 0] + (sp * ct)[:, None] * gT[:, 1] - st[:, None] * gT[:, 2],
            torch.zeros_like(gt) + torch.tensor([0.0, 0, 0, 0, 1.0], dtype=x.dtype, device=x.device), gt]
    last = torch.zeros_like(x)
    last[:, 5] = 1.0
    F = torch.cat([torch.stack(rows, 1), last[:, :, None]], 2)
    return xp, F, st, nT / torch.sqrt(_dot(T, T))


def _highland_var(lam, xx0, cos_inc):
    """Variance of the projected scattering angle (zero without material)."""
    g2 = 1.0 + MASS * MASS * lam * lam
    some = xx0 > 0
    eps = torch.where(some, xx0, torch.ones_like(xx0)) / cos_inc.abs()
    th = 0.0136 * lam.abs() * torch.sqrt(g2) * torch.sqrt(eps) * (1.0 + 0.038 * torch.log(eps * g2))
    return torch.where(some, th * th, torch.zeros_like(th))


def _energy_loss(qop, xx0, cos_inc, sign):
    """New q/p, the Jacobian factor and the straggling variance of q/p."""
    za, iexc, x0rho, cbar, x0, x1, a, k, d0 = SILICON
    kb, me = 0.307075e-3, 0.51099895e-3
    some = xx0 > 0
    thick = xx0 * x0rho / cos_inc.abs()
    p = 1.0 / qop.abs()
    E = torch.sqrt(p * p + MASS * MASS)
    beta, bg = p / E, p / MASS
    b2, gam, rr = bg * bg / (1.0 + bg * bg), torch.sqrt(1.0 + bg * bg), me / MASS
    wmax = 2.0 * me * bg * bg / (1.0 + 2.0 * gam * rr + rr * rr)
    X = torch.log10(bg)
    hi = 2.0 * math.log(10.0) * X - cbar
    delta = torch.where(X >= x1, hi, torch.where(X >= x0, hi + a * torch.clamp(x1 - X, min=0.0) ** k,
                                                 d0 * 10.0 ** (2.0 * (X - x0))))
    dE = kb * za / b2 * (0.5 * torch.log(2.0 * me * bg * bg * wmax / (iexc * iexc)) - b2 - 0.5 * delta) * thick
    E2 = E + (-dE if sign > 0 else dE)
    p2 = torch.sqrt(E2 * E2 - MASS * MASS)
    sig = 2.0 * kb * za * thick / (beta * beta) / (2.0 * math.sqrt(2.0 * math.log(2.0)))
    Ed, pd = (E2, p2) if sign > 0 else (E, p)
    var = (Ed / pd ** 3 * sig) ** 2
    one = torch.ones_like(p)
    return (torch.where(some, torch.sign(qop) / p2, qop), torch.where(some, p ** 3 * E2 / (p2 ** 3 * E), one),
            torch.where(some, var, torch.zeros_like(p)))


def _update(x, C, m, V, keep):
    """Gain-matrix update in Joseph form; tracks with keep False stay as they are."""
    Vm = torch.stack([torch.stack([V[:, 0], V[:, 1]], 1), torch.stack([V[:, 1], V[:, 2]], 1)], 1)
    S = Vm + C[:, :2, :2]
    det = S[:, 0, 0] * S[:, 1, 1] - S[:, 0, 1] * S[:, 1, 0]
    Si = torch.stack([torch.stack([S[:, 1, 1], -S[:, 0, 1]], 1), torch.stack([-S[:, 1, 0], S[:, 0, 0]], 1)], 1)
    Si = Si / det[:, None, None]
    K = C[:, :, :2] @ Si
    r = m - x[:, :2]
    chi2 = (r[:, None, :] @ Si @ r[:, :, None])[:, 0, 0]
    H = torch.zeros(2, 6, dtype=x.dtype, device=x.device)
    H[0, 0] = H[1, 1] = 1.0
    L = torch.eye(6, dtype=x.dtype, device=x.device) - K @ H
    Cf = L @ C @ L.transpose(1, 2) + K @ Vm @ K.transpose(1, 2)
    xf = x + (K @ r[:, :, None])[:, :, 0]
    k1 = keep[:, None]
    return torch.where(k1, xf, x), torch.where(k1[:, :, None], Cf, C), torch.where(keep, chi2, torch.zeros_like(chi2))


_TRI = [(i, j) for i in range(6) for j in range(i + 1)]


def _unpack(c21):
    """[21][T] -> [T,6,6]"""
    rows = [[None] * 6 for _ in range(6)]
    for e, (i, j) in enumerate(_TRI):
        rows[i][j] = rows[j][i] = c21[e]
    return torch.stack([torch.stack(r, 1) for r in rows], 1)


def _pack(C):
    return torch.stack([C[:, i, j] for i, j in _TRI])


def _fit(ev, fld, center, rot, seed, sel, eloss=False, bf=False, smooth=True, states=False):
    """Forward filter and smoother of the tracks in `sel` (a slice): chi2 [T],
    params [6][T], cov [21][T], and the smoothed parameters of every state
    [K][T,6] when asked."""
    off = ev["offsets"].long()
    o0, n = off[:-1][sel], (off[1:] - off[:-1])[sel]
    K = int(n.max())
    x, C = seed.t(), _unpack(ev["seed_cov"][:, sel])
    cen, R = center.t(), rot.reshape(3, 3, -1).permute(2, 0, 1)
    rec = []
    sid0 = ev["surface_id"][o0].long()
    chi2 = torch.zeros_like(x[:, 0])
    for k in range(K):
        act = n > k
        at = o0 + torch.clamp(n - 1, max=k)
        sid = ev["surface_id"][at].long()
        F = None
        if k > 0:
            xp, F, st, ci = _transport(fld, cen[sid0], R[sid0], x, cen[sid], R[sid])
            xx0 = ev["x_over_x0"][sid]
            q = _highland_var(x[:, 4], xx0, ci)
            G = torch.ones_like(xp)
            Q = torch.zeros_like(xp)
            if eloss:
                qop, jac, var = _energy_loss(xp[:, 4], xx0, ci, +1)
                xp = torch.cat([xp[:, :4], qop[:, None], xp[:, 5:]], 1)
                F = torch.cat([F[:, :4], F[:, 4:5] * jac[:, None, None], F[:, 5:]], 1)
            else:
                var = Q[:, 0]
            Q = torch.stack([Q[:, 0], Q[:, 0], q / (st * st), q, var, Q[:, 0]], 1)
            Cp = F @ C @ F.transpose(1, 2) + torch.diag_embed(Q)
        else:
            xp, Cp = x, C
        xf, Cf, c2 = _update(xp, Cp, ev["loc"][:, at].t(), ev["cov"][:, at].t(), act & (ev["is_hole"][at] == 0))
        chi2 = chi2 + c2
        rec.append((xp, Cp, xf, Cf, F, act, sid) if smooth else None)
        a1 = act[:, None]
        x, C = torch.where(a1, xf, x), torch.where(a1[:, :, None], Cf, C)
        sid0 = torch.where(act, sid, sid0)
    if not smooth:
        return chi2, None, None, None
    xs, Cs = x, C
    out = [None] * K
    out[K - 1] = xs
    if bf:
        xb, Cb = x, BF_SCALE * C
    for k in range(K - 1, 0, -1):
        xp, Cp, _, _, F, act, sid = rec[k]
        _, _, xf, Cf, _, _, sidp = rec[k - 1]
        if bf:
            at = o0 + torch.clamp(n - 1, max=k)
            xu, Cu, _ = _update(xb, Cb, ev["loc"][:, at].t(), ev["cov"][:, at].t(), act & (ev["is_hole"][at] == 0))
            T = torch.stack([torch.cos(xu[:, 2]) * torch.sin(xu[:, 3]), torch.sin(xu[:, 2]) * torch.sin(xu[:, 3]),
                             torch.cos(xu[:, 3])], 1)
            ci, xx0 = _dot(R[sid][:, :, 2], T), ev["x_over_x0"][sid]
            q = _highland_var(xu[:, 4], xx0, ci)
            g = torch.ones_like(q)
            var = torch.zeros_like(q)
            if eloss:
                qop, g, var = _energy_loss(xu[:, 4], xx0, ci, -1)
                xu = torch.cat([xu[:, :4], qop[:, None], xu[:, 5:]], 1)
            z = torch.zeros_like(q)
            Cu = Cu + torch.diag_embed(torch.stack([z, z, q / torch.sin(xu[:, 3]) ** 2, q, var, z], 1))
            G = torch.stack([z + 1, z + 1, z + 1, z + 1, g, z + 1], 1)
            Cu = G[:, :, None] * Cu * G[:, None, :]
            xo, Fb, _, _ = _transport(fld, cen[sid], R[sid], xu, cen[sidp], R[sidp])
            Co = Fb @ Cu @ Fb.transpose(1, 2)
            d = 1.0 / torch.sqrt(torch.diagonal(Cf + Co, dim1=1, dim2=2))
            Kt = torch.linalg.solve(d[:, :, None] * (Cf + Co) * d[:, None, :], d[:, :, None] * Cf) * d[:, :, None]
            Kg = Kt.transpose(1, 2)
            xn, Cn = xf + (Kg @ (xo - xf)[:, :, None])[:, :, 0], Cf - Kg @ Cf
            a1 = act[:, None]
            xb, Cb = torch.where(a1, xo, xb), torch.where(a1[:, :, None], Co, Cb)
        else:
            d = 1.0 / torch.sqrt(torch.diagonal(Cp, dim1=1, dim2=2))
            X = torch.linalg.solve(d[:, :, None] * Cp * d[:, None, :], d[:, :, None] * (F @ Cf)) * d[:, :, None]
            A = X.transpose(1, 2)
            xn = xf + (A @ (xs - xp)[:, :, None])[:, :, 0]
            Cn = Cf + A @ (Cs - Cp) @ X
        a1 = act[:, None]
        xs, Cs = torch.where(a1, xn, xs), torch.where(a1[:, :, None], 0.5 * (Cn + Cn.transpose(1, 2)), Cs)
        out[k - 1] = xs
    return chi2, xs.t(), _pack(Cs), out if states else None


def _aligned(ev, align):
    """Geometry with every plane shifted and turned about its own axes."""
    R = ev["rot"].reshape(3, 3, -1).permute(2, 0, 1)
    center = ev["center"] + (R @ align[:3].t()[:, :, None])[:, :, 0].t()
    ca, sa, cb, sb, cg, sg = [f(align[i]) for i in (3, 4, 5) for f in (torch.cos, torch.sin)]
    o, z = torch.ones_like(ca), torch.zeros_like(ca)
    m = lambda *v: torch.stack(v, 1).reshape(-1, 3, 3)  # noqa: E731
    R2 = (R @ m(o, z, z, z, ca, -sa, z, sa, ca) @ m(cb, z, sb, z, o, z, -sb, z, cb)
          @ m(cg, -sg, z, sg, cg, z, z, z, o))
    return center, R2.permute(1, 2, 0).reshape(9, -1)


# --------------------------------------------------------------------------
# inputs
# --------------------------------------------------------------------------

def _torch_field(case, ev):
    dev = _dev()
    fld = {"b": torch.tensor(ev["bfield"], dtype=torch.float64, device=dev)[None], "map": None}
    fm = ev.get("field_map")
    if fm is not None:
        b = torch.as_tensor(fm["b"], device=dev)
        t = lambda v: torch.tensor(v, dtype=torch.float64, device=dev)  # noqa: E731
        fld.update(map=b, n=t([float(b.shape[2]), float(b.shape[1]), float(b.shape[0])]), origin=t(fm["origin"]),
                   spacing=t(fm["spacing"]))
    return fld


def _event(case, seed):
    """A simulated event on the device, in the library's layout."""
    dev, T, P = _dev(), case["tracks"], case["planes"]
    g = torch.Generator(device=dev)
    g.manual_seed(int(seed) * 1_000_003 + 17)
    kw = dict(generator=g, device=dev, dtype=torch.float64)
    uni = lambda lo, hi, *s: lo + (hi - lo) * torch.rand(*s, **kw)  # noqa: E731
    nrm = lambda *s: torch.randn(*s, **kw)  # noqa: E731
    S = P + 1
    # planes perpendicular to x (u = y, v = z, n = x), turned by small angles
    R0 = torch.tensor([[0.0, 0, 1], [1, 0, 0], [0, 1, 0]], dtype=torch.float64, device=dev)
    tilt = uni(-1.0, 1.0, 3, S) * case["tilt"]
    tilt[:, 0] = 0.0
    geo = {"center": torch.zeros(3, S, dtype=torch.float64, device=dev),
           "rot": R0.reshape(9, 1).expand(9, S).contiguous()}
    geo["center"][0] = torch.arange(S, device=dev, dtype=torch.float64) * case["gap"]
    _, rot = _aligned(geo, torch.cat([torch.zeros_like(tilt), tilt]))
    x0 = torch.full((S,), case["x0"], dtype=torch.float64, device=dev)
    x0[0] = 0.0
    b = (0.0, 0.0, 2.0) if case["field"] != "general" else (0.31, -0.62, 1.88)
    ev = {"n_tracks": T, "center": geo["center"].contiguous(), "rot": rot.contiguous(), "x_over_x0": x0, "bfield": b}
    if case["field"] == "map":
        xs = torch.arange(-50.0, 851.0, 25.0, dtype=torch.float64, device=dev)
        yz = torch.arange(-550.0, 551.0, 50.0, dtype=torch.float64, device=dev)
        Z, Y, X = torch.meshgrid(yz, yz, xs, indexing="ij")
        ev["field_map"] = {"b": torch.stack([-1.2e-6 * X * Z, 0 * X, 2.0 - 0.6e-6 * X * X], 3).contiguous(),
                           "origin": (-50.0, -550.0, -550.0), "spacing": (25.0, 50.0, 50.0)}
    fld = _torch_field(case, ev)
    # truth: angles, log-uniform momenta, either charge; scattered at every
    # plane.  More are simulated than wanted: the ones that turn back or leave
    # the 1 m x 1 m planes are dropped.
    want, T = T, T + T // 2 + 64
    good = torch.ones(T, dtype=torch.bool, device=dev)
    q = torch.where(uni(-1.0, 1.0, T) < 0, -1.0, 1.0).double()
    lam = q / torch.exp(uni(math.log(case["pmin"]), math.log(case["pmax"]), T))
    zero = torch.zeros(T, dtype=torch.float64, device=dev)
    x = torch.stack([zero, zero, uni(-0.3, 0.3, T), math.pi / 2 + uni(-0.3, 0.3, T), lam, zero], 1)
    R3 = rot.reshape(3, 3, S).permute(2, 0, 1)
    s = case["sigma"]
    smear = torch.tensor([10 * s, 10 * s, s / 10, s / 10, 0.0, 1.0], dtype=torch.float64, device=dev).expand(T, 6).clone()
    smear[:, 4] = 0.1 * lam.abs()
    z6 = nrm(T, 6)
    Cs = torch.diag_embed(smear * smear)
    if case["corr"]:
        rho = torch.eye(6, dtype=torch.float64, device=dev)
        for i, j, v in ((2, 0, 0.4), (3, 1, -0.3), (4, 2, 0.35), (5, 0, 0.15), (5, 3, -0.1)):
            rho[i, j] = rho[j, i] = v
        z6 = z6 @ torch.linalg.cholesky(rho).t()
        Cs = smear[:, :, None] * rho * smear[:, None, :]
    x0_true = x
    r, Td, _, _ = _bound_to_free(ev["center"].t()[:1].expand(T, 3), R3[:1].expand(T, 3, 3), x)
    t = zero
    loc = torch.zeros(T, S, 2, dtype=torch.float64, device=dev)
    rv = 0.3 if case["corr"] else 0.0
    for k in range(1, S):
        c, n = ev["center"].t()[k:k + 1].expand(T, 3), R3[k, :, 2][None].expand(T, 3)
        r, Td, t, _, _, _ = _propagate(fld, r, Td, t, lam, c, n)
        d = r - c
        ok = ((_dot(n, d).abs() < 1e-6) & (_dot(n, Td) > 0.2) & (d.abs().amax(1) < 500.0))
        good &= ok
        # a dropped track goes on along the normal from the plane's centre
        r, Td, d = [torch.where(ok[:, None], a, b) for a, b in ((r, c), (Td, n), (d, torch.zeros_like(d)))]
        e = nrm(T, 2)
        e = torch.stack([e[:, 0], rv * e[:, 0] + math.sqrt(1 - rv * rv) * e[:, 1]], 1)
        loc[:, k] = torch.stack([_dot(d, R3[k, :, 0][None]), _dot(d, R3[k, :, 1][None])], 1) + s * e
        th = torch.sqrt(_highland_var(lam, x0[k].expand(T), _dot(n, Td)))
        phi = torch.atan2(Td[:, 1], Td[:, 0])
        theta = torch.acos(torch.clamp(Td[:, 2], -1, 1))
        kick = nrm(T, 2)
        phi, theta = phi + th / torch.sin(theta) * kick[:, 0], theta + th * kick[:, 1]
        Td = torch.stack([torch.cos(phi) * torch.sin(theta), torch.sin(phi) * torch.sin(theta), torch.cos(theta)], 1)
    keep = good.nonzero()[:want, 0]
    T = want
    if keep.numel() < T:
        raise ValueError("too few tracks cross every plane: %r" % (case,))
    loc = loc[keep]
    ev["seed_params"] = (x0_true + z6 * smear)[keep].t().contiguous()
    ev["seed_cov"] = _pack(Cs[keep]).contiguous()
    n = torch.full((T,), S, device=dev, dtype=torch.int64)
    if case["ragged"]:
        # every length equally often, in random order: the same number of
        # states for every seed
        n = 6 + torch.randperm(T, generator=g, device=dev) % (P - 4)
    sid = torch.arange(S, device=dev)[None].expand(T, S)
    hole = torch.rand(T, S, **kw) < case["holes"]
    hole &= sid > 3           # at least three measurements
    hole[:, 0] = True         # the seed's reference plane
    live = sid < n[:, None]
    ev["offsets"] = torch.cat([torch.zeros(1, dtype=torch.int64, device=dev), n.cumsum(0)]).int()
    ev["surface_id"] = sid[live].int()
    ev["loc"] = loc[live].t().contiguous()
    M = ev["loc"].shape[1]
    V = torch.tensor([s * s, rv * s * s, s * s], dtype=torch.float64, device=dev)
    ev["cov"] = V[:, None].expand(3, M).contiguous()
    ev["is_hole"] = hole[live].to(torch.uint8)
    ev["max_states"] = int(n.max())
    return ev


def _weights(case, seed, ev):
    """Weights of the differentiated objective: chi2, parameters, covariance."""
    g = torch.Generator(device=_dev())
    g.manual_seed(int(seed) * 7919 + 3)
    kw = dict(generator=g, device=_dev(), dtype=torch.float64)
    T = case["tracks"]
    sd = torch.sqrt(torch.stack([ev["seed_cov"][i * (i + 1) // 2 + i] for i in range(6)]))
    w = 0.5 + torch.rand(T, **kw)
    v = torch.randn(6, T, **kw) / sd
    W = torch.randn(21, T, **kw) / torch.stack([sd[i] * sd[j] for i, j in _TRI])
    S = ev["center"].shape[1]
    align = torch.cat([0.1 * torch.randn(3, S, **kw), 1e-3 * torch.randn(3, S, **kw)])
    align[:, 0] = 0.0
    return w, v, W, align


_HANDLE = None


def _handle():
    global _HANDLE
    if _HANDLE is None:
        _HANDLE = kf.Handle()
    return _HANDLE


def prepare(case, seed):
    ev = _event(case, seed)
    s = {"case": case, "handle": _handle()}
    T, M = case["tracks"], ev["loc"].shape[1]
    if case["call"] in ("chi2_grad", "autograd"):
        s["w"], s["v"], s["W"], s["align"] = _weights(case, seed, ev)
        S = ev["center"].shape[1]
        z = dict(dtype=torch.float64, device=ev["loc"].device)
        s["out"] = {"chi2": torch.empty(T, **z), "seed": torch.empty(6, T, **z), "align": torch.empty(6, S, **z)}
        s["ev"] = ev
        return s
    # the options a user leaves alone are not set: the call takes its defaults
    s["opt"] = kf.kf_default_options(case["precision"], schedule=case["schedule"] if case["schedule"] not in (None, -1)
                                     else None, energy_loss=1 if case["eloss"] else None,
                                     smoother=kf.KF_SMOOTHER_BACKWARD_FILTER if case["bf"] else None)
    if case["call"] == "host":
        pin = lambda v: (v.cpu().pin_memory() if torch.cuda.is_available() else v.cpu()).numpy()  # noqa: E731
        s["ev"] = {k: pin(v) if isinstance(v, torch.Tensor) else v for k, v in ev.items()}
        out = {"params": (6, T), "cov": (21, T), "chi2": (T,)}
        s["out"] = {k: pin(torch.empty(v, dtype=torch.float64)) for k, v in out.items()}
        s["out"].update(ndf=pin(torch.empty(T, dtype=torch.int32)), status=pin(torch.empty(T, dtype=torch.uint8)),
                        states=None)
        return s
    s["ev"], s["out"] = ev, kf.alloc_outputs(T, M, with_states=case["states"])
    if case["schedule"] == -1:
        s["opt"], _ = kf.kf_autotune(s["handle"], ev, s["out"], s["opt"])
    return s


def run(s):
    case, ev, h = s["case"], s["ev"], s["handle"]
    if case["call"] == "chi2_grad":
        o = s["out"]
        kf.kf_chi2_grad(h, ev, align=s["align"], dl_dchi2=s["w"], out_chi2=o["chi2"], grad_seed=o["seed"],
                        grad_align=o["align"])
        return o
    if case["call"] == "autograd":
        seed, align = ev["seed_params"].detach().requires_grad_(), s["align"].detach().requires_grad_()
        chi2, params, cov = kf.fit_autograd(seed, align, ev, h)
        gs, ga = torch.autograd.grad([chi2, params, cov], [seed, align], [s["w"], s["v"], s["W"]])
        return {"chi2": chi2.detach(), "params": params.detach(), "cov": cov.detach(), "seed": gs, "align": ga}
    if case["call"] == "host":
        o = kf.kf_fit_host(h, ev, s["opt"], out=s["out"])
    elif case["call"] == "static":
        o = kf.kf_fit_static(ev, s["out"], s["opt"])
    else:
        o = kf.kf_fit_ex(h, ev, s["out"], s["opt"])
    o = {k: v for k, v in o.items() if v is not None}
    if case["precision"] == 1:
        # the mixed path computes these in float (or float pairs) and hands
        # them over in double containers; a program that chose it keeps floats
        o = {k: v.float() if v.dtype == torch.float64 else v for k, v in o.items()}
    return o


def _mean_states(case):
    return ((5 + case["planes"]) / 2 if case["ragged"] else case["planes"]) + 1


def work(case):
    T, M = case["tracks"], case["tracks"] * _mean_states(case)
    grad = case["call"] in ("chi2_grad", "autograd")
    # offsets, seeds and their covariances, states' surface, hit, its
    # covariance and the hole flag; results per track
    inputs = T * (4 + 27 * 8) + M * (4 + 2 * 8 + 3 * 8 + 1)
    outs = T * (7 * 8 if case["call"] == "chi2_grad" else (28 + 6) * 8 if grad else 28 * 8 + 5)
    if case["states"]:
        outs += M * 48
    # per state, with products that use the symmetry and the zeros: the
    # trajectory and its Jacobian 450, covariance transport 330, noise 15,
    # update 200, smoother 550; a reverse sweep costs twice its forward
    # pass; the backward filter is a second forward pass and a 6x6 solve
    fit = 1545.0 if case["call"] != "chi2_grad" else 995.0
    if case["bf"]:
        fit = 2 * 995.0 + 700.0
    if case["field"] == "map":
        fit += 4 * 3 * 60.0
    if case["eloss"]:
        fit += 80.0
    return {"bytes": inputs + outs, "flops": M * fit * (3.0 if grad else 1.0)}


def exact(case, seed):
    ev = _event(case, seed)
    fld = _torch_field(case, ev)
    T, dev = case["tracks"], _dev()
    grad = case["call"] in ("chi2_grad", "autograd")
    step = 5_000 if grad else 100_000
    if grad:
        w, v, W, align = _weights(case, seed, ev)
        ga = torch.zeros_like(align)
    parts = []
    states = None
    if case["states"]:
        states = torch.zeros(6, ev["loc"].shape[1], dtype=torch.float64, device=dev)
    for a in range(0, T, step):
        sel = slice(a, min(T, a + step))
        if grad:
            whole = case["call"] == "autograd"
            sd = ev["seed_params"][:, sel].detach().requires_grad_()
            al = align.detach().requires_grad_()
            center, rot = _aligned(ev, al)
            chi2, x, C, _ = _fit(ev, fld, center, rot, sd, sel, smooth=whole)
            L = (w[sel] * chi2).sum()
            if whole:
                L = L + (v[:, sel] * x).sum() + (W[:, sel] * C).sum()
            g1, g2 = torch.autograd.grad(L, [sd, al])
            ga += g2
            d = {"chi2": chi2.detach(), "seed": g1}
            if whole:
                d.update(params=x.detach(), cov=C.detach())
            del L, chi2, x, C
        else:
            with torch.no_grad():
                chi2, x, C, st = _fit(ev, fld, ev["center"], ev["rot"], ev["seed_params"][:, sel], sel,
                                      case["eloss"], case["bf"], True, case["states"])
                d = {"chi2": chi2, "params": x, "cov": C}
                if st is not None:
                    off = ev["offsets"].long()
                    o0, n = off[:-1][sel], (off[1:] - off[:-1])[sel]
                    for k, xs in enumerate(st):
                        m = n > k
                        states[:, (o0 + k)[m]] = xs[m].t()
        parts.append(d)
    out = {k: torch.cat([d[k] for d in parts], -1) for k in parts[0]}
    if grad:
        out["align"] = ga
    else:
        out["ndf"] = out["status"] = None
        if states is not None:
            out["states"] = states
    return {k: v.cpu().numpy() if case["call"] == "host" and v is not None else v for k, v in out.items()}
