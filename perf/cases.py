"""Timed cases of the framework's public entry points.

Each case is one call that a survey-prediction program makes through
``paper_2509_04666_gb300.kete.Kete``: the smallest interactive calls (one
orbit, one field list against a thousand bodies), the everyday ones (a
catalogue carried a year ahead, an ephemeris service's chain of epochs, orbit
fits) and the largest (a whole catalogue against two months of a scanning
survey).  ``listed`` names them, ``draw`` gives more of the same ranges.

Populations, cadences, frame sizes and force-model options are those of
``paper_2509_04666_gb300.workloads`` and ``bench.py``.  The planets are those
of one table per span, which a program loads once and keeps: bodies, frames
and observations come from the seed.

``exact`` integrates the same equations with an independent method in plain
torch FP64: a 12-stage Gauss-Legendre collocation (order 24) with fixed steps.
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

from paper_2509_04666_gb300 import kete, workloads as W

DEV = "cuda"
F64 = torch.float64


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------
def listed():
    return [
        # planet positions for the exposures of a survey year: the observer
        # table a user makes before a prediction (config: 150,000 exposures)
        {"name": "ephem_exposures", "kind": "ephem", "n": 150_000, "body": 3},
        # a handful of newly reported orbits carried a year ahead: the
        # smallest interactive call, latency only
        {"name": "few_orbits", "kind": "propagate", "pop": "catalogue", "n": 12, "days": 365.0,
         "mixed": False, "nongrav": False},
        # Monte-Carlo clones of one comet with the JPL non-gravitational
        # model, backward (the long-span configuration, shortened)
        {"name": "comet_clones", "kind": "clones", "n": 1000, "days": -2922.0},
        # a mixed catalogue one year ahead in one leg (the ragged
        # configuration: main belt, NEOs with forced encounters, Trojans,
        # comets), full precision
        {"name": "ragged_year", "kind": "propagate", "pop": "ragged", "n": 250_000,
         "days": 365.0, "mixed": False, "nongrav": False},
        # the same in mixed precision with the non-gravitational terms on the
        # bodies that carry them, an odd number of bodies
        {"name": "ragged_mixed_terms", "kind": "propagate", "pop": "ragged", "n": 100_003,
         "days": 180.0, "mixed": True, "nongrav": True},
        # states at a chain of irregular epochs (an ephemeris service)
        {"name": "state_service", "kind": "stops", "n": 30_011, "stops": 41, "days": 120.0},
        # the small parity configuration: 1,000 bodies x 200 one-degree
        # frames over 30 days, what a user runs for one night's fields
        {"name": "fields_small", "kind": "fields", "n": 1000, "frames": 200, "days": 30.0},
        # extended exposures (one hour in 6 sub-frames), squares and cones,
        # with magnitudes
        {"name": "extended_hours", "kind": "extended", "n": 20_000, "frames": 400, "sub": 6,
         "days": 30.0},
        # two months of the WISE-like scan against the whole catalogue, the
        # full-precision survey prediction
        {"name": "wise_two_months", "kind": "wise", "n": 757_000, "days": 60, "mixed": False},
        # three weeks of ZTF-like nights (8x8 sub-fields), mixed precision,
        # with magnitudes
        {"name": "ztf_three_weeks", "kind": "ztf", "n": 250_000, "exposures": 8000, "days": 20},
        # orbit fits of a catalogue: loss, gradient and predictions of 100,000
        # bodies with 20 observations each over 90 days
        {"name": "orbit_fit", "kind": "fit", "n": 100_000, "obs": 20, "days": 90.0},
        # Jacobian rows of a few hundred fits (covariances)
        {"name": "fit_jacobian", "kind": "jacobian", "n": 300, "obs": 20, "days": 90.0},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["ephem", "propagate", "propagate", "clones", "stops", "fields",
                       "extended", "wise", "ztf", "fit", "jacobian"])
    if kind == "ephem":
        return {"kind": kind, "n": _log(rng, 1, 150_000), "body": rng.randrange(9)}
    if kind == "propagate":
        pop = rng.choice(["catalogue", "ragged"])
        # the ragged population's forced encounters need a year's span
        return {"kind": kind, "pop": pop, "n": _log(rng, 1 if pop == "catalogue" else 400, 200_000),
                "days": float(rng.choice([-1, 1]) * _log(rng, 10, 365)) if pop == "catalogue"
                else float(_log(rng, 30, 365)),
                "mixed": rng.random() < 0.4, "nongrav": rng.random() < 0.3}
    if kind == "clones":
        return {"kind": kind, "n": _log(rng, 20, 1000), "days": -float(_log(rng, 300, 2922))}
    if kind == "stops":
        return {"kind": kind, "n": _log(rng, 100, 30_011), "stops": rng.randint(2, 41),
                "days": float(rng.randint(20, 120))}
    if kind == "fields":
        return {"kind": kind, "n": _log(rng, 50, 5000), "frames": _log(rng, 20, 200),
                "days": float(rng.randint(5, 30))}
    if kind == "extended":
        return {"kind": kind, "n": _log(rng, 500, 20_000), "frames": _log(rng, 40, 400),
                "sub": rng.randint(1, 8), "days": 30.0}
    if kind == "wise":
        return {"kind": kind, "n": _log(rng, 10_000, 500_000), "days": rng.randint(3, 60),
                "mixed": rng.random() < 0.3}
    if kind == "ztf":
        return {"kind": kind, "n": _log(rng, 10_000, 250_000), "exposures": _log(rng, 200, 8000),
                "days": rng.randint(3, 20)}
    if kind == "fit":
        return {"kind": kind, "n": _log(rng, 50, 90_000), "obs": rng.randint(3, 31),
                "days": float(rng.randint(30, 90))}
    return {"kind": "jacobian", "n": _log(rng, 10, 300), "obs": rng.randint(3, 31),
            "days": float(rng.randint(30, 90))}


# ---------------------------------------------------------------------------
# what a program keeps: the table, the engine
# ---------------------------------------------------------------------------
@functools.lru_cache(maxsize=None)
def _planets():
    return W.make_planets(W.SEED_BASE)


@functools.lru_cache(maxsize=None)
def _table(span):
    lo, hi = {"year": (-400.0, 460.0), "decade": (-3000.0, 64.0)}[span]
    return W.build_ephemeris(_planets(), W.T0 + lo, W.T0 + hi)


@functools.lru_cache(maxsize=None)
def _engine(span):
    k = kete.Kete(torch.cuda.current_device())
    k.load_ephem(_table(span).to_bytes())
    return k


def _span(case):
    return "decade" if case["kind"] == "clones" else "year"


@functools.lru_cache(maxsize=None)
def _coef(span):
    return torch.from_numpy(_table(span).coef).to(DEV)   # [body, seg, 3, n_coef]


def _planet(span, body, t, vel=False):
    """Chebyshev sums of one table body at epochs t (float64 CUDA [k])."""
    tab, c = _table(span), _coef(span)[body]
    s = torch.floor((t - tab.t_start) / tab.seg_len).clamp(0, tab.n_seg - 1)
    tau = 2.0 * (t - (tab.t_start + (s + 0.5) * tab.seg_len)) / tab.seg_len
    k = torch.arange(tab.n_coef, device=DEV, dtype=F64)
    th = torch.acos(tau.clamp(-1.0, 1.0))
    T = torch.cos(k * th[:, None])
    p = (c[s.long()] * T[:, None, :]).sum(-1)
    if not vel:
        return p
    Um1, U = torch.ones_like(tau), 2.0 * tau     # T_k' = k U_{k-1}
    d = [torch.zeros_like(tau), torch.ones_like(tau)]
    for j in range(2, tab.n_coef):
        d.append(j * U)
        Um1, U = U, 2.0 * tau * U - Um1
    D = torch.stack(d, -1) * (2.0 / tab.seg_len)
    return p, (c[s.long()] * D[:, None, :]).sum(-1)


# ---------------------------------------------------------------------------
# populations (workloads.population's distributions, drawn on the GPU)
# ---------------------------------------------------------------------------
def _gen(seed, stream):
    g = torch.Generator(device=DEV)
    g.manual_seed((int(seed) * 1_000_003 + stream) % (1 << 62))
    return g


def _u(g, n, lo=0.0, hi=1.0):
    return lo + (hi - lo) * torch.rand(n, generator=g, device=DEV, dtype=F64)


def _rayleigh(g, n, scale, cap):
    # the distribution cut at cap, by its inverse
    top = 1.0 - math.exp(-0.5 * (cap / scale) ** 2)
    return scale * torch.sqrt(-2.0 * torch.log1p(-_u(g, n, 0.0, top)))


def _states(a, e, inc, node, peri, M):
    """Heliocentric elliptic elements at T0 -> barycentric states [6, n]."""
    tau = 2.0 * math.pi
    M = torch.remainder(M, tau)
    E = torch.where(e < 0.8, M, torch.full_like(M, math.pi))
    for _ in range(30):
        E = E - (E - e * torch.sin(E) - M) / (1.0 - e * torch.cos(E))
    b = torch.sqrt(1.0 - e * e)
    x, y = a * (torch.cos(E) - e), a * b * torch.sin(E)
    f = math.sqrt(W.GM_SUN) / (torch.sqrt(a) * (1.0 - e * torch.cos(E)))
    vx, vy = -f * torch.sin(E), f * b * torch.cos(E)
    cO, sO, ci, si = torch.cos(node), torch.sin(node), torch.cos(inc), torch.sin(inc)
    cw, sw = torch.cos(peri), torch.sin(peri)
    P = torch.stack([cO * cw - sO * sw * ci, sO * cw + cO * sw * ci, sw * si])
    Q = torch.stack([-cO * sw - sO * cw * ci, -sO * sw + cO * cw * ci, cw * si])
    ps = _planets()
    s0 = torch.from_numpy(np.concatenate([ps.pos0[0], ps.vel0[0]])).to(DEV)
    return (torch.cat([P * x + Q * y, P * vx + Q * vy]) + s0[:, None]).contiguous()


def _elements(kind, n, g):
    deg = math.pi / 180.0
    node, peri, M = (_u(g, n, 0.0, 2.0 * math.pi) for _ in range(3))
    if kind == "main":
        a, e = _u(g, n, 2.1, 3.3), _rayleigh(g, n, 0.08, 0.3)
        inc = _rayleigh(g, n, 8.0, 90.0) * deg
    elif kind == "neo":
        a, e = _u(g, n, 0.8, 2.0), _u(g, n, 0.0, 0.7)
        inc = _rayleigh(g, n, 15.0, 90.0) * deg
    elif kind == "trojan":
        a, e = torch.full((n,), 5.2, device=DEV, dtype=F64), _rayleigh(g, n, 0.05, 0.3)
        inc = _rayleigh(g, n, 10.0, 60.0) * deg
        ps = _planets()
        jp = ps.pos0[5] - ps.pos0[0]
        side = torch.where(_u(g, n) < 0.5, 1.0, -1.0)
        M = math.atan2(jp[1], jp[0]) + (60.0 * side + _u(g, n, -10.0, 10.0)) * deg - node - peri
    else:
        e, q = _u(g, n, 0.7, 0.99), _u(g, n, 0.5, 3.0)
        a, inc = q / (1.0 - e), _rayleigh(g, n, 20.0, 180.0) * deg
    return a, e, inc, node, peri, M


def _forced(n, seed, days):
    """NEOs placed on an Earth passage of 0.001-0.01 AU (workloads.ragged1y)."""
    rng = np.random.default_rng([int(seed) & 0xFFFFFFFF, 5])
    ps = _planets()
    te = np.sort(rng.uniform(min(30.0, 0.5 * days), max(335.0 * days / 365.0, 15.0), n))
    t = torch.from_numpy(W.T0 + te).to(DEV)
    (sp, sv), (ep, ev) = _planet("year", 0, t, True), _planet("year", 3, t, True)
    rel_p, rel_v = (ep - sp).cpu().numpy(), (ev - sv).cpu().numpy()
    out, todo = np.zeros((6, n)), np.arange(n)
    while todo.size:
        m = todo.size
        d = rng.normal(size=(m, 3)); d /= np.linalg.norm(d, axis=1, keepdims=True)
        u = rng.normal(size=(m, 3)); u -= (u * d).sum(1, keepdims=True) * d
        u /= np.linalg.norm(u, axis=1, keepdims=True)
        r = rel_p[todo] + rng.uniform(0.001, 0.01, (m, 1)) * d
        v = rel_v[todo] + rng.uniform(5.0, 20.0, (m, 1)) * 86400.0 / W.AU_KM * u
        with np.errstate(invalid="ignore"):
            a, e, inc, node, peri, M = W.state_to_elements(r.T, v.T, W.GM_SUN)
        ok = (e < 0.95) & (a > 0) & (a * (1 - e) > 0.2)
        M0 = M[ok] - np.sqrt(W.GM_SUN / a[ok] ** 3) * te[todo[ok]]
        p, q = W.elements_to_state(a[ok], e[ok], inc[ok], node[ok], peri[ok], M0, W.GM_SUN)
        out[:3, todo[ok]] = p + ps.pos0[0][:, None]
        out[3:, todo[ok]] = q + ps.vel0[0][:, None]
        todo = todo[~ok]
    return torch.from_numpy(out).to(DEV)


def _population(pop, n, seed, days=365.0):
    """States [6, n] and labels (numpy; 0 main belt, 1 NEO, 2 Trojan, 3 comet,
    4 forced encounter) of a population, grouped as workloads writes them."""
    g = _gen(seed, 2)
    if pop == "catalogue":      # 2 % NEOs
        parts = [("main", n - n // 50), ("neo", n // 50)]
    else:                       # 60 % main belt, 20 % NEO, 10 % Trojan, 10 % comet
        neo = n // 5
        parts = [("main", n - neo - 2 * (n // 10)), ("neo", neo), ("trojan", n // 10),
                 ("comet", n // 10)]
    label = {"main": 0, "neo": 1, "trojan": 2, "comet": 3}
    st, lab = [], []
    for kind, m in parts:
        st.append(_states(*_elements(kind, m, g)))
        lab.append(np.full(m, label[kind], np.int8))
    st, lab = torch.cat(st, 1).contiguous(), np.concatenate(lab)
    n_force = n // 100
    if pop != "catalogue" and n_force:
        first = parts[0][1]
        st[:, first:first + n_force] = _forced(n_force, seed, days)
        lab[first:first + n_force] = 4
    return st, lab


# ---------------------------------------------------------------------------
# frames and observations
# ---------------------------------------------------------------------------
def _epochs(n):
    return torch.full((n,), W.T0, device=DEV, dtype=F64)


def _square_frames(ep, obs_idx, exposure, centre, width, cones=None):
    """CUDA bytes of square kete_frame records (cones[i]: a cone instead)."""
    c = centre / centre.norm(dim=1, keepdim=True)
    ref = torch.zeros_like(c)
    ref[:, 2] = 1.0
    e = torch.linalg.cross(ref, c)
    e = e / e.norm(dim=1, keepdim=True)
    nn = torch.linalg.cross(c, e)
    s, q = math.sin(width / 2.0), math.cos(width / 2.0)
    m = torch.cat([c * s - e * q, c * s - nn * q, c * s + e * q, c * s + nn * q], 1)
    f = torch.zeros((ep.numel(), 16), device=DEV, dtype=F64)
    i = f.view(torch.int64)
    f[:, 0] = ep
    i[:, 1], i[:, 2], i[:, 3] = obs_idx, exposure, 4
    f[:, 4:] = m
    if cones is not None:
        i[cones, 3] = 0
        f[cones, 4:] = 0.0
        f[cones, 4:7] = c[cones]
        f[cones, 7] = width / 2.0
    return f.view(torch.uint8).reshape(-1).contiguous()


def _aim(states, body, t, obs, span="year"):
    """Directions from obs to bodies on their heliocentric conics at epochs t."""
    ps = _planets()
    hr = states[:3, body].T - torch.from_numpy(ps.pos0[0]).to(DEV)
    hv = states[3:, body].T - torch.from_numpy(ps.vel0[0]).to(DEV)
    r, _ = _two_body(hr, hv, t - W.T0, steps=24)
    d = r + _planet(span, 0, t) - obs
    return d / d.norm(dim=1, keepdim=True)


def _scan_frames(case, seed, sub=0):
    """Frames over the span, half aimed near bodies, seen from the Earth."""
    n, nf, days = case["n"], case["frames"], case["days"]
    states, labels = _population("catalogue", n, seed)
    g = _gen(seed, 3)
    if sub:     # one-hour exposures that do not overlap in time
        gap = days / nf
        dur = min(1.0 / 24.0, 0.8 * gap)
        ep = W.T0 + gap * (torch.arange(nf, device=DEV, dtype=F64) + _u(g, nf, 0.0, 0.19))
        mid = ep + 0.5 * dur
        k = (torch.arange(sub, device=DEV, dtype=F64) + 0.5) * dur / sub
        obs = _planet("year", 3, (ep[:, None] + k).reshape(-1)).contiguous()
        durations = torch.full((nf,), dur, device=DEV, dtype=F64)
    else:
        ep = torch.sort(W.T0 + _u(g, nf, 0.0, days)).values
        mid, durations = ep, None
        obs = _planet("year", 3, ep).contiguous()
    at = _planet("year", 3, mid)
    z = _u(g, nf, -0.5, 0.5)
    lon = _u(g, nf, 0.0, 2.0 * math.pi)
    cen = torch.stack([torch.sqrt(1 - z * z) * torch.cos(lon),
                       torch.sqrt(1 - z * z) * torch.sin(lon), z], 1)
    at_body = torch.randperm(nf, generator=g, device=DEV)[:nf // 2]
    body = torch.randint(0, n, (nf // 2,), generator=g, device=DEV)
    jit = math.radians(0.2) * torch.randn(nf // 2, 3, generator=g, device=DEV, dtype=F64)
    cen[at_body] = _aim(states, body, mid[at_body], at[at_body]) + jit
    cones = torch.arange(nf, device=DEV) % 3 == 2 if sub else None
    f = _square_frames(ep, torch.arange(nf, device=DEV) * max(1, sub),
                       torch.arange(nf, device=DEV), cen, math.radians(1.0), cones)
    return states, labels, f, obs, durations


def _observations(case, seed):
    """Truth states, fit states and observation records of an orbit fit: the
    circular 1-AU observer of the scanning survey, 0.1 arcsec noise."""
    n, m, days = case["n"], case["obs"], case["days"]
    states, _ = _population("catalogue", n, seed)
    g = _gen(seed, 6)
    ep = torch.sort(_u(g, n * m, 0.0, days).reshape(n, m), 1).values + W.T0
    th = 0.3 + W.GAUSS_K * (ep - W.T0)
    sun = _planet("year", 0, ep.reshape(-1)).reshape(n, m, 3)
    obs = torch.zeros((n, m, 6), device=DEV, dtype=F64)
    obs[..., 0] = ep
    obs[..., 3:] = sun + torch.stack([torch.cos(th), torch.sin(th), torch.zeros_like(th)], -1)
    noise = math.radians(0.1 / 3600.0) * torch.randn(n, m, 2, generator=g, device=DEV, dtype=F64)
    off = torch.randn(6, n, generator=g, device=DEV, dtype=F64)
    off[:3] *= 1e-6
    off[3:] *= 1e-8
    ra, dec = _predict(states, obs, days)
    obs[..., 1] = ra + noise[..., 0] / torch.cos(dec)
    obs[..., 2] = dec + noise[..., 1]
    return (states + off).contiguous(), obs.contiguous()


# ---------------------------------------------------------------------------
# prepare and run
# ---------------------------------------------------------------------------
def _nongrav(labels, seed):
    return kete.nongrav_to_device(
        W.nongrav_params(np.where(labels == 4, 1, labels), seed=W.SEED_BASE + int(seed) % 997), DEV)


def prepare(case, seed):
    kind, span = case["kind"], _span(case)
    s = {"kind": kind, "k": _engine(span), "case": case}
    if kind == "ephem":
        g = _gen(seed, 1)
        s["t"] = torch.sort(W.T0 + _u(g, case["n"], 0.0, 365.0)).values.contiguous()
    elif kind == "propagate":
        s["states"], labels = _population(case["pop"], case["n"], seed, abs(case["days"]))
        s["fm"] = kete.force_model(
            precision=kete.MIXED if case["mixed"] else kete.FP64,
            nongrav=_nongrav(labels, seed) if case["nongrav"] else None)
    elif kind == "clones":
        el = W.CLONE_ELEMENTS
        d = math.radians
        one = lambda x: torch.full((1,), float(x), device=DEV, dtype=F64)  # noqa: E731
        nominal = _states(one(el["a"]), one(el["e"]), one(d(el["inc"])), one(d(el["node"])),
                          one(d(el["peri"])), one(el["M"]))
        g = _gen(seed, 12)
        off = torch.randn(6, case["n"], generator=g, device=DEV, dtype=F64)
        off[:3] *= 1e-6
        off[3:] *= 1e-8
        s["states"] = (nominal + off).contiguous()
        ng = torch.zeros((case["n"], 10), device=DEV, dtype=F64)
        scat = 1.0 + 0.05 * torch.randn(2, case["n"], generator=g, device=DEV, dtype=F64)
        ng[:, 0], ng[:, 1] = 1e-8 * scat[0], 5e-10 * scat[1]
        ng[:, 3], ng[:, 4], ng[:, 5], ng[:, 6], ng[:, 7] = 0.1112620426, 2.808, 2.15, 5.093, 4.6142
        s["fm"] = kete.force_model(nongrav=ng)
    elif kind == "stops":
        s["states"], _ = _population("catalogue", case["n"], seed)
        rng = np.random.default_rng([int(seed) & 0xFFFFFFFF, 7])
        k, gap = case["stops"], case["days"] / case["stops"]
        s["stops"] = W.T0 + gap * (np.arange(k) + rng.uniform(0.1, 0.9, k))
        s["fm"] = kete.force_model()
    elif kind in ("fields", "extended"):
        sub = case.get("sub", 0)
        s["states"], labels, s["frames"], s["obs"], s["dur"] = _scan_frames(case, seed, sub)
        s["mag"] = kete.mag_params_to_device(W.mag_params(labels), DEV) if sub else None
        s["cap"] = max(4096, 64 * case["frames"])
        s["fm"] = kete.force_model()
    elif kind in ("wise", "ztf"):
        s["states"], labels = _population("catalogue", case["n"], seed)
        if kind == "wise":
            fr, obs = _wise(case["days"])
            s["cap"] = int(16 * fr.numel() // 128 * max(0.1, case["n"] / 757_000)) + 4096
            s["mag"] = None
            mixed = case["mixed"]
        else:
            rng = np.random.default_rng([int(seed) & 0xFFFFFFFF, 3])
            f, o, _, _ = W.ztf_frames(_planets(), case["exposures"], case["days"], seed_rng=rng)
            fr, obs = kete.frames_to_device(f, DEV), torch.from_numpy(np.ascontiguousarray(o)).to(DEV)
            s["cap"] = int(24 * fr.numel() // 128 * max(0.1, case["n"] / 757_000)) + 4096
            s["mag"] = kete.mag_params_to_device(W.mag_params(labels), DEV)
            mixed = True
        s["frames"], s["obs"] = fr, obs
        s["fm"] = kete.force_model(precision=kete.MIXED if mixed else kete.FP64)
    else:
        s["states"], s["obs"] = _observations(case, seed)
        s["fm"] = kete.force_model()
        s["opts"] = kete.survey_opts(mem_budget_gb=24.0)
    if "states" in s:
        s["epochs"] = _epochs(s["states"].shape[1])
    if "cap" in s:
        s["hits"] = torch.full((s["cap"], 4), -1, dtype=torch.int64, device=DEV)
    return s


@functools.lru_cache(maxsize=4)
def _wise(days):
    """The scanning survey's first `days` days: its plan, the same for any catalogue."""
    f, o, _, _ = W.wise_frames(_planets(), 3288 * days, days)
    return kete.frames_to_device(f, DEV), torch.from_numpy(np.ascontiguousarray(o)).to(DEV)


def _hits(h, n, status):
    """The user's hit buffer by column: rows past n_hits stay as prepare left them."""
    return {"n_hits": n, "frame": h[:, 0], "body": h.view(torch.int32)[:, 2],
            "mag": h.view(torch.float32)[:, 3], "ra": h.view(F64)[:, 2], "dec": h.view(F64)[:, 3],
            "status": status}


def run(s):
    k, kind = s["k"], s["kind"]
    if kind == "ephem":
        return k.ephem_eval(s["t"], s["case"]["body"])
    if kind in ("propagate", "clones"):
        st, ep = s["states"].clone(), s["epochs"].clone()   # the catalogue stays
        status = k.propagate(st, ep, W.T0 + s["case"]["days"], fm=s["fm"])
        return {"states": st, "epochs": ep, "status": status}
    if kind == "stops":
        out, status = k.propagate_stops(s["states"], s["epochs"], s["stops"], fm=s["fm"])
        return {"states": out, "status": status}
    if kind == "extended":
        return _hits(*k.fov_check_extended(s["states"], s["epochs"], s["frames"], s["dur"],
                                           s["case"]["sub"], s["obs"], fm=s["fm"], hits=s["hits"],
                                           mag_params=s["mag"]))
    if kind in ("fields", "wise", "ztf"):
        return _hits(*k.fov_check(s["states"], s["epochs"], s["frames"], s["obs"], fm=s["fm"],
                                  hits=s["hits"], mag_params=s["mag"]))
    if kind == "fit":
        loss, grad, pred, status = k.adjoint(s["states"], s["epochs"], s["obs"], fm=s["fm"],
                                             opts=s["opts"], ckpt_days=8.0, pred=True)
        return {"loss": loss, "grad": grad, "pred": pred, "status": status}
    jac, pred, status = k.sky_jacobian(s["states"], s["epochs"], s["obs"], fm=s["fm"],
                                       opts=s["opts"], ckpt_days=8.0, pred=True)
    return {"jac": jac, "pred": pred, "status": status}


# ---------------------------------------------------------------------------
# work: inputs read once, outputs written once; FLOPs of the natural method
# ---------------------------------------------------------------------------
# A main-belt body's Gauss-Radau step is ~16 days of 22 force evaluations with
# ~330 FP64 operations each and ~4,400 of the corrector (bench.py's counts):
# ~730 a body-day; NEOs and comets step more often.
_PER_DAY = {"catalogue": 800.0, "ragged": 1200.0}


def work(case):
    kind, n = case["kind"], case["n"]
    if kind == "ephem":
        return {"bytes": n * 56.0, "flops": n * 145.0}
    if kind in ("propagate", "clones"):
        per = _PER_DAY[case["pop"]] if kind == "propagate" else 900.0
        extra = 80.0 * n if kind == "clones" or case["nongrav"] else 0.0
        return {"bytes": n * (56.0 + 56.0 + 4.0) + extra, "flops": n * abs(case["days"]) * per}
    if kind == "stops":
        return {"bytes": n * (60.0 + 48.0 * case["stops"]), "flops": n * case["days"] * 800.0}
    if kind in ("fields", "extended"):
        sub = case.get("sub", 1)
        return {"bytes": n * 60.0 + case["frames"] * (128.0 + 24.0 * sub),
                "flops": n * case["days"] * 800.0}
    if kind == "wise":     # ~7.1 hits per frame and 757,000 bodies, 835 operations each
        nf = 3288.0 * case["days"]
        hits = 7.1 * nf * n / 757_000.0
        return {"bytes": n * 60.0 + nf * 152.0 + 32.0 * hits,
                "flops": n * case["days"] * 800.0 + 835.0 * hits}
    if kind == "ztf":      # ~11.1 hits per sub-field and 757,000 bodies
        nf = 64.0 * case["exposures"]
        hits = 11.1 * nf * n / 757_000.0
        return {"bytes": n * 84.0 + nf * 128.0 + 32.0 * hits,
                "flops": n * case["days"] * 400.0 + 835.0 * hits}
    m = case["obs"]
    out = 60.0 + 16.0 * m if kind == "fit" else 112.0 * m
    return {"bytes": n * (60.0 + 48.0 * m + out),
            "flops": n * case["days"] * 1600.0 + n * m * 3000.0}


# ---------------------------------------------------------------------------
# an independent FP64 model: Gauss-Legendre collocation in plain torch
# ---------------------------------------------------------------------------
_S = 12


@functools.lru_cache(maxsize=None)
def _gauss():
    """Nodes on [0, 1], the matrix from values at the nodes to Legendre
    coefficients, and a function giving the weights of the first and second
    integrals from 0 to s in those coefficients (the double integral's
    weight is int_0^s (s - q) a(q) dq)."""
    x, w = np.polynomial.legendre.leggauss(_S)
    P = np.polynomial.legendre.legvander(x, _S - 1)
    C = (2.0 * np.arange(_S) + 1.0)[:, None] / 2.0 * (P * w[:, None]).T
    return 0.5 * (x + 1.0), C


def _integrals(s):
    """(I1, I2)[..., j] of Legendre polynomial j (argument 2 q - 1) from 0 to s."""
    u = 2.0 * s - 1.0
    lib = torch if isinstance(s, torch.Tensor) else np
    p = [lib.ones_like(u), u]
    for j in range(2, _S + 2):
        p.append(((2 * j - 1) * u * p[-1] - (j - 1) * p[-2]) / j)
    # int_{-1}^{u} P_j = (P_{j+1} - P_{j-1}) / (2 j + 1), once more for the second
    f1 = [u + 1.0] + [(p[j + 1] - p[j - 1]) / (2 * j + 1) for j in range(1, _S + 1)]
    f2 = [0.5 * (u + 1.0) ** 2] + [(f1[j + 1] - f1[j - 1]) / (2 * j + 1) for j in range(1, _S)]
    return lib.stack(f1[:_S], -1) * 0.5, lib.stack(f2, -1) * 0.25


def _poles():
    fm = kete.force_model()
    ce, se = math.cos(W.OBLIQUITY), math.sin(W.OBLIQUITY)
    out = {}
    for b in (0, 5):
        ra, de = fm.pole_ra[b], fm.pole_dec[b]
        e = (math.cos(de) * math.cos(ra), math.cos(de) * math.sin(ra), math.sin(de))
        pole = (e[0], ce * e[1] + se * e[2], -se * e[1] + ce * e[2])
        out[b] = (1.5 * fm.j2[b] * fm.radius[b] ** 2, pole)
    return out


def _accel(x, v, pl, ng):
    """Eq. A.1 at x, v [s, n, 3]; pl[body] = (position, velocity) [s, 1, 3]."""
    c2 = (299792.458 * 86400.0 / W.AU_KM) ** 2
    poles = _poles()
    a = torch.zeros_like(x)
    for b in range(9):
        mu = W.GM[b]
        r = x - pl[b][0]
        rr = (r * r).sum(-1, keepdim=True)
        i1 = torch.rsqrt(rr)
        i3 = i1 / rr
        f = -mu * i3
        if b in (0, 3, 5):
            w = v - pl[b][1]
            k = (mu / c2) * i3
            f = f + k * (4.0 * mu * i1 - (w * w).sum(-1, keepdim=True))
            a = a + 4.0 * k * (r * w).sum(-1, keepdim=True) * w
        if b in poles:
            j, p = poles[b]
            p = torch.tensor(p, device=DEV, dtype=F64)
            z = (r * p).sum(-1, keepdim=True)
            psi = j * mu * i3 / rr
            f = f - psi * (1.0 - 5.0 * z * z / rr)
            a = a - 2.0 * psi * z * p
        a = a + f * r
        if b == 0:
            hr, hi = r, i1
    if ng is not None:      # JPL comet model without lag
        w = v - pl[0][1]
        a1, a2, a3, al, r0, m, q, k = (ng[:, i][:, None] for i in range(8))
        u = 1.0 / (hi * r0)
        gr = al * u ** (-m) * (1.0 + u ** q) ** (-k)
        h = torch.linalg.cross(hr, w)
        nh = h / h.norm(dim=-1, keepdim=True)
        rh = hr * hi
        a = a + gr * (a1 * rh + a2 * torch.linalg.cross(nh, rh) + a3 * nh)
    return a


def _integrate(states, t_a, marks, h_max, span, ng=None, dense=None):
    """States [6, n] from t_a through the epochs `marks` (in order): the list of
    states at the marks.  dense: a list that receives every step as
    (t, h, x0, v0, a at the nodes)."""
    c, C = _gauss()
    I1, I2 = _integrals(c)
    node = torch.from_numpy(c).to(DEV)
    cs = node[:, None, None]
    A1 = torch.from_numpy(I1 @ C).to(DEV)       # velocities at the nodes
    A2 = torch.from_numpy(I2 @ C).to(DEV)       # positions at the nodes
    e1, e2 = _integrals(np.ones(1))
    b1, b2 = (torch.from_numpy((e[0] @ C)).to(DEV) for e in (e1, e2))
    x, v = states[:3].T.contiguous(), states[3:].T.contiguous()
    n = x.shape[0]
    out, t = [], float(t_a)
    a_end = None
    for mark in marks:
        k = max(1, int(math.ceil(abs(mark - t) / h_max - 1e-9)))
        t0, hs = t, (mark - t) / k
        for j in range(k):
            ta = t0 + j * hs
            tb = mark if j == k - 1 else t0 + (j + 1) * hs
            h = tb - ta
            pl = [tuple(y[:, None, :] for y in _planet(span, b, ta + node * h, True))
                  for b in range(9)]
            F = (a_end if a_end is not None else torch.zeros_like(x)).expand(_S, n, 3)
            last = None
            for it in range(12):
                m = F.reshape(_S, -1)
                X = x + cs * h * v + h * h * (A2 @ m).reshape(_S, n, 3)
                V = v + h * (A1 @ m).reshape(_S, n, 3)
                F = _accel(X, V, pl, ng)
                if it >= 4 and it % 2 == 0:
                    if last is not None and bool((X - last).abs().max() < 2e-15):
                        break
                last = X
            m = F.reshape(_S, -1)
            if dense is not None:
                dense.append((ta, h, x, v, F))
            x = x + h * v + h * h * (b2 @ m).reshape(n, 3)
            v = v + h * (b1 @ m).reshape(n, 3)
            a_end = F[-1]
        t = float(mark)
        out.append(torch.cat([x.T, v.T]))
    return out


def _dense_at(dense, t, rows):
    """States [k, 6] of bodies `rows` [k] at epochs t [k] from the steps."""
    _, C = _gauss()
    Cm = torch.from_numpy(C).to(DEV)
    out = torch.empty((t.numel(), 6), device=DEV, dtype=F64)
    for i, (ta, h, x, v, F) in enumerate(dense):
        last = i == len(dense) - 1
        sel = torch.nonzero(((t >= ta) | (i == 0)) & ((t < ta + h) | last)).reshape(-1)
        if not sel.numel():
            continue
        s = (t[sel] - ta) / h
        I1, I2 = _integrals(s)
        w1, w2 = I1 @ Cm, I2 @ Cm
        b = rows[sel]
        for a in range(0, sel.numel(), 1 << 20):
            q = slice(a, a + (1 << 20))
            Fb = F[:, b[q]]
            out[sel[q], :3] = (x[b[q]] + (s[q] * h)[:, None] * v[b[q]]
                               + h * h * torch.einsum("ks,skc->kc", w2[q], Fb))
            out[sel[q], 3:] = v[b[q]] + h * torch.einsum("ks,skc->kc", w1[q], Fb)
    return out


def _two_body(r0, v0, dt, steps=1):
    """Heliocentric states [k, 3] advanced by dt [k] (universal variables, the
    Stumpff series; long intervals in `steps` pieces)."""
    mu, sq = W.GM_SUN, W.GAUSS_K
    d = dt / steps
    for _ in range(steps):
        rn = r0.norm(dim=1)
        al = 2.0 / rn - (v0 * v0).sum(1) / mu
        A, B = (r0 * v0).sum(1) / sq, 1.0 - al * rn
        chi = sq * d / rn
        for _ in range(9):
            C, S, z = _stumpff(al, chi)
            f = A * chi ** 2 * C + B * chi ** 3 * S + rn * chi - sq * d
            df = A * chi * (1.0 - z * S) + B * chi ** 2 * C + rn
            chi = chi - f / df
        C, S, z = _stumpff(al, chi)
        ff, gg = 1.0 - chi ** 2 * C / rn, d - chi ** 3 * S / sq
        r = ff[:, None] * r0 + gg[:, None] * v0
        rm = r.norm(dim=1)
        fd, gd = sq / (rm * rn) * chi * (z * S - 1.0), 1.0 - chi ** 2 * C / rm
        r0, v0 = r, fd[:, None] * r0 + gd[:, None] * v0
    return r0, v0


def _stumpff(al, chi):
    z = al * chi * chi
    c, s = torch.zeros_like(z), torch.zeros_like(z)
    for k in range(12, -1, -1):
        c = c * -z + 1.0 / math.factorial(2 * k + 2)
        s = s * -z + 1.0 / math.factorial(2 * k + 3)
    return c, s, z


def _apparent(y, t_ref, t_obs, obs, span="year"):
    """Apparent direction vectors [k, 3] of states y [k, 6] at t_ref: two-body
    to t_obs - tau, three light-time iterations."""
    sun, vs = _planet(span, 0, t_ref, True)
    hr, hv = y[:, :3] - sun, y[:, 3:] - vs
    ic = W.AU_KM / (299792.458 * 86400.0)
    tau = torch.zeros_like(t_obs)
    for it in range(5):
        r, _ = _two_body(hr, hv, (t_obs - t_ref) - tau)
        u = r + _planet_off(span, t_obs, -tau) - obs
        if it < 4:
            tau = u.norm(dim=1) * ic
    return u


def _planet_off(span, t, off):
    """The Sun at t + off, the small offset kept out of the absolute epoch."""
    p, v = _planet(span, 0, t, True)
    return p + off[:, None] * v


def _radec(u):
    ce, se = math.cos(W.OBLIQUITY), math.sin(W.OBLIQUITY)
    x, y, z = u[:, 0], ce * u[:, 1] - se * u[:, 2], se * u[:, 1] + ce * u[:, 2]
    ra = torch.atan2(y, x)
    return torch.where(ra < 0, ra + 2.0 * math.pi, ra), torch.atan2(z, torch.sqrt(x * x + y * y))


def _midpoints(ep):
    """Batch midpoint of every observation: batches of epochs within 3 days of
    their first [n, m]."""
    first, ref = ep[:, 0].clone(), torch.empty_like(ep)
    start = torch.zeros_like(ep)
    for j in range(ep.shape[1]):
        new = ~((ep[:, j] == first) | (ep[:, j] - first < 3.0))
        first = torch.where(new, ep[:, j], first)
        start[:, j] = first
    end = ep[:, -1].clone()
    for j in range(ep.shape[1] - 1, -1, -1):
        if j + 1 < ep.shape[1]:
            end = torch.where(start[:, j + 1] != start[:, j], ep[:, j], end)
        ref[:, j] = 0.5 * (start[:, j] + end)
    return ref


def _predict(states, obs, days):
    """RA, Dec [n, m] of every observation record, from states [6, n] at T0."""
    n, m = obs.shape[:2]
    ref = _midpoints(obs[..., 0].contiguous()).reshape(-1)
    ra, dec = (torch.empty(n * m, device=DEV, dtype=F64) for _ in range(2))
    flat = obs.reshape(n * m, 6)
    for a in range(0, n, 50_000):
        b = min(n, a + 50_000)
        dense = []
        _integrate(states[:, a:b].contiguous(), W.T0, [W.T0 + days], 5.0, "year", dense=dense)
        q = slice(a * m, b * m)
        rows = torch.arange(b - a, device=DEV).repeat_interleave(m)
        y = _dense_at(dense, ref[q].contiguous(), rows)
        ra[q], dec[q] = _radec(_apparent(y, ref[q], flat[q, 0], flat[q, 3:]))
    return ra.reshape(n, m), dec.reshape(n, m)


def exact(case, seed):
    kind = case["kind"]
    if kind in ("wise", "ztf", "extended"):
        return None     # hit lists of millions of pairs
    s = prepare(case, seed)
    if kind == "ephem":
        p, v = _planet("year", case["body"], s["t"], True)
        return p, v
    if kind == "propagate":
        # forced passages and thermal lags need an adaptive integration
        if case["pop"] != "catalogue" or case["nongrav"] or case["n"] > 20_000:
            return None
        y = _integrate(s["states"], W.T0, [W.T0 + case["days"]], 1.0, "year")[0]
        return {"states": y, "epochs": s["epochs"] + case["days"], "status": None}
    if kind == "clones":
        ng = s["fm"]._nongrav
        y = _integrate(s["states"], W.T0, [W.T0 + case["days"]], 4.0, "decade", ng=ng)[0]
        return {"states": y, "epochs": s["epochs"] + case["days"], "status": None}
    if kind == "stops":
        y = _integrate(s["states"], W.T0, list(s["stops"]), 2.0, "year")
        return {"states": torch.stack(y), "status": None}
    if kind == "fields":
        return _exact_fields(s)
    ra, dec = _predict(s["states"], s["obs"], case["days"])
    pred = torch.stack([ra, dec], -1)
    if kind == "fit":
        o = s["obs"]
        d = torch.remainder(ra - o[..., 1] + math.pi, 2.0 * math.pi) - math.pi
        loss = ((d * torch.cos(o[..., 2])) ** 2 + (dec - o[..., 2]) ** 2).sum(1)
        return {"loss": loss, "grad": None, "pred": pred, "status": None}
    n, m = s["obs"].shape[:2]
    jac = torch.empty((n, m, 2, 6), device=DEV, dtype=F64)
    for c in range(6):
        e = 3e-5 if c < 3 else 3e-7
        pm = []
        for q in (e, -e, 2 * e, -2 * e):      # fourth-order central difference
            y = s["states"].clone()
            y[c] += q
            r, d = _predict(y, s["obs"], case["days"])
            pm.append(torch.stack([torch.remainder(r - ra + math.pi, 2 * math.pi) - math.pi, d - dec], -1))
        jac[..., c] = (8.0 * (pm[0] - pm[1]) - (pm[2] - pm[3])) / (12.0 * e)
    return {"jac": jac, "pred": pred, "status": None}


def _exact_fields(s):
    """Brute force: every body against every frame of the list."""
    f = s["frames"].view(F64).reshape(-1, 16)
    ep, nrm = f[:, 0], f[:, 4:].reshape(-1, 4, 3)
    t = ep.cpu().numpy()
    ref, a = np.empty_like(t), 0
    while a < len(t):
        b = a
        while b + 1 < len(t) and (t[b + 1] == t[a] or t[b + 1] - t[a] < 3.0):
            b += 1
        ref[a:b + 1] = 0.5 * (t[a] + t[b])
        a = b + 1
    marks = sorted(set(ref.tolist()))
    ys = dict(zip(marks, _integrate(s["states"], W.T0, marks, 2.0, "year")))
    n = s["states"].shape[1]
    hit = {"frame": [], "body": [], "ra": [], "dec": []}
    for i in range(len(t)):
        y = ys[float(ref[i])].T
        one = torch.ones(n, device=DEV, dtype=F64)
        u = _apparent(y, ref[i] * one, t[i] * one, s["obs"][i].expand(n, 3))
        b = torch.nonzero(((u @ nrm[i].T) > 0).all(1)).reshape(-1)
        r, d = _radec(u[b])
        for key, val in (("frame", torch.full_like(b, i)), ("body", b), ("ra", r), ("dec", d)):
            hit[key].append(val)
    out = {key: torch.cat(v) for key, v in hit.items()}
    rest = s["cap"] - out["ra"].numel()     # the buffer's unused rows hold no number
    ra, dec = (torch.cat([out[key], torch.full((rest,), math.nan, device=DEV, dtype=F64)])
               for key in ("ra", "dec"))
    return {"n_hits": None, "frame": None, "body": None, "mag": None, "ra": ra, "dec": dec,
            "status": None}
