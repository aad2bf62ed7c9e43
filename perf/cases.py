"""The work that users of this framework have it do, as cases to be measured.

A case is a batch of synthetic events of one size and occupancy, taken through
one of the public calls: the direct calls on device buffers (seeding_run,
matching_run, ut_run), a captured graph of a batch, the allocation-free entry
point, matching alone, or the serving pipeline on host buffers.
"""

import math
from functools import lru_cache

import numpy as np
import torch

from paper_2606_14480_gb300 import st

# ---------------------------------------------------------------------------
# cases
# ---------------------------------------------------------------------------


def _case(call, events, tracks=150.0, spread=0.0, noise=0.3, ghosts=0.2, method="hlt1", ut=False, final=False,
          check=False, requests=1):
    """tracks: Poisson mean per event, or with spread > 0 the median of a
    log-normal clipped to [5, 800].  method: hlt1 (two independent iterations,
    iterative UV), hough (Hough-cluster UV) or hlt2 (three iterations in
    sequence).  final: ghost network and clone removal.  ut: UT hits of the
    Long tracks.  check: hits given with their z and stereo slope."""
    return {"call": call, "events": events, "tracks": tracks, "spread": spread, "noise": noise, "ghosts": ghosts,
            "method": method, "ut": ut, "final": final, "check": check, "requests": requests}


def listed():
    return [
        # one event as it arrives, by the plain calls: what a monitoring job
        # or a program without batching does
        dict(_case("direct", 1), name="one_event"),
        # a handful of events of ragged number with everything a Long track gets
        dict(_case("direct", 13, tracks=90.0, ut=True), name="small_ut"),
        # a short batch replayed as a graph: a low-latency trigger node
        dict(_case("graph", 67), name="graph_67"),
        # the Run-3-like batch of about 1000 events, the usual batch of a trigger node
        dict(_case("graph", 1000), name="graph_run3"),
        # real occupancies: a log-normal mix from nearly empty to 12 000 hits an event
        dict(_case("graph", 2000, tracks=120.0, spread=0.65), name="graph_uneven"),
        # the same calls without a graph, on a batch that is not round
        dict(_case("direct", 301, noise=0.25), name="direct_301"),
        # Hough-cluster UV seeding
        dict(_case("graph", 250, method="hough"), name="hough_250"),
        # iterations in sequence with hit cleanup, as an offline-like second level runs them
        dict(_case("direct", 250, method="hlt2"), name="hlt2_250"),
        # matching alone in dense VELO environments (400 segments an event)
        dict(_case("match", 500, tracks=280.0, noise=0.4, ghosts=0.4286), name="match_dense"),
        # Long tracks to the end: matching, ghost network, clone removal, UT hits
        dict(_case("match", 1000, ut=True, final=True), name="long_final"),
        # seeding where nothing may be allocated, hits given with their geometry
        dict(_case("static", 100, check=True), name="static_100"),
        # served: requests of a few to many hundred events, in flight together, from pinned host memory
        dict(_case("serve", 1500, requests=6), name="serve_mix"),
    ]


def draw(rng):
    call = rng.choice(["direct", "direct", "graph", "graph", "match", "static", "serve"])
    tracks = math.exp(rng.uniform(math.log(20.0), math.log(280.0)))
    most = {"direct": 600, "graph": 1400, "match": 900, "static": 100, "serve": 1200}[call]
    most = max(2, int(most * min(1.0, (120.0 / tracks) ** 1.5)))
    events = int(math.exp(rng.uniform(0.0, math.log(most + 1))))
    method = rng.choice(["hlt1", "hlt1", "hough", "hlt2"]) if call in ("direct", "graph") else "hlt1"
    return _case(call, events, tracks=round(tracks, 1), spread=rng.choice([0.0, 0.0, 0.5]) if call != "static" else 0.0,
                 noise=round(rng.uniform(0.1, 0.5), 2), ghosts=round(rng.uniform(0.0, 0.45), 2), method=method,
                 ut=call in ("direct", "match") and rng.random() < 0.4, final=call == "match" and rng.random() < 0.4,
                 check=call in ("direct", "static") and rng.random() < 0.3,
                 requests=min(events, rng.randint(1, 8)) if call == "serve" else 1)


# ---------------------------------------------------------------------------
# events: the toy detector of the benchmark (12 SciFi layers x-u-v-x, a kink
# magnet, VELO and UT in front of it)
# ---------------------------------------------------------------------------

T5 = math.tan(math.radians(5.0))
Z = [7826.0, 7896.0, 7966.0, 8036.0, 8508.0, 8578.0, 8648.0, 8718.0, 9193.0, 9263.0, 9333.0, 9403.0]
SLOPE = [0.0, T5, -T5, 0.0] * 3
Z_REF, D_RATIO, Z_VELO, Z_KINK, KAPPA = 8520.0, -2.6e-4, 770.0, 5200.0, 1.0e-2
UT_Z, UT_SLOPE = [2327.5, 2372.5, 2597.5, 2642.5], [0.0, T5, -T5, 0.0]
UT_GAMMA = (7.707063e-11, -7.817364e-3)
ZMX = [5156.02066, 0.0, 0.0, 0.0, 0.0]  # the kink position fitted on this detector


def _tracks(n, g, dev):
    """n tracks inside the detector: slopes, momentum, the x-z model downstream."""
    z = torch.tensor(Z, dtype=torch.float64, device=dev)
    slope = torch.tensor(SLOPE, dtype=torch.float64, device=dev)
    dz = z - Z_REF
    f = dz * dz * (1.0 + D_RATIO * dz)
    got, have = [], 0
    while have < n:
        r = torch.rand(4, max(1024, 3 * (n - have)), generator=g, device=dev, dtype=torch.float64)
        p = 2.0 * 50.0 ** r[0]
        q = torch.where(r[1] < 0.5, -1.0, 1.0).double()
        tx, ty = 0.6 * r[2] - 0.3, 0.5 * r[3] - 0.25
        b = tx + 1.2 * q / p
        a = tx * Z_KINK + b * (Z_REF - Z_KINK)
        c = KAPPA * q / (1000.0 * p)
        x = a[:, None] + b[:, None] * dz + c[:, None] * f
        y = ty[:, None] * z
        xh = x - y * slope
        ok = (b.abs() < 0.3) & (x.abs() < 3200.0).all(1) & (y.abs() < 2500.0).all(1) & (xh.abs() < 3200.0).all(1)
        got.append(torch.cat([torch.stack([p, q, tx, ty], 1), xh], 1)[ok])
        have += got[-1].shape[0]
    t = torch.cat(got)[:n]
    return t[:, 0], t[:, 1], t[:, 2], t[:, 3], t[:, 4:]


def _by_event(ev, n_events, g, *arrays):
    """The arrays sorted by event and shuffled inside each, and the offsets."""
    key = torch.rand(ev.shape[0], generator=g, device=ev.device, dtype=torch.float64)
    order = torch.argsort(ev.double() + key)
    off = torch.zeros(n_events + 1, dtype=torch.int64, device=ev.device)
    off[1:] = torch.cumsum(torch.bincount(ev, minlength=n_events), 0)
    return [off] + [a[order] for a in arrays]


def make_events(case, seed):
    """Hits, VELO segments and UT hits of the case's events (device tensors, CSR per event)."""
    dev = torch.device("cuda")
    g = torch.Generator(device=dev)
    g.manual_seed(int(seed))
    E = case["events"]
    if case["spread"] > 0:
        nt = torch.randn(E, generator=g, device=dev, dtype=torch.float64) * case["spread"] + math.log(case["tracks"])
        nt = nt.exp().round().clamp(5, 800).long()
    else:
        nt = torch.poisson(torch.full((E,), case["tracks"], device=dev, dtype=torch.float64), generator=g).long()
    T = int(nt.sum())
    trk_ev = torch.repeat_interleave(torch.arange(E, device=dev), nt)
    p, q, tx, ty, xh = _tracks(T, g, dev)

    def rand(*s):
        return torch.rand(*s, generator=g, device=dev, dtype=torch.float64)

    def normal(*s):
        return torch.randn(*s, generator=g, device=dev, dtype=torch.float64)

    def noise_of(ev):
        n = torch.bincount(ev, minlength=E).double().mul(case["noise"]).round().long()
        return torch.repeat_interleave(torch.arange(E, device=dev), n)

    # SciFi hits: 98% efficient, 0.07 mm, noise uniform in x on any layer and half
    ti, li = torch.nonzero(rand(T, 12) < 0.98, as_tuple=True)
    sx = (xh + 0.07 * normal(T, 12))[ti, li]
    zone = 2 * li + (ty[ti] >= 0)
    n_ev = noise_of(trk_ev[ti])
    N = n_ev.shape[0]
    hit_off, x, zone = _by_event(torch.cat([trk_ev[ti], n_ev]), E, g, torch.cat([sx, 6400.0 * rand(N) - 3200.0]),
                                 torch.cat([zone, (24 * rand(N)).long().clamp(max=23)]))
    # VELO segments: the tracks' (0.015 mm, 2e-4) and ghosts
    G = torch.repeat_interleave(torch.arange(E, device=dev), (case["ghosts"] * nt.double()).round().long())
    gt = rand(len(G), 2) * torch.tensor([0.6, 0.5], device=dev) - torch.tensor([0.3, 0.25], device=dev)
    tt = torch.stack([tx, ty], 1)
    velo = torch.cat([torch.cat([tt * Z_VELO + 0.015 * normal(T, 2), tt + 2e-4 * normal(T, 2)], 1),
                      torch.cat([gt * Z_VELO + normal(len(G), 2), gt], 1)])
    velo_off, velo = _by_event(torch.cat([trk_ev, G]), E, g, velo)
    out = {"ev_off": hit_off, "x": x.float(), "zone": zone.int(), "velo_off": velo_off, "velo": velo.float()}
    if case["call"] == "match":
        # seeds of 97% of the tracks (0.05 mm, 1e-5) and of 3% that are none, half 0 first
        keep = rand(T) < 0.97
        zS = 7826.0 - Z_REF
        a, c = tx * Z_KINK + (tx + 1.2 * q / p) * (Z_REF - Z_KINK), KAPPA * q / (1000.0 * p)
        b = tx + 1.2 * q / p
        s = torch.stack([a + b * zS + c * zS * zS * (1 + D_RATIO * zS), ty * 7826.0,
                         b + c * (2 * zS + 3 * D_RATIO * zS * zS), ty], 1)
        s = s + normal(T, 4) * torch.tensor([0.05, 0.5, 1e-5, 1e-4], device=dev, dtype=torch.float64)
        s[rand(T) < 0.03, 0] += 40.0
        s, ev = s[keep], trk_ev[keep]
        seed_off, s = _by_event(2 * ev + (s[:, 3] >= 0), 2 * E, g, s)
        n = torch.stack([5 + (rand(len(s)) < 0.88), 4 + (3 * rand(len(s))).long()], 1)
        out.update(seed_off=seed_off[::2].int(), seed_state=s.float(), seed_n=n.to(torch.int8))
    if case["check"]:
        layer = (zone >> 1)
        out["z"] = torch.tensor(Z, device=dev, dtype=torch.float32)[layer]
        out["dxdy"] = torch.tensor(SLOPE, device=dev, dtype=torch.float32)[layer]
    if case["ut"]:
        dz = torch.tensor(UT_Z, device=dev, dtype=torch.float64) - Z_VELO
        gam = UT_GAMMA[0] + UT_GAMMA[1] * q / (1000.0 * p)
        ux = tx[:, None] * (dz + Z_VELO) + gam[:, None] * dz * dz
        ux = ux - ty[:, None] * (dz + Z_VELO) * torch.tensor(UT_SLOPE, device=dev, dtype=torch.float64)
        ux = ux + 0.05 * normal(T, 4)
        ti, li = torch.nonzero((rand(T, 4) < 0.99) & (ux.abs() < 900.0), as_tuple=True)
        n_ev = noise_of(trk_ev[ti])
        N = n_ev.shape[0]
        ut_off, ut_x, ut_l = _by_event(torch.cat([trk_ev[ti], n_ev]), E, g,
                                       torch.cat([ux[ti, li], 1800.0 * rand(N) - 900.0]),
                                       torch.cat([li, (4 * rand(N)).long().clamp(max=3)]))
        out.update(ut_off=ut_off, ut_x=ut_x.float(), ut_layer=ut_l.int())
    return out


@lru_cache(maxsize=1)
def _ghost_weights():
    """Weights of the shape the ghost network takes (mean, inverse scale, W1, b1, w2, b2)."""
    rng = np.random.default_rng(1009)
    mean = [5200.0, 0.0, 0.0, 0.0, 0.0, 1.0, 2.0, 10.0]
    scale = [200.0, 10.0, 50.0, 0.1, 0.005, 1.0, 1.0, 1.0]
    return np.concatenate([mean, 1.0 / np.array(scale), rng.normal(0.0, 8.0 ** -0.5, 256), rng.normal(0.0, 0.3, 32),
                           rng.normal(0.0, 4.0 * 32.0 ** -0.5, 32), [1.5]]).astype(np.float32)


# ---------------------------------------------------------------------------
# prepare and run
# ---------------------------------------------------------------------------

def _mean_tracks(case):
    return case["tracks"] * math.exp(case["spread"] ** 2 / 2)


def _cap(case, events):
    """Room for the seeds of so many events: twice the expected tracks."""
    return int(2.0 * events * _mean_tracks(case)) + 512


def _requests(case):
    """Events of each request of a served case: from small to large, adding up to all."""
    k, n = case["requests"], case["events"]
    w = [4.0 ** i for i in range(k)]
    sizes = [max(1, int((n - k) * v / sum(w))) for v in w]
    sizes[-1] += n - sum(sizes)
    return sizes


def _config(case):
    over = {"zmx": ZMX}
    if case["method"] == "hough":
        over["uv_mode"] = 1
    elif case["method"] == "hlt2":
        over.update(iter_mode=1, n_iter=3, p_min_iter=[5000.0, 3000.0, 1500.0])
    if case["final"]:
        over["final_sel"] = 1
    return st.st_config_default(**over)


class State:
    pass


def prepare(case, seed):
    ev = make_events(case, seed)
    s = State()
    s.case, call = case, case["call"]
    cfg = _config(case)
    if call == "serve":
        s.ctx = st.Context(cfg)
        s.ctx.st_pipeline_configure(n_slots=4, max_events_per_slot=2048, max_hits_per_slot=2048 * 4000,
                                    max_velo_per_slot=2048 * 512)
        h = {k: v.cpu().numpy() for k, v in ev.items()}
        s.requests, e0 = [], 0
        for n in _requests(case):
            eo, vo = h["ev_off"][e0:e0 + n + 1], h["velo_off"][e0:e0 + n + 1]
            hits, velo, keep = st.HostBuffers.inputs(eo - eo[0], h["x"][eo[0]:eo[-1]], h["zone"][eo[0]:eo[-1]],
                                                     vo - vo[0], h["velo"][vo[0]:vo[-1]], pinned=True)
            s.requests.append((hits, velo, keep, st.HostBuffers(n, _cap(case, n), pinned=True)))
            e0 += n
        return s
    s.db = st.DeviceBatch(ev["ev_off"].cpu().numpy(), ev["x"].cpu().numpy(), ev["zone"].cpu().numpy(),
                          ev["velo_off"].cpu().numpy(), ev["velo"].cpu().numpy(),
                          z=ev["z"].cpu().numpy() if "z" in ev else None,
                          dxdy=ev["dxdy"].cpu().numpy() if "dxdy" in ev else None)
    if case["ut"]:
        s.db.add_ut(ev["ut_off"].cpu().numpy(), ev["ut_x"].cpu().numpy(), ev["ut_layer"].cpu().numpy())
    s.out = st.DeviceOutputs(case["events"], _cap(case, case["events"]))
    if call == "static":
        s.cfg = cfg
        return s
    s.ctx = st.Context(cfg)
    if case["final"]:
        s.ctx.st_set_ghost_nn(_ghost_weights())
    if call == "graph":
        s.graph = s.ctx.st_graph_create(s.db.hits, s.db.velo_s, s.out.seeds, s.out.long)
        return s
    s.ctx.st_reserve(case["events"], case["events"] * s.db.max_hits, s.db.max_hits, s.out.cap)
    if call == "match":
        s.out.ev_off.copy_(ev["seed_off"])
        s.out.state[:len(ev["seed_state"])] = ev["seed_state"]
        s.out.n_hits[:len(ev["seed_n"])] = ev["seed_n"]
    return s


def _outputs(o, call, ut, final):
    out = {"ev_off": o.ev_off, "status": o.status, "hits": o.hits, "params": o.params, "state": o.state,
           "n_hits": o.n_hits}
    if call == "match":
        out = {"status": o.status}
    if call != "static":
        out.update(velo_idx=o.velo_idx, chi2=o.chi2, n_long=o.n_long)
    if final:
        out["ghost_prob"] = o.ghost_prob
    if ut:
        out.update(ut_hits=o.ut_hits, ut_n=o.ut_n, ut_gamma=o.ut_gamma)
    return out


def run(s):
    case, call = s.case, s.case["call"]
    if call == "serve":
        tickets = [s.ctx.pipeline_submit(hits, velo) for hits, velo, _, _ in s.requests]
        for t, (_, _, _, buf) in zip(tickets, s.requests):
            rc, _ = s.ctx.pipeline_poll(t, buf.seeds, buf.long, 60_000_000)
            if rc != st.ST_OK:
                raise RuntimeError(f"request not served: {rc}")
        return [_outputs(buf, call, False, False) if i in (0, len(s.requests) - 1) else
                {"params": buf.params, "chi2": buf.chi2, "hits": buf.hits, "velo_idx": buf.velo_idx}
                for i, (_, _, _, buf) in enumerate(s.requests)]
    if call == "static":
        rc, msg = st.seeding_run_static(s.cfg, s.db.hits, s.out.seeds)
        if rc != st.ST_OK:
            raise RuntimeError(msg)
    elif call == "graph":
        s.graph.st_graph_launch()
    else:
        if call == "direct":
            s.ctx.seeding_run(s.db.hits, s.out.seeds)
        s.ctx.matching_run(s.db.velo_s, s.out.seeds, s.out.long)
        if case["ut"]:
            s.ctx.ut_run(s.db.velo_s, s.out.seeds, s.db.ut, s.out.long, s.out.ut_out)
    return _outputs(s.out, call, case["ut"], case["final"])


def work(case):
    """Each hit, VELO segment and UT hit read once, each seed written once; the
    arithmetic of the searches at the case's mean occupancy."""
    E, T = case["events"], _mean_tracks(case)
    m2 = math.exp(case["spread"] ** 2)  # mean square over squared mean of the occupancy
    hits, seeds = E * T * 11.76 * (1 + case["noise"]), E * T
    velo = E * T * (1 + case["ghosts"])
    zone = T * 0.98 * (1 + case["noise"]) / 2  # hits of one layer and half
    n, f = 0.0, 0.0
    if case["call"] != "match":
        n += hits * (16 if case["check"] else 8) + seeds * 98
        f += E * m2 * 4 * 0.138 * zone * zone * 24      # two-hit windows, momentum and third-hit band
        f += seeds * (2 * 0.057 * zone * 160 + 6 * 120)  # stereo chains and fits
    if case["call"] != "static":
        n += velo * 16 + seeds * 8 + (seeds * 16 if case["call"] == "match" else 0)
        f += E * m2 * 0.10 * T * T * (1 + case["ghosts"]) * 45
    if case["final"]:
        n += seeds * 6
        f += seeds * 640
    if case["ut"]:
        n += E * T * 4 * (1 + case["noise"]) * 8 + seeds * 21
        f += seeds * 4 * 40
    return {"bytes": n, "flops": f}


# ---------------------------------------------------------------------------
# the same in 64 bits, in numpy
# ---------------------------------------------------------------------------

XL, UL = [0, 3, 4, 7, 8, 11], [1, 2, 5, 6, 9, 10]
ZX, ZU, TU = (np.array([Z[i] for i in XL]), np.array([Z[i] for i in UL]), np.array([SLOPE[i] for i in UL]))


def _f(z):
    return (z - Z_REF) ** 2 * (1.0 + D_RATIO * (z - Z_REF))


def _gains():
    """Least-squares gain of (1, z, f) for all six x-layers and for each one missing."""
    scale = np.array([1.0, 1e-3, 1e-9])
    phi = np.stack([np.ones(6), ZX - Z_REF, _f(ZX)], 1) * scale
    G = {}
    for miss in range(-1, 6):
        keep = np.array([s != miss for s in range(6)])
        g = np.zeros((3, 6))
        g[:, keep] = np.linalg.pinv(phi[keep], rcond=1e-14) * scale[:, None]
        G[miss] = g
    return G


GAIN = _gains()
ITER = [(0, 2, 5), (1, 3, 4), (0, 3, 5)]  # x-slots of T1, T2, T3


def _spread(first, count):
    """Owner and running index of each element of the ranges [first, first + count)."""
    own = np.repeat(np.arange(len(count)), count)
    return own, first[own] + np.arange(len(own)) - np.repeat(np.cumsum(count) - count, count)


def _closest(xs, xp, tol):
    """Index of the hit closest to each xp within tol, ties to the smaller x; -1 for none."""
    if len(xs) == 0:
        return np.full(len(xp), -1)
    r = np.searchsorted(xs, xp, "left")
    a, b = np.maximum(r - 1, 0), np.minimum(r, len(xs) - 1)
    da, db = np.abs(xs[a] - xp), np.abs(xs[b] - xp)
    best = np.where(da <= db, a, b)
    best = np.searchsorted(xs, xs[best], "left")
    return np.where(np.minimum(da, db) <= tol, best, -1)


def _xz(X, it, p_min):
    """Candidates of one iteration: hits per slot, model, chi2, score."""
    s1, s2, s3 = ITER[it]
    z1, z2, z3 = ZX[s1], ZX[s2], ZX[s3]
    A, B = 1.6322e-7, -5.0217e-12
    alpha = 2.180e6 / (z1 / (z3 - z1) * (p_min + 1073.0))
    dx3 = (z3 - z1) / (2 * z1 * B) * (-A + math.sqrt(A * A + 4 * B / p_min))
    w3 = (z2 - z1) / (z3 - z1)
    k3 = _f(z2) - _f(z1) - w3 * (_f(z3) - _f(z1))
    c0 = 5.0 * 0.07 * math.sqrt(1.0 + (1 - w3) ** 2 + w3 ** 2) / abs(k3)
    x1, x2, x3 = X[s1], X[s2], X[s3]
    xc = (z3 + alpha) / z1 * x1
    lo = np.searchsorted(x3, xc - dx3, "left")
    i1, i3 = _spread(lo, np.searchsorted(x3, xc + dx3, "right") - lo)
    t13 = (x3[i3] - x1[i1]) / (z3 - z1)
    x0 = x1[i1] - z1 * t13
    ip = A * np.abs(x0) + B * x0 * x0
    sg = np.where(x0 > 0, 1.0, -1.0)
    base = x1[i1] + (z2 - z1) * t13
    xa, xb = base - k3 * sg * (0.5 * KAPPA * ip - c0), base - k3 * sg * (1.5 * KAPPA * ip + c0)
    lo = np.searchsorted(x2, np.minimum(xa, xb), "left")
    n = np.where(ip > 0, np.searchsorted(x2, np.maximum(xa, xb), "right") - lo, 0)
    o, i2 = _spread(lo, n)
    i1, i3, t13, base = i1[o], i3[o], t13[o], base[o]
    c = (x2[i2] - base) / k3
    b = t13 - c * (_f(z3) - _f(z1)) / (z3 - z1)
    a = x1[i1] - b * (z1 - Z_REF) - c * _f(z1)
    pos = np.full((len(a), 6), -1)
    pos[:, s1], pos[:, s2], pos[:, s3] = i1, i2, i3
    for s in range(6):
        if s not in (s1, s2, s3):
            pos[:, s] = _closest(X[s], a + b * (ZX[s] - Z_REF) + c * _f(ZX[s]), 1.0)
    ok = (pos >= 0).sum(1) >= 5
    pos, th = pos[ok], np.stack([a, b, c], 1)[ok]
    phi = np.stack([np.ones(6), ZX - Z_REF, _f(ZX)], 1)
    xh = np.stack([X[s][np.maximum(pos[:, s], 0)] if len(X[s]) else np.zeros(len(pos)) for s in range(6)], 1)
    y = np.where(pos >= 0, xh - th @ phi.T, 0.0)
    miss = np.where((pos >= 0).all(1), -1, np.argmin(pos, 1))
    d = np.zeros_like(th)
    for m, g in GAIN.items():
        d[miss == m] = y[miss == m] @ g.T
    r = np.where(pos >= 0, y - d @ phi.T, 0.0)
    chi2, nx = (r * r).sum(1) / 0.07 ** 2, (pos >= 0).sum(1)
    ok = chi2 <= 10.0 * (nx - 3)
    th = th + d
    score = np.where(nx == 6, 1.0, 10.0) * (1000.0 * chi2 + np.abs(th[:, 2]))
    return pos[ok], th[ok], chi2[ok], score[ok]


def _unclone(pos, score, X):
    """The candidates that own enough of their hits."""
    rank = np.empty(len(score), np.int64)
    rank[np.lexsort((np.arange(len(score)), score))] = np.arange(len(score))
    owned = np.zeros(len(score), np.int64)
    for s in range(6):
        best = np.full(len(X[s]) + 1, len(score))
        np.minimum.at(best, pos[:, s], rank)  # the entry of -1 is the spare last one
        owned += (pos[:, s] >= 0) & (best[pos[:, s]] == rank)
    return (owned >= 3) | ((owned >= 2) & (pos >= 0).all(1))


def _uv_chains(U, xu, half):
    """The iterative variant: seed, order and stereo hits of every chain."""
    ylo, yhi = (-50.0, 2500.0) if half else (-2500.0, 50.0)
    found = []
    for first in (0, 1):
        e = np.stack([xu[:, first] - yhi * TU[first], xu[:, first] - ylo * TU[first]])
        lo = np.searchsorted(U[first], e.min(0), "left")
        j, k = _spread(lo, np.searchsorted(U[first], e.max(0), "right") - lo)
        ty = (xu[j, first] - U[first][k]) / TU[first] / ZU[first]
        pos = np.full((len(j), 6), -1)
        pos[:, first] = k
        for u in range(6):
            if u == first:
                continue
            pos[:, u] = _closest(U[u], xu[j, u] - TU[u] * ty * ZU[u], 2.0)
            hit = pos[:, u] >= 0
            yl = (xu[j, u] - (U[u][np.maximum(pos[:, u], 0)] if len(U[u]) else 0.0)) / TU[u]
            ty = np.where(hit, 0.5 * (ty + yl / ZU[u]), ty)
        found.append((j, np.arange(len(j)) + first * 10 ** 6, pos))
    return [np.concatenate([a[i] for a in found]) for i in range(3)]


def _uv_fit(j, order, pos, U, xu):
    """The best stereo combination of each seed: its seed, hit count, y0, ty, chi2."""
    have = pos >= 0
    ok = have.sum(1) >= 4
    j, order, pos, have = j[ok], order[ok], pos[ok], have[ok]
    n = have.sum(1)
    xh = np.stack([U[u][np.maximum(pos[:, u], 0)] if len(U[u]) else np.zeros(len(j)) for u in range(6)], 1)
    y = (xu[j] - xh) / TU
    zm = np.where(have, ZU, 0.0).sum(1) / n
    ym = np.where(have, y, 0.0).sum(1) / n
    dz, dy = np.where(have, ZU - zm[:, None], 0.0), np.where(have, y - ym[:, None], 0.0)
    ty = (dz * dy).sum(1) / (dz * dz).sum(1)
    chi2 = ((dy - ty[:, None] * dz) ** 2).sum(1) / (0.07 / T5) ** 2
    best = np.lexsort((order, chi2, -n, j))
    best = best[np.concatenate([[True], j[best][1:] != j[best][:-1]])] if len(best) else best
    return j[best], n[best], (ym - ty * zm)[best], ty[best], chi2[best], pos[best]


def _seeds_of_half(zones, half):
    """Rows of (params, state, hit count) of the half's seeds, iterations in sequence."""
    X, U = [zones[l] for l in XL], [zones[l] for l in UL]
    rows = []
    for it, p_min in enumerate((5000.0, 3000.0, 1500.0)):
        pos, th, chi2, score = _xz(X, it, p_min)
        keep = _unclone(pos, score, X)
        pos, th, chi2 = pos[keep], th[keep], chi2[keep]
        xu = th @ np.stack([np.ones(6), ZU - Z_REF, _f(ZU)])
        j, n, y0, ty, c2y, upos = _uv_fit(*_uv_chains(U, xu, half), U, xu)
        a, b, c = th[j].T
        zb = 7826.0 - Z_REF
        rows.append(np.stack([a, b, c, chi2[j], y0, ty, c2y, 0 * a, a + b * zb + c * _f(7826.0), y0 + ty * 7826.0,
                              b + c * (2 * zb + 3 * D_RATIO * zb * zb), ty], 1))
        # the seeds' hits are gone for the iterations after this
        X = [np.delete(X[s], pos[j, s][pos[j, s] >= 0]) for s in range(6)]
        U = [np.delete(U[u], upos[:, u][upos[:, u] >= 0]) for u in range(6)]
    return np.concatenate(rows)


def _match(V, S):
    """chi2 and VELO index of each seed's Long track, and the pair quantities of all pairs."""
    dtx, dty = V[None, :, 2] - S[:, 2, None], V[None, :, 3] - S[:, 3, None]
    zm = ZMX[0]
    dx = V[None, :, 0] + (zm - Z_VELO) * V[None, :, 2] - (S[:, 0] + (zm - 7826.0) * S[:, 2])[:, None]
    dy = V[None, :, 1] + (1e4 - Z_VELO) * V[None, :, 3] - (S[:, 1] + (1e4 - 7826.0) * S[:, 3])[:, None]
    c2 = (dx ** 2 / (0.8 * (10.12 ** 2 + 101.0 ** 2 * dtx ** 2))
          + dy ** 2 / (0.2 * (1.59 ** 2 + 212.1 ** 2 * (V[:, 2] ** 2 + V[:, 3] ** 2)))
          + dtx ** 2 / 0.5 + dty ** 2 * 937.5)
    ok = (np.abs(dx) < 20) & (np.abs(dy) < 150) & (np.abs(dtx) < 1.5) & (np.abs(dty) < 0.02) & (c2 < 2)
    c2 = np.where(ok, c2, np.inf)
    v = c2.argmin(1)
    best = c2[np.arange(len(S)), v]
    return np.where(np.isfinite(best), v, -1), np.where(np.isfinite(best), best, 0.0), dx, dy, dtx, dty


def _ghosts(v, c2, V, S, nh, pair):
    """Ghost probabilities, and the matches left after the cut and the clone removal."""
    w = _ghost_weights().astype(np.float64)
    s = np.nonzero(v >= 0)[0]
    tx, ty = V[v[s], 2], V[v[s], 3]
    dx, dy, dtx, dty = (p[s, v[s]] for p in pair)
    eta = np.arcsinh(1.0 / np.maximum(np.hypot(tx, ty), 1e-6))
    f = np.stack([np.full(len(s), ZMX[0]), dx, dy, dtx, dty, c2[s], eta, nh[s]], 1)
    hid = np.maximum(((f - w[:8]) * w[8:16]) @ w[16:272].reshape(32, 8).T + w[272:304], 0.0)
    prob = np.ones(len(v))
    prob[s] = 1.0 / (1.0 + np.exp(-(hid @ w[304:336] + w[336])))
    v = np.where(prob < 0.8, v, -1)
    low = np.full(len(V) + 1, np.inf)
    np.minimum.at(low, v, prob)
    v = np.where((v >= 0) & (prob - low[v] >= 0.05), -1, v)
    return prob, v, np.where(v >= 0, c2, 0.0)


def _ut(v, c2, V, S, ux, ul):
    """gamma of each Long track after the UT search, and the chi2 of those that keep three hits."""
    loose = np.array([(0.8333, 3.3333, 1.2, 8.5), (0.8333, 3.3333, 1.2, 8.5), (1.3333, 3.3333, 1.5, 9.5), (0,) * 4])
    tight = np.array([(0,) * 4, (0.2, 0.6, 0.5, 2.0), (0.4, 1.2, 1.0, 4.0), (0.4, 1.2, 1.0, 4.0)])
    s = np.nonzero(v >= 0)[0]
    x, y, tx, ty = V[v[s]].T
    qop = (S[s, 2] - tx) / 1200.0
    g, n = UT_GAMMA[0] + UT_GAMMA[1] * qop, np.zeros(len(s), int)
    for l in range(4):
        xs = np.sort(ux[ul == l])
        w = np.where(n[:, None] > 0, tight[l], loose[l]).T
        win = np.minimum(np.maximum(w[0] + w[1] * 1000.0 * np.abs(qop), w[2]), w[3])
        dz = UT_Z[l] - Z_VELO
        ys = (y + ty * dz) * UT_SLOPE[l]
        k = _closest(xs, x + tx * dz + g * dz * dz - ys, win)
        hit = (k >= 0) & (w[3] > 0)
        if hit.any():
            g = np.where(hit & (n == 0), (xs[k] + ys - x - tx * dz) / dz ** 2, g)
        n += hit
    gam, c2 = np.zeros(len(v)), c2.copy()
    gam[s] = g
    c2[s[n < 3]] = 0.0
    return gam, c2


def exact(case, seed):
    # With independent iterations both find most tracks, as two candidates of
    # the same hits whose scores differ by rounding alone; which of them stays
    # sets the row of the seed, so the rows have no order in 64 bits.  Beyond
    # some 500 events of 150 tracks the seeding takes too long here.
    seeding = case["call"] != "match"
    if seeding and (case["method"] != "hlt2" or work(case)["flops"] > 5.0e8):
        return None
    ev = {k: v.cpu().numpy() for k, v in make_events(case, seed).items()}
    seeds, chi2, prob, gam = [], [], [], []
    for e in range(case["events"]):
        if seeding:
            h = slice(ev["ev_off"][e], ev["ev_off"][e + 1])
            x, zone = ev["x"][h].astype(np.float64), ev["zone"][h]
            S = np.concatenate([_seeds_of_half([np.sort(x[zone == 2 * l + half]) for l in range(12)], half)
                                for half in (0, 1)])
            seeds.append(S)
            S = S[:, 8:]
        else:
            h = slice(ev["seed_off"][e], ev["seed_off"][e + 1])
            S, nh = ev["seed_state"][h].astype(np.float64), ev["seed_n"][h].astype(np.float64).sum(1)
        V = ev["velo"][ev["velo_off"][e]:ev["velo_off"][e + 1]].astype(np.float64)
        if not len(V) or not len(S):
            v, c2, pr = np.full(len(S), -1), np.zeros(len(S)), np.ones(len(S))
        else:
            v, c2, *pair = _match(V, S)
            pr, v, c2 = _ghosts(v, c2, V, S, nh, pair) if case["final"] else (c2, v, c2)
        if case["ut"]:
            u = slice(ev["ut_off"][e], ev["ut_off"][e + 1])
            g, c2 = _ut(v, c2, V, S, ev["ut_x"][u].astype(np.float64), ev["ut_layer"][u])
            gam.append(g)
        chi2.append(c2), prob.append(pr)

    def rows(per_event):
        a = np.concatenate(per_event)
        return np.concatenate([a, np.zeros((_cap(case, case["events"]) - len(a),) + a.shape[1:])])

    out = _outputs(Nothing(), case["call"], case["ut"], case["final"])
    out["chi2"] = rows(chi2)
    if seeding:
        out.update(params=rows([s[:, :8] for s in seeds]), state=rows([s[:, 8:] for s in seeds]))
    if case["final"]:
        out["ghost_prob"] = rows(prob)
    if case["ut"]:
        out["ut_gamma"] = rows(gam)
    return out


class Nothing:
    """Stands for the outputs that have no value in 64 bits."""

    def __getattr__(self, name):
        return None
