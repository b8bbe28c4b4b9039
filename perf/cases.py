"""Performance cases of the tracking library: the calls its users make, over the sizes they make them at.

The sizes follow the benchmark's and the tests' workloads: single trigger events of a few hundred to a
few thousand tracks, the 20 x 5000-track plain workload, and batches of up to 640 events with lognormal
track counts (median 3000) and 20-50 % noise hits; on the ten-layer barrel, on modules off its cylinders,
on the ten-disk endcap tracker and on the barrel with pixel inner layers.

Inputs are generated on the GPU from the seed alone: a flat-pT gun (0.5-10 GeV) through the detector with
multiple scattering, Gaussian hit smearing and uniform noise, hits grouped by event and layer in a random
order.  `exact` is a plain double-precision Kalman filter and combinatorial builder in torch.
"""
import math
import random
import statistics

import numpy as np
import torch

from paper_1702_06359_gb300 import tkf

L = 10
KB = 0.00299792458 * 3.8     # curvature per q/pT: 1 / (GeV cm)
MASS = 0.13957
X0 = 0.03                    # x/X0 of every layer
RADII = [4.0 * (l + 1) for l in range(L)]
DISK_Z = [8.0 * (l + 1) for l in range(L)]
MODULE_DR = 0.5              # modules lie this far inside or outside their layer's radius
PRIOR = [0.1, 0.1, 1.0, 0.5, 0.05, 0.05]
FORWARD_PRIOR = [0.3, 0.3, 1.0, 5.0, 0.1, 0.1]
CUT = 30.0
BACK_SCALE = 1e4
PRECISION = {"fp32": tkf.FP32, "mixed": tkf.MIXED, "fp64": tkf.FP64}
DEV = "cuda"


# ------------------------------------------------------------------------------------ cases

def case_of(name, kind, events, tracks, spread=0.8, geometry="barrel", precision="fp32", n_cand=6, extra=False):
    """events x tracks (the median; lognormal with sigma `spread`, 0: all alike).  `extra`: the backward
    pass (fit, pipeline) or every final candidate (build)."""
    c = dict(kind=kind, events=events, tracks=tracks, spread=spread, geometry=geometry, precision=precision,
             n_cand=n_cand, extra=extra)
    return dict(c, name=name) if name else c


def listed():
    return [
        # a trigger's single event through the whole step: launches and latency
        case_of("pipeline_one_event", "pipeline", 1, 1000, 0.0),
        # offline reconstruction of a full batch, the headline workload
        case_of("pipeline_640_events", "pipeline", 640, 3000),
        # the numerically safer mode with the track state carried back to the vertex
        case_of("pipeline_mixed_back", "pipeline", 40, 3001, precision="mixed", extra=True),
        # a stream of events from host memory, submitted as they come
        case_of("server_12_events", "server", 12, 4997, 0.0),
        # indexing a handful of dense events, before any of the steps below
        case_of("index_20_events", "index", 20, 5000, 0.0),
        # indexing a large batch
        case_of("index_512_events", "index", 512, 2500),
        # refitting known tracks: a large sample, forward only
        case_of("fit_one_million", "fit", 250, 4000, 0.0),
        # a precision study: double throughout, forward and backward
        case_of("fit_fp64_back", "fit", 20, 2003, 0.0, precision="fp64", extra=True),
        # building with more candidates, all of them kept for a later stage
        case_of("build_ten_cand", "build", 20, 3000, 0.0, n_cand=10, extra=True),
        # building on modules off the cylinders (two steps per hit)
        case_of("build_modules", "build", 60, 2999, geometry="modules"),
        # building in the endcaps
        case_of("build_disks", "build", 240, 749, geometry="disks"),
        # finding the seeds on the device
        case_of("seeds_160_events", "seeds", 160, 3000, geometry="pixels"),
    ]


def draw(rng):
    log = lambda a, b: int(round(math.exp(rng.uniform(math.log(a), math.log(b)))))  # noqa: E731
    kind = rng.choice(["pipeline", "pipeline", "build", "build", "index", "fit", "seeds", "server"])
    tracks = log(200, 6000)
    most = {"pipeline": 400_000, "build": 300_000, "index": 1_500_000, "fit": 1_200_000, "seeds": 200_000,
            "server": 60_000}[kind]
    events = log(1, max(1, min(640 if kind != "server" else 12, most // tracks)))
    geometry = rng.choice({"pipeline": ["barrel", "barrel", "modules", "disks"], "build": ["barrel", "modules", "disks"],
                           "index": ["barrel", "disks"], "fit": ["barrel", "modules", "disks"], "seeds": ["pixels"],
                           "server": ["barrel"]}[kind])
    precision = rng.choice({"fit": ["fp32", "mixed", "fp64"], "pipeline": ["fp32", "mixed"], "build": ["fp32", "mixed"],
                            "server": ["fp32", "mixed"]}.get(kind, ["fp32"]))
    if precision != "fp32":
        events = max(1, min(events, 150_000 // tracks))
    extra = kind in ("fit", "pipeline", "build") and rng.random() < 0.4 and geometry != "modules"
    if kind == "build" and extra:
        events = max(1, min(events, 150_000 // tracks))
    return case_of(None, kind, events, tracks, rng.choice([0.0, 0.8]), geometry, precision,
                   rng.choice([4, 6, 6, 10]) if kind in ("build", "pipeline") else 6, extra)


def event_tracks(case):
    """Tracks of each event: the quantiles of the lognormal in a mixed order, the same for every seed."""
    n, nd = case["events"], statistics.NormalDist()
    t = [case["tracks"] * math.exp(case["spread"] * nd.inv_cdf((i + 0.5) / n)) for i in range(n)]
    random.Random(n).shuffle(t)
    return [int(min(max(round(v), 20), 20000)) for v in t]


def event_noise(case):
    """Noise hits per layer of each event: 20 to 50 % of its tracks."""
    n = case["events"]
    return [int(round((0.2 + 0.3 * (i * 7 % n) / max(1, n - 1)) * t)) for i, t in enumerate(event_tracks(case))]


def work(case):
    T, H = sum(event_tracks(case)), L * (sum(event_tracks(case)) + sum(event_noise(case)))
    es = 8 if case["precision"] == "fp64" else 4
    state = 28 * es + 4
    bins = case["events"] * L * (60 if case["geometry"] == "disks" else 40) * 63
    index = {"bytes": 24 * H + 28 * H + 20 * bins, "flops": 40 * H}
    prop, upd, sca, chi = 593, 335, 30, 39
    fit = {"bytes": T * (L * (20 + 4) + 2 * state), "flops": T * ((L - 1) * (prop + sca) + L * upd)}
    # per seed: about 20 propagated candidates, 190 scored hits, 18 updates over the seven built layers
    scored = {"barrel": 190 * chi, "pixels": 190 * chi, "modules": 213 * 14 + 26 * 405 + 18 * prop, "disks": 218 * 57}
    build = {"bytes": T * (2 * state + 4 * L) + 24 * H * (L - 3) // L,
             "flops": T * (20 * prop + scored[case["geometry"]] + 18 * upd + 19 * sca) * max(1, case["n_cand"] / 6)}
    k = case["kind"]
    if k == "index":
        return index
    if k == "fit":
        n = 2 if case["extra"] else 1
        return {"bytes": n * fit["bytes"], "flops": n * fit["flops"]}
    if k == "build":
        every = T * case["n_cand"] * (state + 4 * L) if case["extra"] else 0
        return {"bytes": build["bytes"] + every, "flops": build["flops"] + T * 3 * (prop + upd)}
    if k == "seeds":
        return {"bytes": 16 * H * 4 // L + 20 * T, "flops": T * 3000}
    n = 2 if case["extra"] else 1
    return {"bytes": index["bytes"] + build["bytes"] + n * fit["bytes"],
            "flops": index["flops"] + build["flops"] + n * fit["flops"]}


# ------------------------------------------------------------------------------------ helix, double precision

def sinc(a):
    return torch.where(a.abs() < 1e-4, 1 - a * a / 6, torch.sin(a) / torch.where(a == 0, torch.ones_like(a), a))


def wrap(phi):
    return torch.remainder(phi + math.pi, 2 * math.pi) - math.pi


def helix_xy(p, s):
    """Transverse position and direction angle after the transverse path s."""
    a = -KB * p[:, 3] * s
    c = 0.5 * a * sinc(0.5 * a) ** 2
    sp, cp, S = torch.sin(p[:, 4]), torch.cos(p[:, 4]), sinc(a)
    return p[:, 0] + s * (cp * S - sp * c), p[:, 1] + s * (sp * S + cp * c), p[:, 4] + a


def path_to_radius(p, R, inner=False):
    """Transverse path to the cylinder of radius R: the next crossing ahead; inner: the nearer of two."""
    A = p[:, 0] * torch.cos(p[:, 4]) + p[:, 1] * torch.sin(p[:, 4])
    d = (A * A + R * R - p[:, 0] ** 2 - p[:, 1] ** 2).clamp(min=0).sqrt()
    s = -A - d if inner else torch.where(A > 0, (R * R - p[:, 0] ** 2 - p[:, 1] ** 2) / (A + d).clamp(min=1e-9), d - A)
    for _ in range(10):
        x, y, f = helix_xy(p, s)
        s = s - (x * x + y * y - R * R) / (2 * (x * torch.cos(f) + y * torch.sin(f)))
    return s


def path_to_plane(p, zp):
    return (zp - p[:, 2]) * torch.tan(p[:, 5])


def at_path(p, s):
    x, y, f = helix_xy(p, s)
    q = p.clone()
    q[:, 0], q[:, 1], q[:, 2], q[:, 4] = x, y, p[:, 2] + s / torch.tan(p[:, 5]), wrap(f)
    return q


# ------------------------------------------------------------------------------------ inputs

def prior_of(case):
    return FORWARD_PRIOR if case["geometry"] == "disks" else PRIOR


def config(case):
    kw = dict(precision=PRECISION[case["precision"]], n_cand=case["n_cand"], seed_order=1)
    if case["geometry"] == "modules":
        kw["hit_dr"] = MODULE_DR
    if case["geometry"] == "disks":
        kw.update(radius=(40.0,) * L, disk_z=DISK_Z, eta_min=-3.0, n_eta_bins=60, prior_sigma=FORWARD_PRIOR)
    return tkf.default_config(**kw)


def module_radius(l, phi):
    n = 2 * max(2, math.ceil(math.pi * RADII[l] / 2.0))
    k = torch.clamp(torch.floor((phi + math.pi) / (2 * math.pi) * n), 0, n - 1)
    return RADII[l] + torch.where(torch.remainder(k, 2) == 0, -MODULE_DR, MODULE_DR)


def kicked(p, cosa, g):
    """A multiple-scattering kick: two Gaussian angles of Highland width, |p| kept."""
    st, ct, sp, cp = torch.sin(p[:, 5]), torch.cos(p[:, 5]), torch.sin(p[:, 4]), torch.cos(p[:, 4])
    mom = 1 / (p[:, 3].abs() * st)
    b2 = mom * mom / (mom * mom + MASS * MASS)
    t = X0 / cosa
    th0 = 0.0136 / (b2.sqrt() * mom) * t.sqrt() * (1 + 0.038 * torch.log(t / b2))
    a, b = th0 * torch.randn(len(p), generator=g, device=DEV, dtype=torch.float64), \
        th0 * torch.randn(len(p), generator=g, device=DEV, dtype=torch.float64)
    dx, dy, dz = st * cp + a * ct * cp - b * sp, st * sp + a * ct * sp + b * cp, ct - a * st
    q = p.clone()
    q[:, 5] = torch.atan2((dx * dx + dy * dy).sqrt(), dz)
    q[:, 4] = torch.atan2(dy, dx)
    q[:, 3] = torch.sign(p[:, 3]) / (mom * torch.sin(q[:, 5]))
    return q


def events(case, seed):
    """Hits (float32 x, y, z, var_u, var_v, int32 layer, event_off) and the tracks' hit ids [L, T]."""
    g = torch.Generator(device=DEV).manual_seed(seed)
    f8 = dict(generator=g, device=DEV, dtype=torch.float64)
    nt, nn = torch.tensor(event_tracks(case), device=DEV), torch.tensor(event_noise(case), device=DEV)
    E, T, N = len(nt), int(nt.sum()), int(nn.sum())
    disks = case["geometry"] == "disks"
    tev = torch.repeat_interleave(torch.arange(E, device=DEV), nt, output_size=T)
    nev = torch.repeat_interleave(torch.arange(E, device=DEV), nn, output_size=N)
    p = torch.empty((T, 6), device=DEV, dtype=torch.float64)
    p[:, 0], p[:, 1], p[:, 2] = (s * torch.randn(T, **f8) for s in (0.01, 0.01, 1.0))
    p[:, 3] = torch.where(torch.rand(T, **f8) < 0.5, 1.0, -1.0) / (0.5 + 9.5 * torch.rand(T, **f8))
    p[:, 4] = math.pi * (2 * torch.rand(T, **f8) - 1)
    eta = 2 * torch.rand(T, **f8) - 1
    if disks:
        eta = torch.sign(eta) * (1.7 + 0.8 * eta.abs())
    p[:, 5] = 2 * torch.atan(torch.exp(-eta))
    key, xyz, var = [], [], []
    for l in range(L):
        su, sv = (0.002, 0.005) if case["geometry"] == "pixels" and l < 4 else (0.01, 0.1)
        gu, gv = su * torch.randn(T, **f8), sv * torch.randn(T, **f8)
        nphi, u = math.pi * (2 * torch.rand(N, **f8) - 1), 2 * torch.rand(N, **f8) - 1
        if disks:
            p = at_path(p, path_to_plane(p, torch.sign(torch.cos(p[:, 5])) * DISK_Z[l]))
            f, r, z = torch.atan2(p[:, 1], p[:, 0]), torch.hypot(p[:, 0], p[:, 1]), p[:, 2]
            f, r = f + gu / r, r + gv
            nr, nz = DISK_Z[l] / torch.sinh(1.5 + 1.2 * u.abs()), torch.sign(u) * DISK_Z[l]
            cosa = torch.cos(p[:, 5]).abs()
        else:
            R = torch.full((T,), RADII[l], device=DEV, dtype=torch.float64)
            if case["geometry"] == "modules":
                x, y, _ = helix_xy(p, path_to_radius(p, R))
                R = module_radius(l, torch.atan2(y, x))
            p = at_path(p, path_to_radius(p, R))
            f, r, z = torch.atan2(p[:, 1], p[:, 0]), R, p[:, 2] + gv
            cosa = (torch.sin(p[:, 5]) * torch.cos(p[:, 4] - f)).abs()
            f = f + gu / r
            nr = module_radius(l, nphi) if case["geometry"] == "modules" else torch.full_like(nphi, RADII[l])
            nz = u * (RADII[l] * math.sinh(1.0) + 3.0)
        f, r, z = torch.cat([f, nphi]), torch.cat([r, nr]), torch.cat([z, nz])
        xyz.append(torch.stack([r * torch.cos(f), r * torch.sin(f), z]).float())
        key.append(torch.cat([tev, nev]) * L + l + torch.rand(T + N, **f8))
        var.append((su * su, sv * sv))
        p = kicked(p, cosa, g)
    at = torch.argsort(torch.cat(key))
    rank = torch.empty_like(at)
    rank[at] = torch.arange(len(at), device=DEV)
    trk = torch.stack([rank[l * (T + N):l * (T + N) + T] for l in range(L)]).int().contiguous()
    layer = torch.repeat_interleave(torch.arange(L, device=DEV), T + N)[at]
    xyz = torch.cat(xyz, 1)[:, at]
    var = torch.tensor(var, device=DEV, dtype=torch.float32)[layer]
    off = torch.zeros(E + 1, device=DEV, dtype=torch.int32)
    off[1:] = torch.cumsum(L * (nt + nn), 0)
    hits = tkf.DeviceHits(*(v.contiguous() for v in (xyz[0], xyz[1], xyz[2], var[:, 0], var[:, 1], layer.int())), off)
    return hits, trk, tev.int()


# ------------------------------------------------------------------------------------ the calls

def prepare(case, seed):
    hits, trk, ev = events(case, seed)
    n, prec, kind = trk.shape[1], PRECISION[case["precision"]], case["kind"]
    s = dict(case=case, n=n, hits=hits)
    if kind == "server":
        # host buffers in pinned memory, lent to the server; limits a little above the burst
        off, toff = hits.event_off.tolist(), [0] + torch.cumsum(torch.bincount(ev), 0).tolist()
        host = {k: getattr(hits, k).cpu().numpy() for k in ("x", "y", "z", "var_u", "var_v", "layer")}
        first = trk[:3].cpu().numpy()
        s["held"] = []
        s["events"] = [tkf.HostEvent(*(host[k][a:b] for k in host), first[:, t0:t1] - a, borrow=True)
                       for a, b, t0, t1 in zip(off, off[1:], toff, toff[1:])]
        s["burst"] = (tkf.Event * len(s["events"]))(*(e.struct for e in s["events"]))
        s["server"] = tkf.Server(config(case), n_slots=3, max_batch_events=4, max_batch_tracks=max(4 * 5100, n // 2),
                                 max_batch_hits=max(600_000, len(hits.x) // 2))
        s["hits"] = None
        return s
    s["ctx"] = ctx = tkf.Context(config(case))
    s["seed_hits"], s["event"], s["trk"] = trk[:3].contiguous(), ev, trk
    empty = lambda m=n: tkf.DeviceTracks.empty(m, L, prec)  # noqa: E731
    if kind == "pipeline":
        s["pipe"] = tkf.DevicePipeline(ctx, len(hits.x), case["events"], n)
        if case["extra"]:
            s["pipe"].set_backward(BACK_SCALE)
    elif kind == "index":
        s["index"] = None
    elif kind == "fit":
        s["init"], s["out"], s["back"] = empty(), empty(), empty() if case["extra"] else None
    elif kind == "build":
        s["index"] = ctx.build_hit_index(hits)
        s["init"], s["out"] = empty(), empty()
        s["init"].event = ev
        s["all"] = empty(n * case["n_cand"]) if case["extra"] else None
        s["n_cand"] = torch.zeros(n, dtype=torch.int32, device=DEV)
    elif kind == "seeds":
        s["index"] = ctx.build_hit_index(hits)
        m = s["max"] = int((hits.layer == 0).sum())
        s["found"], s["fev"] = (torch.full(z, -1, dtype=torch.int32, device=DEV) for z in ((3, m), (m,)))
        s["score"], s["count"] = torch.zeros(m, device=DEV), torch.zeros(1, dtype=torch.int32, device=DEV)
    return s


def planes(t):
    return dict(par=t.par, cov=t.cov, chi2=t.chi2, nhits=t.nhits)


class View:
    """An array of the library's memory, device or pinned host; `owner` stays alive with it."""

    def __init__(self, owner, device, **interface):
        self.owner = owner
        setattr(self, "__cuda_array_interface__" if device else "__array_interface__", dict(interface, version=3))


def device_view(owner, ptr, shape, kind):
    return torch.as_tensor(View(owner, True, shape=shape, typestr=kind, data=(ptr, False)), device=DEV)


def track_views(owner, t, precision):
    f, n = "<f8" if precision == "fp64" else "<f4", t.stride
    return dict(par=device_view(owner, t.par, (6, n), f), cov=device_view(owner, t.cov, (21, n), f),
                chi2=device_view(owner, t.chi2, (n,), f), nhits=device_view(owner, t.nhits, (n,), "<i4"),
                hit_idx=device_view(owner, t.hit_idx, (L, n), "<i4"))


def run(s):
    case, kind = s["case"], s["case"]["kind"]
    if kind == "server":
        server = s["server"]
        if s["held"]:  # the last burst's results are done with
            server.release_many(s["held"])
        code, tickets = server.submit_many(s["burst"])
        if code != tkf.OK:
            raise RuntimeError("submit_many: status %d" % code)
        code, res = server.wait_all(tickets)
        s["held"] = tickets
        if code != tkf.OK:
            raise RuntimeError("wait_all: status %d" % code)
        return [server_result(s, r) for r in res]
    ctx, hits = s["ctx"], s["hits"]
    if kind == "pipeline":
        s["pipe"].run(hits, s["seed_hits"], s["event"], s["n"])
        _, _, fitted = s["pipe"].outputs()
        out = track_views(s, fitted, case["precision"])
        if case["extra"]:
            back = track_views(s, s["pipe"].backward_outputs(), case["precision"])
            out.update({"back_" + k: back[k] for k in ("par", "cov", "chi2", "nhits")})
        return out
    if kind == "index":
        s["index"] = ctx.build_hit_index(hits, reuse=s["index"])
        v = s["index"].view()
        segs = v.n_events * v.n_layers
        parts = dict(xyzi=(v.hit_xyzi, (v.n, 4)), var=(v.hit_var, (v.n, 2)), sub=(v.bin_sub, (segs * v.n_bins, 4)),
                     pos=(v.pos_of_hit, (v.n,)), off=(v.bin_off, (segs * v.n_bins + 1,)), var_max=(v.var_max, (segs, 2)))
        return {k: device_view(s, ptr, shape, "<i4") for k, (ptr, shape) in parts.items()}
    if kind == "fit":
        ctx.seed_state(hits, s["seed_hits"], s["init"])
        ctx.fit(hits, s["init"], 0, L - 1, s["out"], hit_idx=s["trk"])
        out = dict(planes(s["out"]), seed_par=s["init"].par)
        if case["extra"]:
            ctx.fit_backward(hits, s["out"], L - 1, 0, s["back"], cov_scale=BACK_SCALE, hit_idx=s["trk"])
            out.update({"back_" + k: v for k, v in planes(s["back"]).items()})
        return out
    if kind == "build":
        ctx.seed_fit(hits, s["seed_hits"], 2, s["init"])
        ctx.build_tracks(s["index"], s["init"], s["out"], s["all"], s["n_cand"])
        out = dict(planes(s["out"]), hit_idx=s["out"].hit_idx, n_cand=s["n_cand"])
        if case["extra"]:
            out.update({"all_" + k: v for k, v in dict(planes(s["all"]), hit_idx=s["all"].hit_idx).items()})
        return out
    ctx.find_seeds(s["index"], tkf.default_seed_cuts(), s["max"], s["found"], s["fev"], s["count"], s["score"])
    return dict(hits=s["found"], event=s["fev"], count=s["count"], score=s["score"])


def server_result(owner, r):
    """numpy views of one event's result in the server's pinned memory (valid until it is released)."""
    def rows(ptr, k, kind):
        return np.asarray(View(owner, False, shape=(k, r.n_tracks), typestr=kind, data=(ptr, True), strides=(4 * r.stride, 4)))
    return [rows(r.par, 6, "<f4"), rows(r.cov, 21, "<f4"), rows(r.chi2, 1, "<f4"), rows(r.nhits, 1, "<i4"),
            rows(r.hit_idx, L, "<i4")]


# ------------------------------------------------------------------------------------ the same in 64 bits

class Exact:
    """Kalman filter and combinatorial building in double precision, dense 6x6 algebra."""

    def __init__(self, case, hits):
        self.case, self.disks = case, case["geometry"] == "disks"
        self.h = torch.stack([hits.x, hits.y, hits.z, hits.var_u, hits.var_v], 1).double()
        self.layer = hits.layer.long()
        self.off = hits.event_off.long()

    def seed(self, ids):
        a, b, c = (self.h[ids[k].long()] for k in range(3))
        ab, bc, ac = b - a, c - b, c - a
        d = [torch.hypot(v[:, 0], v[:, 1]) for v in (ab, bc, ac)]
        kappa = 2 * (ab[:, 0] * bc[:, 1] - ab[:, 1] * bc[:, 0]) / (d[0] * d[1] * d[2])
        h12, h13 = (0.5 * kappa * d[0]).clamp(-1, 1), (0.5 * kappa * d[2]).clamp(-1, 1)
        over = torch.where(h13.abs() < 1e-4, 1 + h13 ** 2 / 6, torch.asin(h13) / torch.where(h13 == 0, torch.ones_like(h13), h13))
        p = torch.stack([a[:, 0], a[:, 1], a[:, 2], -kappa / KB,
                         wrap(torch.atan2(ab[:, 1], ab[:, 0]) - torch.asin(h12)),
                         torch.atan2(torch.ones_like(kappa), ac[:, 2] / (d[2] * over))], 1)
        prior = torch.tensor(prior_of(self.case), device=DEV, dtype=torch.float64) ** 2
        if self.disks:
            prior[2] = 0
        return p, torch.diag(prior).expand(len(p), 6, 6).clone()

    def move(self, p, P, s, plane=False):
        q = at_path(p, s)
        a = -KB * p[:, 3] * s
        S, C = sinc(a), 0.5 * a * sinc(0.5 * a) ** 2
        safe = torch.where(a.abs() < 1e-3, torch.ones_like(a), a)
        Sd = torch.where(a.abs() < 1e-3, -a / 3 + a ** 3 / 30, (torch.cos(a) - S) / safe)
        Cd = torch.where(a.abs() < 1e-3, 0.5 - a * a / 8, (torch.sin(a) - C) / safe)
        sp, cp, st = torch.sin(p[:, 4]), torch.cos(p[:, 4]), torch.sin(p[:, 5])
        cot = torch.cos(p[:, 5]) / st
        c1, s1 = torch.cos(p[:, 4] + a), torch.sin(p[:, 4] + a)
        J = torch.eye(6, device=DEV, dtype=torch.float64).repeat(len(p), 1, 1)
        J[:, 0, 3], J[:, 1, 3] = -KB * s * s * (cp * Sd - sp * Cd), -KB * s * s * (sp * Sd + cp * Cd)
        J[:, 0, 4], J[:, 1, 4] = p[:, 1] - q[:, 1], q[:, 0] - p[:, 0]
        J[:, 2, 5], J[:, 4, 3] = -s / st ** 2, -KB * s
        if plane:
            ds = -J[:, 2] / cot[:, None]
        else:
            ds = -(q[:, :1] * J[:, 0] + q[:, 1:2] * J[:, 1]) / (q[:, 0] * c1 + q[:, 1] * s1)[:, None]
        J += torch.stack([c1, s1, cot, 0 * a, -KB * p[:, 3], 0 * a], 1)[:, :, None] * ds[:, None, :]
        return q, J @ P @ J.transpose(1, 2)

    def radius_of(self, l, hid):
        h = self.h[hid.long()]
        return torch.hypot(h[:, 0], h[:, 1])

    def to_layer(self, p, P, l, hid=None, inner=False):
        if self.disks:
            zp = torch.where(p[:, 2] >= 0, DISK_Z[l], -DISK_Z[l])
            return self.move(p, P, path_to_plane(p, zp), True)
        R = torch.full_like(p[:, 0], RADII[l])
        if hid is not None and self.case["geometry"] == "modules":
            R = torch.where(hid >= 0, self.radius_of(l, hid.clamp(min=0)), R)
        return self.move(p, P, path_to_radius(p, R, inner))

    def measure(self, p, P, h):
        """Residual [M, 2], H P [M, 2, 6] and S [M, 2, 2]."""
        r = torch.hypot(h[:, 0], h[:, 1])
        sh, ch = h[:, 1] / r, h[:, 0] / r
        dx, dy = h[:, 0] - p[:, 0], h[:, 1] - p[:, 1]
        B0 = ch[:, None] * P[:, 1] - sh[:, None] * P[:, 0]
        if self.disks:
            v, B1 = ch * dx + sh * dy, ch[:, None] * P[:, 0] + sh[:, None] * P[:, 1]
            S01, S11 = ch * B0[:, 0] + sh * B0[:, 1], ch * B1[:, 0] + sh * B1[:, 1]
        else:
            v, B1 = h[:, 2] - p[:, 2], P[:, 2]
            S01, S11 = B0[:, 2], B1[:, 2]
        S = torch.stack([ch * B0[:, 1] - sh * B0[:, 0] + h[:, 3], S01, S01, S11 + h[:, 4]], 1).view(-1, 2, 2)
        return torch.stack([ch * dy - sh * dx, v], 1), torch.stack([B0, B1], 1), S

    @staticmethod
    def inverse(S):
        det = S[:, 0, 0] * S[:, 1, 1] - S[:, 0, 1] ** 2
        return torch.stack([S[:, 1, 1], -S[:, 0, 1], -S[:, 0, 1], S[:, 0, 0]], 1).view(-1, 2, 2) / det[:, None, None]

    def update(self, p, P, hid):
        """The update of the states with a hit (hid >= 0) and their chi2."""
        h = self.h[hid.clamp(min=0).long()]
        r, B, S = self.measure(p, P, h)
        Si = self.inverse(S)
        K = B.transpose(1, 2) @ Si
        c2 = ((r[:, None] @ Si) @ r[:, :, None])[:, 0, 0]
        has = hid >= 0
        q = torch.where(has[:, None], p + (K @ r[:, :, None])[:, :, 0], p)
        q[:, 4] = wrap(q[:, 4])
        D = B.transpose(1, 2) - K @ S
        Q = P - (K @ B + D @ K.transpose(1, 2))
        return q, torch.where(has[:, None, None], Q, P), torch.where(has, c2, torch.zeros_like(c2))

    def scatter(self, p, P):
        st, ct = torch.sin(p[:, 5]), torch.cos(p[:, 5])
        w = p[:, 3]
        mom = 1 / (w.abs() * st)
        b2 = mom * mom / (mom * mom + MASS * MASS)
        if self.disks:
            cosa = ct.abs()
        else:
            cosa = (st * (p[:, 0] * torch.cos(p[:, 4]) + p[:, 1] * torch.sin(p[:, 4])) / torch.hypot(p[:, 0], p[:, 1])).abs()
        t = X0 / cosa
        v = (0.0136 / (b2.sqrt() * mom) * t.sqrt() * (1 + 0.038 * torch.log(t / b2))) ** 2
        cot = ct / st
        P[:, 3, 3] += w * w * cot * cot * v
        P[:, 5, 3] -= w * cot * v
        P[:, 3, 5] -= w * cot * v
        P[:, 4, 4] += v / (st * st)
        P[:, 5, 5] += v

    def fit(self, p, P, c2, ids, first, last, prop_first):
        for l in range(first, last + 1):
            if l > first or prop_first:
                p, P = self.to_layer(p, P, l, ids[l])
            p, P, d = self.update(p, P, ids[l])
            c2 = c2 + d
            if l < L - 1:
                self.scatter(p, P)
        return p, P, c2

    @staticmethod
    def reverse(p, P, scale):
        q = p.clone()
        q[:, 3], q[:, 4], q[:, 5] = -p[:, 3], wrap(p[:, 4] + math.pi), math.pi - p[:, 5]
        sg = torch.tensor([1., 1., 1., -1., 1., -1.], device=DEV, dtype=torch.float64)
        return q, P * (scale * sg[:, None] * sg[None, :])

    def backward(self, p, P, ids):
        p, P = self.reverse(p, P, BACK_SCALE)
        c2 = torch.zeros_like(p[:, 0])
        for l in range(L - 1, -1, -1):
            if l < L - 1:
                p, P = self.to_layer(p, P, l, ids[l], True)
            p, P, d = self.update(p, P, ids[l])
            c2 = c2 + d
            self.scatter(p, P)
        return *self.reverse(p, P, 1.0), c2

    def layer_hits(self, l):
        """Hits of layer l ordered by (event, azimuth), copies beyond +-pi included: keys and ids."""
        ids = torch.nonzero(self.layer == l)[:, 0]
        ev = torch.searchsorted(self.off, ids, right=True) - 1
        phi = torch.atan2(self.h[ids, 1], self.h[ids, 0])
        key = torch.cat([20 * ev + phi, 20 * ev + phi + 2 * math.pi, 20 * ev + phi - 2 * math.pi])
        key, at = torch.sort(key)
        return key, torch.cat([ids, ids, ids])[at]

    def branches(self, p, P, ev, l, hits):
        """(candidate, hit, chi2) of every hit below the cut."""
        key, ids = hits
        r = torch.hypot(p[:, 0], p[:, 1])
        st = p[:, 1] / r
        ct = p[:, 0] / r
        Suu = st * st * P[:, 0, 0] - 2 * st * ct * P[:, 0, 1] + ct * ct * P[:, 1, 1]
        U = 1.01 * torch.sqrt(CUT * (Suu + 1.1e-4))
        if self.case["geometry"] == "modules":
            f = p[:, 4] - torch.atan2(p[:, 1], p[:, 0])
            t = MODULE_DR / torch.cos(f).abs().clamp(min=0.01)
            U = U + 1.1 * t * (torch.sin(f).abs() + t * KB * p[:, 3].abs())
            U = U + math.sqrt(CUT) * t / torch.cos(f).abs().clamp(min=0.01) * (P[:, 4, 4].sqrt() + Suu.sqrt() / r) * 1.1
        half = torch.asin((U / r).clamp(max=1)) + 1e-3
        phi = 20 * ev + torch.atan2(p[:, 1], p[:, 0])
        lo, hi = torch.searchsorted(key, phi - half), torch.searchsorted(key, phi + half)
        cum = torch.cumsum(hi - lo, 0)
        got, a = [], 0
        while a < len(p):  # a bounded number of pairs at a time
            start = int(cum[a - 1]) if a else 0
            b = max(a + 1, int(torch.searchsorted(cum, start + 20_000_000, right=True)))
            n = hi[a:b] - lo[a:b]
            c = torch.repeat_interleave(torch.arange(a, min(b, len(p)), device=DEV), n)
            first = torch.repeat_interleave(lo[a:b] - (cum[a:b] - n - start), n)
            h = ids[first + torch.arange(len(c), device=DEV)]
            hh = self.h[h]
            near = (hh[:, 2] * p[c, 2] > 0) if self.disks else \
                (hh[:, 2] - p[c, 2]).abs() < 10 + 6 * torch.sqrt(P[c, 2, 2])
            c, h, hh = c[near], h[near], hh[near]
            q, Q = p[c], P[c]
            if self.case["geometry"] == "modules":
                uv = hh[:, 0] * q[:, 1] - hh[:, 1] * q[:, 0]
                zok = (hh[:, 2] - q[:, 2]).abs() < 1.5 * torch.sqrt(CUT * (Q[:, 2, 2] + 0.011)) + 2
                ok = (uv.abs() / r[c] < 1.5 * U[c] + 0.1) & zok
                c, h, hh, q, Q = c[ok], h[ok], hh[ok], q[ok], Q[ok]
                q, Q = self.move(q, Q, path_to_radius(q, torch.hypot(hh[:, 0], hh[:, 1])))
            res, _, S = self.measure(q, Q, hh)
            c2 = ((res[:, None] @ self.inverse(S)) @ res[:, :, None])[:, 0, 0]
            ok = c2 < CUT
            got.append((c[ok], h[ok], c2[ok]))
            a = b
        return [torch.cat(v) for v in zip(*got)]

    def build(self, p, P, c2, tev, ids):
        """The best N candidates of every seed: state, chi2, hits [.., L], all seed-major, rank order."""
        N, S = self.case["n_cand"], len(p)
        seed = torch.arange(S, device=DEV)
        rank, nh = torch.zeros_like(seed), torch.full_like(seed, 3)
        hits = torch.full((S, L), -1, device=DEV, dtype=torch.int64)
        hits[:, :3] = ids[:3].T
        for l in range(3, L):
            p, P = self.to_layer(p, P, l)
            c, h, d = self.branches(p, P, tev[seed], l, self.layer_hits(l))
            hole = torch.ones(len(p), dtype=torch.bool, device=DEV)
            hole[c] = False
            hole = torch.nonzero(hole)[:, 0]
            par = torch.cat([c, hole])
            hid = torch.cat([h, torch.full_like(hole, -1)])
            tot = torch.cat([c2[c] + d, c2[hole]])
            n = torch.cat([nh[c] + 1, nh[hole]])
            at = torch.argsort(rank[par], stable=True)  # order: seed, more hits, smaller chi2, parent
            at = at[torch.argsort(tot[at], stable=True)]
            at = at[torch.argsort(-n[at], stable=True)]
            at = at[torch.argsort(seed[par[at]], stable=True)]
            own = seed[par[at]]
            pos = torch.arange(len(at), device=DEV) - torch.searchsorted(own, own)
            at, rank = at[pos < N], pos[pos < N]
            par, hid = par[at], hid[at]
            seed, nh, c2 = seed[par], n[at], tot[at]
            p, P, hits = p[par], P[par], hits[par]
            hits[:, l] = hid
            if self.case["geometry"] == "modules":
                has = torch.nonzero(hid >= 0)[:, 0]
                q, Q = self.move(p[has], P[has], path_to_radius(p[has], self.radius_of(l, hid[has])))
                p[has], P[has] = q, Q
            p, P, _ = self.update(p, P, hid)
            if l < L - 1:
                self.scatter(p, P)
        return p, P, c2, hits, rank


def packed(P):
    return torch.stack([P[:, i, j] for i in range(6) for j in range(i + 1)])


def exact(case, seed):
    T, kind = sum(event_tracks(case)), case["kind"]
    if kind in ("index", "seeds"):  # whole numbers; a search over every triplet is too slow
        return None
    if T > (1_500_000 if kind == "fit" else 250_000):
        return None
    hits, trk, tev = events(case, seed)
    x = Exact(case, hits)
    p0, P0 = x.seed(trk)
    if kind == "fit":
        out = dict(seed_par=p0.T.contiguous())
        states = []
        for a in range(0, T, 100_000):
            b = min(T, a + 100_000)
            q, Q, c = x.fit(p0[a:b], P0[a:b], torch.zeros(b - a, device=DEV, dtype=torch.float64), trk[:, a:b], 0, L - 1, False)
            st = (q.T, packed(Q), c)
            if case["extra"]:
                q, Q, c = x.backward(q, Q, trk[:, a:b])
                st += (q.T, packed(Q), c)
            states.append(st)
        for k, v in zip(("par", "cov", "chi2", "back_par", "back_cov", "back_chi2"), zip(*states)):
            out[k] = torch.cat(v, -1)
        return out
    zero = torch.zeros(T, device=DEV, dtype=torch.float64)
    s = x.fit(p0, P0, zero, trk, 0, 2, False)
    p, P, c2, hl, rank = x.build(*s, tev.long(), trk.long())
    best = rank == 0
    if kind == "build":
        # the runners-up are ranked by sums that may be as close as their rounding: none of theirs
        return dict(par=p[best].T, cov=packed(P[best]), chi2=c2[best])
    ids = hl[best].T
    f = x.fit(*s, ids, 3, L - 1, True)
    if kind == "server":
        n = torch.bincount(tev.long()).tolist()
        cols = [t.split(n, 1) for t in (f[0].T, packed(f[1]), f[2][None])]
        return [[*(c.cpu().numpy() for c in one), None, None] for one in zip(*cols)]
    out = dict(par=f[0].T, cov=packed(f[1]), chi2=f[2])
    if case["extra"]:
        b = x.backward(f[0], f[1], ids)
        out.update(back_par=b[0].T, back_cov=packed(b[1]), back_chi2=b[2])
    return out
