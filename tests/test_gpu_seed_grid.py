"""tkf_find_seeds over its launch variants and window forms: every number of lanes per first hit gives
an event the seeds it has alone, and windows that wrap around phi = +-pi, cover whole rows, or are
widened for hits off the cylinders lose no seed of the oracle's brute-force search."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

import oracle as O  # noqa: E402
from _gpu import device_hits  # noqa: E402
from paper_1702_06359_gb300 import tkf  # noqa: E402
from synth import Detector, EventSpec, generate  # noqa: E402

pytestmark = pytest.mark.gpu


def _seeds(hits, cuts, cap, **cfg):
    ctx = tkf.Context(tkf.default_config(**cfg))
    idx = ctx.build_hit_index(hits)
    h, e = (torch.full(s, -7, dtype=torch.int32, device="cuda") for s in ((3, cap), (cap,)))
    sc, n = torch.zeros(cap, device="cuda"), torch.zeros(1, dtype=torch.int32, device="cuda")
    ctx.find_seeds(idx, cuts, cap, h, e, n, sc)
    ctx.sync_status()
    idx.free()
    ctx.close()
    k = int(n)
    return h[:, :k], e[:k], sc[:k]


@pytest.mark.parametrize("events", [1, 11, 40, 105, 800, 1700])
def test_events_of_a_batch_have_the_seeds_they_have_alone(events):
    """Copies of one 1 003-track event: 1 and 11 copies run on 8 and 4 lanes per first hit, the
    largest batches on 2 and 1."""
    b = generate(EventSpec(seed=91, n_events=1, n_tracks=1003, noise_frac=0.3), Detector(pixel_layers=4))
    one = device_hits(b)
    n, n0 = b.n_hits, int((b.layer == 0).sum())
    cuts = tkf.default_seed_cuts()
    h1, _, s1 = _seeds(one, cuts, n0)
    assert h1.shape[1] > 900
    many = tkf.DeviceHits(*(getattr(one, k).repeat(events) for k in ("x", "y", "z", "var_u", "var_v", "layer")),
                          torch.arange(events + 1, dtype=torch.int32, device="cuda") * n)
    h, e, s = _seeds(many, cuts, n0 * events)
    k = h1.shape[1]
    assert h.shape[1] == k * events
    assert torch.equal(e, torch.arange(events, dtype=torch.int32, device="cuda").repeat_interleave(k))
    assert torch.equal(h, h1.repeat(1, events) + (e * n)[None])
    assert torch.equal(s, s1.repeat(events))


# pt_min 0.06 GeV: circles that do not reach layer 2 at all, so windows of whole rows
@pytest.mark.parametrize("pt_min,d0,hit_dr", [(0.5, 0.08, 0.0), (0.5, 0.08, 0.5), (0.15, 0.5, 0.0), (0.06, 0.3, 0.3)])
def test_windows_lose_no_seed_of_the_brute_force_search(pt_min, d0, hit_dr):
    det = Detector(pixel_layers=4, module_dr=2 * hit_dr)
    b = generate(EventSpec(seed=92, n_events=3, n_tracks=np.array([90, 1, 40]), noise_frac=0.5), det)
    cuts = tkf.default_seed_cuts(pt_min=pt_min, d0_max=d0)
    h, e, s = (t.cpu().numpy() for t in _seeds(device_hits(b), cuts, b.n_hits, hit_dr=hit_dr))
    got = {int(a): (int(p), int(q), float(v)) for a, p, q, v in zip(h[0], h[1], h[2], s)}
    co = O.SeedCuts(cuts.pt_min, cuts.kappa_slack, cuts.z_vertex, cuts.d0_max, cuts.dz_max, cuts.conf_rphi, cuts.conf_z, 1)
    g = O.make_geom(det)
    found = 0
    for ev in range(b.n_events):
        o = int(b.hit_off[ev])
        sl = slice(o, int(b.hit_off[ev + 1]))
        picks = O.find_seeds(g, co, O.hits_of(b, sl))
        for a in np.nonzero(b.layer[sl] == 0)[0]:
            p, mine = picks[a], got.get(o + int(a))
            if p["margin"] < 1e-4 or p["gap"] < 1e-4:  # a decision FP32 may take the other way
                continue
            if p["h1"] < 0:
                assert mine is None
            else:
                assert mine is not None and mine[:2] == (o + p["h1"], o + p["h2"]) and abs(mine[2] - p["score"]) <= 2e-4
                found += 1
    assert found >= 100


# cuts so wide that circles far from the one through the beam line pass, on layers of unequal steps (16 - 6 > 6,
# where the chord cut leaves a circle's far branch), with and without the confirmation
@pytest.mark.parametrize("confirm", [0, 1])
@pytest.mark.parametrize("radii,pt_min,d0", [((3, 6, 16, 25), 0.06, 1.5), ((4, 8, 12, 16), 0.06, 1.0), ((4, 8, 20, 24), 0.1, 1.0),
                                             ((3, 10, 13, 17), 0.2, 0.5)])
def test_wide_cuts_on_random_hits_lose_no_seed(radii, pt_min, d0, confirm):
    rng = np.random.default_rng(int(100 * d0) + confirm)
    n_ev, per = 40, 24
    layer = np.tile(np.repeat(np.arange(4), per), n_ev)
    r, phi = np.array(radii, float)[layer], rng.uniform(-np.pi, np.pi, len(layer))
    x, y, z = (a.astype(np.float32) for a in (r * np.cos(phi), r * np.sin(phi), rng.uniform(-1, 1, len(layer))))
    t = lambda a: torch.as_tensor(a, device="cuda")  # noqa: E731
    v = torch.full((len(layer),), 1e-4, device="cuda")
    off = np.arange(n_ev + 1, dtype=np.int32) * 4 * per
    cuts = tkf.default_seed_cuts(pt_min=pt_min, d0_max=d0, z_vertex=100.0, dz_max=50.0, conf_rphi=1.0, conf_z=50.0, confirm=confirm)
    h, _, s = (a.cpu().numpy() for a in _seeds(tkf.DeviceHits(t(x), t(y), t(z), v, v, t(layer.astype(np.int32)), t(off)), cuts,
                                               len(layer), n_layers=4, radius=radii))
    got = {int(a): (int(p), int(q), float(w)) for a, p, q, w in zip(h[0], h[1], h[2], s)}
    det = Detector(radii=tuple(float(r) for r in radii), x_over_x0=(0.03,) * 4)
    g = O.make_geom(det)
    co = O.SeedCuts(*(getattr(cuts, k) for k in ("pt_min", "kappa_slack", "z_vertex", "d0_max", "dz_max", "conf_rphi", "conf_z")), confirm)
    found = 0
    for ev in range(n_ev):
        sl = slice(off[ev], off[ev + 1])
        hits = np.zeros(4 * per, O.HIT_DTYPE)
        for k, a in (("x", x), ("y", y), ("z", z), ("layer", layer)):
            hits[k] = a[sl]
        picks = O.find_seeds(g, co, hits)
        for a in range(per):
            p, mine = picks[a], got.get(int(off[ev]) + a)
            if p["margin"] < 1e-4 or p["gap"] < 1e-4:
                continue
            if p["h1"] < 0:
                assert mine is None
            else:
                assert mine is not None and mine[:2] == (off[ev] + p["h1"], off[ev] + p["h2"]) and abs(mine[2] - p["score"]) <= 2e-4
                found += 1
    assert found >= 100
