"""The two forms of the hit index, one block per layer of an event (k_index_segment) and
the kernels that spread a batch over the GPU in several launches, give the same index bit for bit.  A
batch takes the second form where its (event, layer) segments hold more than 16384 hits on average or
its bins are outside 16 .. 4096; empty events bring the average down and the batch into the first."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_1702_06359_gb300 import tkf  # noqa: E402

pytestmark = pytest.mark.gpu
L = 10


def _view(ptr, shape, kind):
    class W:
        __cuda_array_interface__ = {"shape": shape, "typestr": kind, "data": (ptr, False), "version": 3}
    return torch.as_tensor(W(), device="cuda").clone()


def _planes(v, n, segs, nb, events):
    return dict(xyzi=_view(v.hit_xyzi, (n, 4), "<i4"), var=_view(v.hit_var, (n, 2), "<i4"), pos=_view(v.pos_of_hit, (n,), "<i4"),
                off=_view(v.bin_off, (segs * nb + 1,), "<i4"), sub=_view(v.bin_sub, (segs * nb, 4), "<i4"),
                vmax=_view(v.var_max, (segs, 2), "<i4"), ev=_view(v.event_off, (events + 1,), "<i4"))


def _hits(per, order, disks, seed=4):
    """per: hits of each layer of each event"""
    rng = np.random.default_rng(seed)
    layer = []
    for p in per:
        a = np.repeat(np.arange(L), p)
        layer.append(rng.permutation(a) if order == "random" else a)
        if order == "split":  # every layer in two runs
            layer[-1] = np.concatenate([a[::2], a[1::2]])
    off = np.concatenate([[0], np.cumsum([len(a) for a in layer])])
    layer = np.concatenate(layer)
    n, phi = len(layer), rng.uniform(-np.pi, np.pi, len(layer))
    if disks:
        z = np.sign(rng.uniform(-1, 1, n)) * 8.0 * (layer + 1)
        r = np.abs(z) / np.sinh(rng.uniform(1.4, 2.7, n))
    else:
        r = 4.0 * (layer + 1)
        z = r * np.sinh(rng.uniform(-2.1, 2.1, n))
    f = [np.asarray(a, np.float32) for a in (r * np.cos(phi), r * np.sin(phi), z, rng.uniform(1e-4, 2e-4, n), rng.uniform(1e-3, 2e-3, n))]
    return f, layer.astype(np.int32), off.astype(np.int32)


def _device(f, layer, off):
    return tkf.DeviceHits(*(torch.as_tensor(a, device="cuda") for a in (*f, layer, off)))


def _config(n_eta, n_phi, disks):
    kw = dict(n_eta_bins=n_eta, n_phi_bins=n_phi, eta_bin_w=4.0 / n_eta)
    if disks:
        kw.update(radius=(40.0,) * L, disk_z=[8.0 * (l + 1) for l in range(L)], eta_min=-3.0, eta_bin_w=6.0 / n_eta)
    return tkf.default_config(**kw)


# hits of each layer: around the most that a block holds with its keys (37 697 with 2520 bins) and without
# (65 535; 50 168 with 4096 bins), more (in parts), small and empty segments
MIXED = [65535, 65536, 25, 70001, 0, 50168, 50169, 37698, 1, 37697]
EVEN = [17000] * L


@pytest.mark.parametrize("order", ["grouped", "random", "split"])
@pytest.mark.parametrize("n_eta,n_phi,disks", [(40, 63, False), (60, 63, True), (64, 64, False), (16, 16, False)])
@pytest.mark.parametrize("per", [MIXED, EVEN], ids=["mixed", "even"])
def test_segments_equal_the_multi_launch_index(per, n_eta, n_phi, disks, order):
    f, layer, off = _hits([per], order, disks)
    n, nb = len(layer), n_eta * n_phi
    ctx = tkf.Context(_config(n_eta, n_phi, disks))
    got = []
    for empty in (0, 4):
        idx = ctx.build_hit_index(_device(f, layer, np.concatenate([off, np.full(empty, n)]).astype(np.int32)))
        ctx.sync_status()
        got.append(_planes(idx.view(), n, (1 + empty) * L, nb, 1 + empty))
        idx.free()
    ctx.close()
    a, b = got
    for k in ("xyzi", "var", "pos"):
        assert torch.equal(a[k], b[k]), k
    assert torch.equal(a["off"], b["off"][:L * nb + 1]) and (b["off"][L * nb:] == n).all()
    assert torch.equal(a["sub"], b["sub"][:L * nb]) and (b["sub"][L * nb:] == 0).all()
    assert torch.equal(a["vmax"], b["vmax"][:L]) and (b["vmax"][L:] == 0).all()


@pytest.mark.parametrize("events", [2, 40])
def test_noalloc_multi_launch_index_equals_the_allocating_one(events):
    """Few bins and dense events (multi launch), and 15 bins (below the segment form's 16)."""
    cfg = _config(40, 63, False) if events == 2 else _config(5, 3, False)
    per = [EVEN, [16500] * L] if events == 2 else [[k % 37] * L for k in range(events)]
    f, layer, off = _hits(per, "grouped", False)
    hits, n, nb, E = _device(f, layer, off), len(layer), cfg.n_eta_bins * cfg.n_phi_bins, events
    assert n <= tkf.NOALLOC_MAX_HITS and E * L * nb <= tkf.NOALLOC_MAX_BINS
    full = lambda s, d: torch.full(s, -7, dtype=d, device="cuda")  # noqa: E731
    out = dict(hit_xyzi=full((n, 4), torch.float32), hit_var=full((n, 2), torch.float32), bin_sub=full((E * L * nb, 4), torch.int32),
               pos_of_hit=full((n,), torch.int32), bin_off=full((E * L * nb + 1,), torch.int32), var_max=full((E * L, 2), torch.float32),
               event_off=full((E + 1,), torch.int32))
    ctx = tkf.Context(cfg)
    for _ in range(2):
        assert tkf.build_hit_index_noalloc(cfg, hits, out) == tkf.OK
        idx = ctx.build_hit_index(hits)
        ctx.sync_status()
        want = _planes(idx.view(), n, E * L, nb, E)
        for a, b in zip(("hit_xyzi", "hit_var", "pos_of_hit", "bin_off", "bin_sub", "var_max", "event_off"),
                        ("xyzi", "var", "pos", "off", "sub", "vmax", "ev")):
            assert torch.equal(out[a].view(torch.int32), want[b]), a
        idx.free()
    ctx.close()


# hits at the centres of (eta bin, phi sixteenth) cells: the whole index is known on the host
@pytest.mark.parametrize("order", ["grouped", "random"])
@pytest.mark.parametrize("n_eta,n_phi,per,dense", [
    (8, 2, [60000, 0, 20000, 70001, 3, 57820, 57821, 100, 65535, 65536], 0),  # 16 bins, thousands of hits in each
    (40, 63, [40000, 90000, 10, 37697, 0, 65536, 1, 2, 3, 38000], 0.7),  # a bin of more hits than a part holds
    (40, 63, [38000, 0, 10, 70000, 0, 5, 1, 2, 3, 65536], 1.0),  # nothing else
    (63, 65, [50200, 10, 26000, 50300, 60000, 90000, 1, 2, 3, 50000], 0.2)])
def test_dense_bins_and_large_segments_have_the_index_of_their_cells(n_eta, n_phi, per, dense, order):
    rng = np.random.default_rng(6)
    events = [per, [5] * L, [0] * L, [20] * L]
    layer = [np.repeat(np.arange(L), p) for p in events]
    if order == "random":
        layer = [rng.permutation(a) for a in layer]
    off = np.concatenate([[0], np.cumsum([len(a) for a in layer])]).astype(np.int32)
    layer, n, E, nb = np.concatenate(layer), off[-1], len(events), n_eta * n_phi
    eb, pb, sub = (rng.integers(0, k, n) for k in (n_eta, n_phi, 16))
    hot = rng.uniform(size=n) < dense
    eb[hot], pb[hot] = n_eta // 2, n_phi // 3
    w = 4.0 / n_eta
    phi = -np.pi + (pb + (sub + 0.5) / 16) * 2 * np.pi / n_phi
    r = 4.0 * (layer + 1)
    f = [np.asarray(a, np.float32) for a in (r * np.cos(phi), r * np.sin(phi), r * np.sinh(-2.0 + (eb + 0.5) * w),
                                             rng.uniform(1e-4, 2e-4, n), rng.uniform(1e-3, 2e-3, n))]
    ctx = tkf.Context(_config(n_eta, n_phi, False))
    idx = ctx.build_hit_index(_device(f, layer.astype(np.int32), off))
    ctx.sync_status()
    got = {k: v.cpu().numpy() for k, v in _planes(idx.view(), n, E * L, nb, E).items()}
    idx.free()
    ctx.close()
    ev = np.repeat(np.arange(E), np.diff(off))
    cell = ((ev * L + layer) * nb + eb * n_phi + pb) * 16 + sub
    at = np.lexsort((np.arange(n), cell))
    assert np.array_equal(got["pos"][at], np.arange(n))
    assert np.array_equal(got["xyzi"].view(np.float32)[:, :3], np.stack(f[:3], 1)[at])
    assert np.array_equal(got["xyzi"][:, 3], (np.arange(n) - off[ev])[at])
    assert np.array_equal(got["var"].view(np.float32), np.stack(f[3:], 1)[at])
    count = np.bincount(cell, minlength=E * L * nb * 16).reshape(-1, 16)
    assert np.array_equal(got["off"], np.concatenate([[0], np.cumsum(count.sum(1))]))
    starts = np.zeros((E * L * nb, 16), np.int64)
    starts[:, :15] = np.cumsum(count, 1)[:, :15]
    starts[count.sum(1) > 255] = 255
    assert np.array_equal(got["sub"].view(np.uint8).reshape(-1, 16), starts)
    vmax = np.zeros((E * L, 2), np.float32)
    np.maximum.at(vmax, ev * L + layer, np.stack(f[3:], 1))
    assert np.array_equal(got["vmax"].view(np.float32), vmax)


# 40 events run in two size classes, ten in one; with 60 x 63 bins the smaller class has no room for hits
@pytest.mark.parametrize("n_eta,n_phi", [(40, 63), (57, 62), (60, 63), (64, 64)])
def test_size_classes_give_the_same_index(n_eta, n_phi):
    per = [[int(900 * (1 + (3 * e + l) % 11)) if l < 4 else 10 * l for l in range(L)] for e in range(40)]
    f, layer, off = _hits(per, "grouped", False)
    nb = n_eta * n_phi
    ctx = tkf.Context(_config(n_eta, n_phi, False))

    def index(e0, e1):
        a, b = off[e0], off[e1]
        idx = ctx.build_hit_index(_device([x[a:b] for x in f], layer[a:b], off[e0:e1 + 1] - a))
        ctx.sync_status()
        got = _planes(idx.view(), int(b - a), (e1 - e0) * L, nb, e1 - e0)
        idx.free()
        return got
    whole = index(0, 40)
    for e0 in range(0, 40, 10):
        part, a, b, s = index(e0, e0 + 10), int(off[e0]), int(off[e0 + 10]), slice(e0 * L, (e0 + 10) * L)
        for k in ("xyzi", "var"):
            assert torch.equal(whole[k][a:b], part[k])
        assert torch.equal(whole["pos"][a:b], part["pos"] + a)
        assert torch.equal(whole["off"][e0 * L * nb:(e0 + 10) * L * nb + 1], part["off"] + a)
        assert torch.equal(whole["sub"][e0 * L * nb:(e0 + 10) * L * nb], part["sub"]) and torch.equal(whole["vmax"][s], part["vmax"])
    ctx.close()
