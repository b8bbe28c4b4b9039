"""The hit index built by one block per layer of an event (k_index_segment), against an index made on the
host from the library's own bins: order by (event, layer, bin, phi sixteenth, id), bin offsets,
sixteenth starts, positions and largest variances, bit for bit.  Segments at the edges of its size
classes, hits of a layer that are not consecutive, empty layers and events, a dense bin."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_1702_06359_gb300 import tkf  # noqa: E402

pytestmark = pytest.mark.gpu
L, NETA, NPHI = 10, 40, 63
NB = NETA * NPHI


def _view(ptr, shape, kind):
    class W:
        __cuda_array_interface__ = {"shape": shape, "typestr": kind, "data": (ptr, False), "version": 3}
    return torch.as_tensor(W(), device="cuda").cpu().numpy()


def _index(x, y, z, layer, off):
    n = len(x)
    rng = np.random.default_rng(5)
    vu, vv = (rng.uniform(1e-4, 2e-4, n).astype(np.float32) for _ in range(2))
    t = lambda a: torch.as_tensor(np.ascontiguousarray(a), device="cuda")  # noqa: E731
    # one byte offset of four from an aligned address, as a slice of a larger array has
    lay = torch.zeros(n + 1, dtype=torch.int32, device="cuda")
    lay[1:] = t(layer)
    ctx = tkf.Context()
    idx = ctx.build_hit_index(tkf.DeviceHits(t(x), t(y), t(z), t(vu), t(vv), lay[1:], t(off)))
    ctx.sync_status()
    v = idx.view()
    E = len(off) - 1
    got = dict(xyzi=_view(v.hit_xyzi, (n, 4), "<f4"), var=_view(v.hit_var, (n, 2), "<f4"), pos=_view(v.pos_of_hit, (n,), "<i4"),
               off=_view(v.bin_off, (E * L * NB + 1,), "<i4"), sub=_view(v.bin_sub, (E * L * NB, 4), "<u4"),
               vmax=_view(v.var_max, (E * L, 2), "<f4"), ev=_view(v.event_off, (E + 1,), "<i4"))
    idx.free()
    ctx.close()
    return got, vu, vv


def _check(x, y, z, layer, off):
    got, vu, vv = _index(x, y, z, layer, off)
    n, E = len(x), len(off) - 1
    ev = np.repeat(np.arange(E), np.diff(off))
    ids = np.arange(n) - off[ev]
    pos = got["pos"]
    assert np.array_equal(np.sort(pos), np.arange(n)) and np.array_equal(got["ev"], off)
    # the bin of a hit: where its position lies in the offsets; the sixteenth from the packed starts
    bin_ = np.searchsorted(got["off"], pos, side="right") - 1
    assert np.array_equal(bin_ // NB, ev * L + layer)
    start = got["off"][bin_]
    count = got["off"][bin_ + 1] - start
    by = got["sub"].view(np.uint8).reshape(-1, 16)[bin_][:, :15].astype(int)
    known = count <= 255
    sub = (by <= (pos - start)[:, None]).sum(1)
    assert (got["sub"][bin_[~known]] == 0xFFFFFFFF).all()
    # the library's bins to rounding of an edge: eta and phi in double
    R = 4.0 * (layer + 1)
    eb = np.clip((np.arcsinh(z / R) + 2.0) / 0.1, 0, NETA - 1e-9)
    pc = (np.arctan2(y, x) + np.pi) * NPHI / (2 * np.pi)
    local = bin_ % NB
    assert (np.abs(eb - local // NPHI - 0.5) <= 0.5 + 1e-4).all()
    assert (np.abs(pc - local % NPHI - 0.5) <= 0.5 + 1e-4).all()
    frac = (pc - local % NPHI) * 16
    assert (np.abs(frac - sub - 0.5)[known] <= 0.5 + 1e-2).all()
    # order inside a bin: sixteenth, then id
    at = np.argsort(pos)
    b, s, i = bin_[at], sub[at], ids[at]
    same = (b[1:] == b[:-1]) & known[at][1:]
    assert ((s[1:] > s[:-1]) | ((s[1:] == s[:-1]) & (i[1:] > i[:-1])))[same].all()
    big = (b[1:] == b[:-1]) & ~known[at][1:]  # sixteenths unknown: frac is sorted up to its rounding
    f = frac[at]
    assert (np.floor(f[1:] + 1e-2) >= np.floor(f[:-1] - 1e-2))[big].all()
    assert np.array_equal(got["xyzi"][pos, :3], np.stack([x, y, z], 1)) and np.array_equal(got["xyzi"][pos, 3].view(np.int32), ids)
    assert np.array_equal(got["var"][pos], np.stack([vu, vv], 1))
    vmax = np.zeros((E * L, 2), np.float32)
    np.maximum.at(vmax, ev * L + layer, np.stack([vu, vv], 1))
    assert np.array_equal(got["vmax"], vmax)


def _hits(rng, layer, width=np.pi):
    R = 4.0 * (layer + 1)
    phi = rng.uniform(-width, width, len(layer))
    return tuple(a.astype(np.float32) for a in (R * np.cos(phi), R * np.sin(phi), R * np.sinh(rng.uniform(-2.1, 2.1, len(layer)))))


# hits of the first layer: the small class holds 8512, the large one 37697 (226 KB less the counters)
@pytest.mark.parametrize("first", [0, 1, 31, 8511, 8512, 8513, 37697, 37698])
def test_segments_at_the_edges_of_their_classes(first):
    rng = np.random.default_rng(first)
    per = [[first, 5, 0, 1, 700, 33, 2, 1, 0, 3]] + [list(rng.integers(0, 40, L)) for _ in range(20)] + [[0] * L]
    layer = np.concatenate([np.repeat(np.arange(L), p) for p in per])
    off = np.concatenate([[0], np.cumsum([sum(p) for p in per])]).astype(np.int32)
    _check(*_hits(rng, layer), layer, off)


@pytest.mark.parametrize("n", [3, 500, 30000])
@pytest.mark.parametrize("order", ["random", "descending", "split"])
def test_layers_whose_hits_are_not_in_order(n, order):
    rng = np.random.default_rng(n)
    layer = np.sort(rng.integers(0, L, n))
    if order == "random":
        layer = rng.permutation(layer)
    elif order == "descending":
        layer = layer[::-1].copy()
    else:  # one layer in two runs
        layer = np.concatenate([layer[layer != 4], layer[layer == 4]])
        layer = np.roll(layer, n // 100)
    off = np.array([0, n // 3, n // 3, n], dtype=np.int32)
    _check(*_hits(rng, layer), layer, off)


def test_events_with_their_layers_mixed_among_events_in_order():
    """Every order within one batch, at sizes around the words and warps the layers are counted in, and a
    segment of more than the large class holds."""
    rng = np.random.default_rng(11)
    layer = []
    for k, n in enumerate([0, 1, 3, 4, 5, 31, 32, 33, 127, 129, 1023, 1024, 1025, 4099, 33000, 3 * L]):
        for order in range(3):
            a = np.sort(rng.integers(0, L, n))
            layer.append(a if order == 0 else rng.permutation(a) if order == 1 else np.roll(np.arange(n) % L, k))
    layer.append(rng.permutation(np.concatenate([np.full(38000, 7), np.arange(500) % L])))
    off = np.concatenate([[0], np.cumsum([len(a) for a in layer])]).astype(np.int32)
    layer = np.concatenate(layer)
    _check(*_hits(rng, layer), layer, off)


def test_a_dense_bin_and_many_equal_sixteenths():
    rng = np.random.default_rng(3)
    layer = np.repeat(np.arange(L), 3000)
    _check(*_hits(rng, layer, width=0.03), layer, np.array([0, len(layer)], dtype=np.int32))


@pytest.mark.parametrize("order", ["grouped", "random"])
def test_an_event_over_the_hit_limit_fills_its_part_of_the_index(order):
    """2^23 + 5 hits of one event among enough small ones for k_index_segment; the last five lie where the
    first five do, so that they share their sixteenths with ids equal to theirs in the lowest 23 bits."""
    rng = np.random.default_rng(8)
    big, small = (1 << 23) + 5, 40
    n_ev = 60  # 16384 hits per segment on average would be 9.8 M
    layer = rng.integers(0, L, big)
    if order == "grouped":
        layer = np.sort(layer)
    layer[-5:] = layer[:5]
    layer = np.concatenate([layer, np.tile(np.arange(small) // 4, n_ev - 1)])
    off = np.concatenate([[0], big + small * np.arange(n_ev)]).astype(np.int32)
    x, y, z = _hits(rng, layer)
    for a in (x, y, z):
        a[big - 5:big] = a[:5]
    t = lambda a: torch.as_tensor(np.ascontiguousarray(a), device="cuda")  # noqa: E731
    n = len(layer)
    v = torch.full((n,), 1e-4, device="cuda")
    ctx = tkf.Context()
    idx = ctx.build_hit_index(tkf.DeviceHits(t(x), t(y), t(z), v, v, t(layer.astype(np.int32)), t(off)))
    with pytest.raises(tkf.TkfError, match="8388606"):
        ctx.sync_status()
    w = idx.view()
    pos, xyzi = _view(w.pos_of_hit, (n,), "<i4"), _view(w.hit_xyzi, (n, 4), "<f4")
    assert np.array_equal(np.sort(pos), np.arange(n))
    ev = np.repeat(np.arange(n_ev), np.diff(off))
    assert np.array_equal(xyzi[pos, :3], np.stack([x, y, z], 1))
    assert np.array_equal(xyzi[pos, 3].view(np.int32), np.arange(n) - off[ev])
    idx.free()
    ctx.close()
