"""Hits whose layer is out of range: they are reported, take no part in any step, and leave nothing of an
earlier batch where the index has a place for them."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

from _gpu import device_hits  # noqa: E402
from paper_1702_06359_gb300 import tkf  # noqa: E402
from synth import Detector, EventSpec, generate  # noqa: E402

pytestmark = pytest.mark.gpu


def _steps(ctx, hits, sh, event, index=None):
    """Index (a reused one if given), seeds, seed fit and building; results and the index's positions."""
    L, n = ctx.cfg.n_layers, sh.shape[1]
    idx = ctx.build_hit_index(hits, index)
    cap = hits.x.numel()
    found, fev = (torch.full(s, -1, dtype=torch.int32, device="cuda") for s in ((3, cap), (cap,)))
    count = torch.zeros(1, dtype=torch.int32, device="cuda")
    ctx.find_seeds(idx, tkf.default_seed_cuts(), cap, found, fev, count)
    seeds, built = tkf.DeviceTracks.empty(n, L), tkf.DeviceTracks.empty(n, L)
    seeds.event = event
    ctx.seed_fit(hits, sh, 2, seeds)
    ctx.build_tracks(idx, seeds, built)
    torch.cuda.synchronize()

    class W:
        __cuda_array_interface__ = {"shape": (cap, 4), "typestr": "<f4", "data": (idx.view().hit_xyzi, False), "version": 3}
    xyzi = torch.as_tensor(W(), device="cuda").clone()
    return idx, (seeds, built), found[:, :int(count)], xyzi


# 2 events run in one size class of the index, 40 in two; 4 layers: the seeding reads the last layer
@pytest.mark.parametrize("events,layers", [(2, 10), (2, 4), (40, 10)])
def test_hits_without_a_layer_change_nothing(events, layers):
    det = Detector(radii=tuple(4.0 * (l + 1) for l in range(layers)), x_over_x0=(0.03,) * layers, pixel_layers=4)
    b = generate(EventSpec(seed=23, n_events=events, n_tracks=220, noise_frac=0.4), det)
    clean, off = device_hits(b), b.hit_off.astype(int)
    sh = torch.as_tensor(np.ascontiguousarray(b.trk_hits[:, :3].T), dtype=torch.int32, device="cuda")
    event = torch.as_tensor(b.trk_event, dtype=torch.int32, device="cuda")
    ctx = tkf.Context(tkf.default_config(n_layers=layers))
    _, want, want_seeds, _ = _steps(ctx, clean, sh, event)
    ctx.sync_status()
    # 37 such hits behind the others of every event but the last: copies of its hits on the last layer
    bad, where = 37, []
    for e in range(events):
        own = np.arange(off[e], off[e + 1])
        where.append(own)
        if e + 1 < events:
            where.append(own[b.layer[own] == layers - 1][:bad])
    take = torch.as_tensor(np.concatenate(where), device="cuda")
    layer = torch.as_tensor(np.concatenate([b.layer[w] if k % 2 == 0 else np.where(np.arange(bad) % 2, -1, layers)
                                            for k, w in enumerate(where)]), dtype=torch.int32, device="cuda")
    shift = torch.arange(events, device="cuda", dtype=torch.int32) * bad
    off2 = torch.as_tensor(off, dtype=torch.int32, device="cuda")
    off2[:events] += shift
    off2[events] += bad * (events - 1)
    hits = tkf.DeviceHits(*(getattr(clean, k)[take].contiguous() for k in ("x", "y", "z", "var_u", "var_v")), layer, off2)
    # the index held a batch before this one: the same size, every hit on the last layer at the last bin
    n = hits.x.numel()
    near = torch.zeros(n, device="cuda")
    last = 4.0 * layers
    before = tkf.DeviceHits(near - last, near + 1e-3, near + last * 3.5, near + 1e-4, near + 1e-2,
                            torch.full((n,), layers - 1, dtype=torch.int32, device="cuda"), off2)
    idx = ctx.build_hit_index(before)
    ctx.sync_status()
    _, got, got_seeds, xyzi = _steps(ctx, hits, sh + shift[event.long()][None], event, idx)
    with pytest.raises(tkf.TkfError, match="layer"):
        ctx.sync_status()
    for g, w in zip(got, want):
        for k in ("par", "cov", "chi2", "nhits"):
            assert torch.equal(getattr(g, k), getattr(w, k)), k
    moved = torch.where(want[1].hit_idx >= 0, want[1].hit_idx + shift[event.long()][None], want[1].hit_idx)
    assert torch.equal(got[1].hit_idx, moved)
    seed_event = torch.searchsorted(torch.as_tensor(off, device="cuda"), want_seeds[0].long(), right=True) - 1
    assert want_seeds.shape[1] > 50 * events and torch.equal(got_seeds, want_seeds + shift[seed_event][None])
    free = torch.cat([torch.arange(int(o) - bad, int(o), device="cuda") for o in off2[1:events]])
    assert torch.isnan(xyzi[free, :3]).all() and (xyzi[free, 3].view(torch.int32) == 0).all()
    assert int(torch.isnan(xyzi[:, :3]).any(1).sum()) == len(free)
