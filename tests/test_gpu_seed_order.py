"""Building with the seeds grouped by (event, eta bin, phi bin) gives what building in input order gives, bit for
bit, at a size where the grouping takes place (3.5 M seeds times candidates)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

from _gpu import device_hits  # noqa: E402
from paper_1702_06359_gb300 import tkf  # noqa: E402
from synth import Detector, EventSpec, generate  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [218750, 218749, 250003])  # times 16: from 3.5 M on, one seed fewer, a ragged number
@pytest.mark.parametrize("precision", [tkf.FP32, tkf.MIXED, tkf.FP64], ids=["fp32", "mixed", "fp64"])
def test_grouped_seeds_build_the_tracks_of_seeds_in_order(precision, n):
    b = generate(EventSpec(seed=31, n_events=7, n_tracks=np.array([300, 1, 0, 500, 90, 400, 250]), noise_frac=0.3), Detector())
    hits = device_hits(b)
    rng = np.random.default_rng(n)
    pick = rng.integers(0, b.n_tracks, n)  # every track some 140 times, in no order
    sh = torch.as_tensor(np.ascontiguousarray(b.trk_hits[pick, :3].T), dtype=torch.int32, device="cuda")
    event = torch.as_tensor(b.trk_event[pick], dtype=torch.int32, device="cuda")
    got = []
    for order in (0, 1):
        ctx = tkf.Context(tkf.default_config(precision=precision, n_cand=16, seed_order=order))
        L = ctx.cfg.n_layers
        seeds, built = (tkf.DeviceTracks.empty(n, L, precision) for _ in range(2))
        ctx.seed_fit(hits, sh, 2, seeds)
        seeds.event = event
        idx = ctx.build_hit_index(hits)
        for _ in range(2):  # (the ordering's counters are back to zero for the second)
            ctx.build_tracks(idx, seeds, built)
        ctx.sync_status()
        got.append([getattr(built, k).clone() for k in ("par", "cov", "chi2", "nhits", "hit_idx")])
        idx.free()
        ctx.close()
    assert (got[0][3] >= 5).float().mean() > 0.9
    assert all(torch.equal(x, y) for x, y in zip(*got))
