"""The double-precision fit and backward pass on strongly bent tracks, against the oracle: turning
angles between layers from 0.05 to 0.5 rad, on both sides of the limit (0.25) below which the helix
functions use their series, and steps that meet the inner layers at small angles."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

import oracle as O  # noqa: E402
from _gpu import device_hits, device_tracks, host_tracks, param_violations  # noqa: E402
from paper_1702_06359_gb300 import tkf  # noqa: E402
from synth import Detector, EventSpec, generate  # noqa: E402

pytestmark = pytest.mark.gpu


# blocks of one warp: fewer tracks than a warp, one more than a block, many
@pytest.mark.parametrize("n", [7, 33, 1500])
@pytest.mark.parametrize("module_dr", [0.0, 1.0])
def test_f64_fit_and_backward_of_low_momentum_tracks(n, module_dr):
    det = Detector(module_dr=module_dr)
    L = det.n_layers
    b = generate(EventSpec(seed=95, n_tracks=n, pt_min=0.26, pt_max=0.6, scatter=False), det)
    g, hits, ids = O.make_geom(det), O.hits_of(b), b.trk_hits
    p0, c0 = O.seed_estimate(g, hits, ids[:, :3])
    pf, cf, c2, nh, st = O.fit(g, hits, p0, c0, ids, 0, L - 1)
    ok = st == 0
    assert ok.mean() > 0.9
    kappa = 0.00299792458 * det.bz * np.abs(pf[ok, 3])
    assert n < 100 or (4.0 * kappa < 0.1).any() and (5.0 * kappa > 0.2).any()
    ctx = tkf.Context(tkf.default_config(precision=tkf.FP64, hit_dr=0.5 * module_dr))
    dh = device_hits(b)
    out, back = (tkf.DeviceTracks.empty(n, L, tkf.FP64) for _ in range(2))
    ctx.fit(dh, device_tracks(p0, c0, np.zeros(n), np.zeros(n), ids, precision=tkf.FP64), 0, L - 1, out)
    ctx.fit_backward(dh, device_tracks(pf, cf, np.zeros(n), nh, ids, precision=tkf.FP64), L - 1, 0, back, cov_scale=1e4)
    ctx.sync_status()
    ctx.close()
    rb = O.fit_backward(g, hits, pf, cf, ids, L - 1, 0, 1e4)
    both = ok & (rb[4] == 0)
    # double against double in other formulas: 1e-8 of the parameters, as the other double tests
    for got, ref in ((host_tracks(out), pf), (host_tracks(back), rb[0])):
        assert param_violations(got["par"][both], ref[both], rel=1e-8)[1] <= 1.0
    assert np.array_equal(host_tracks(out)["nhits"][both], nh[both])
