"""Calls issued one after another on a stream, without a synchronisation and on the same buffers: the
kernels of a call may be set up while the call before it still runs, and must neither read what it
has not written yet nor write what it still reads."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

from _gpu import device_hits  # noqa: E402
from paper_1702_06359_gb300 import tkf  # noqa: E402
from synth import Detector, EventSpec, generate  # noqa: E402

pytestmark = pytest.mark.gpu


class Chain:
    """Index, seeds, seed fit, building, final fit and backward pass into one set of buffers."""

    def __init__(self, batch, precision):
        self.ctx = tkf.Context(tkf.default_config(precision=precision))
        self.hits, n, L = device_hits(batch), batch.n_tracks, self.ctx.cfg.n_layers
        self.sh = torch.as_tensor(np.ascontiguousarray(batch.trk_hits[:, :3].T), dtype=torch.int32, device="cuda")
        self.trk = [tkf.DeviceTracks.empty(n, L, precision) for _ in range(4)]
        self.trk[0].event = torch.as_tensor(batch.trk_event, dtype=torch.int32, device="cuda")
        self.cap = int((batch.layer == 0).sum())
        self.found, self.fev = (torch.full(s, -1, dtype=torch.int32, device="cuda") for s in ((3, self.cap), (self.cap,)))
        self.count = torch.zeros(1, dtype=torch.int32, device="cuda")
        self.idx = self.ctx.build_hit_index(self.hits)

    def run(self, xyz, stream):
        for dst, src in zip((self.hits.x, self.hits.y, self.hits.z), xyz):
            dst.copy_(src)
        seeds, built, final, back = self.trk
        L, s = self.ctx.cfg.n_layers, stream
        self.found.fill_(-1)
        self.ctx.build_hit_index(self.hits, self.idx, stream=s)
        self.ctx.find_seeds(self.idx, tkf.default_seed_cuts(), self.cap, self.found, self.fev, self.count, stream=s)
        self.ctx.seed_fit(self.hits, self.sh, 2, seeds, stream=s)
        self.ctx.build_tracks(self.idx, seeds, built, stream=s)
        self.ctx.fit(self.hits, seeds, 3, L - 1, final, hit_idx=built.hit_idx, continue_fit=True, stream=s)
        self.ctx.fit_backward(self.hits, final, L - 1, 0, back, hit_idx=built.hit_idx, stream=s)

    def results(self):
        return [t.clone() for k in self.trk for t in (k.par, k.cov, k.chi2, k.nhits)] + [
            self.trk[1].hit_idx.clone(), self.found.clone(), self.count.clone()]


@pytest.mark.parametrize("precision", [tkf.FP32, tkf.MIXED, tkf.FP64], ids=["fp32", "mixed", "fp64"])
@pytest.mark.parametrize("events,tracks", [(1, 33), (1, 1000), (3, 900), (40, 250), (20, 1024)])
def test_a_chain_of_calls_gives_what_single_calls_give(events, tracks, precision):
    b = generate(EventSpec(seed=17, n_events=events, n_tracks=tracks, noise_frac=0.4), Detector())
    chain = Chain(b, precision)
    x, y, z = chain.hits.x.clone(), chain.hits.y.clone(), chain.hits.z.clone()
    inputs = [(x, y, z), (-y, x, -z)]  # the batch, and it turned by a right angle and mirrored
    stream = torch.cuda.Stream()
    want = []
    for xyz in inputs:
        with torch.cuda.stream(stream):
            chain.run(xyz, stream)
        torch.cuda.synchronize()
        want.append(chain.results())
    assert not torch.equal(want[0][0], want[1][0])
    got = []
    with torch.cuda.stream(stream):
        for k in range(12):
            chain.run(inputs[k % 2], stream)
            got.append(chain.results())
    torch.cuda.synchronize()
    # and captured: the same calls as one graph
    graphs = []
    for xyz in inputs:
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=stream):
            chain.run(xyz, stream)
        graphs.append(g)
    with torch.cuda.stream(stream):
        for k in range(12):
            graphs[k % 2].replay()
            got.append(chain.results())
    torch.cuda.synchronize()
    chain.ctx.sync_status()
    for k, r in enumerate(got):
        assert all(torch.equal(a, w) for a, w in zip(r, want[k % 2])), k
