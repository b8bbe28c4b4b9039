"""The mixed-precision Kalman update against the same update in double precision on the host.

A fit over the outermost layer alone is one update (no propagation, no scattering).  The hit lies
at (1, 0, z), so its tangent direction is exactly (0, 1) in the kernel's float arithmetic and the
only differences left are the update's own: each covariance element is the exact one rounded to
float, within half a unit of its last place plus 2^-42 of the elements it is made from (pairs of
floats carry 2^-45 per operation)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

from _gpu import device_tracks, unpack_cov  # noqa: E402
from paper_1702_06359_gb300 import tkf  # noqa: E402

pytestmark = pytest.mark.gpu
L = 10


@pytest.mark.parametrize("disk", [False, True], ids=["cylinder", "disk"])
# the variance shrinks by up to S / V: below 2^16 the update runs on pairs, above it in double
@pytest.mark.parametrize("shrink", [0.1, 1.0, 1e3, 3e4, 6.4e4, 6.7e4, 1e6, 1e9])
def test_mixed_update_is_the_double_update_rounded(disk, shrink):
    n = 777
    rng = np.random.default_rng(int(np.log10(shrink) * 10) + 100)
    A = rng.normal(size=(n, 6, 6)) + 2.0 * np.eye(6)
    sd = np.array([1e-2, 1e-2, 1e-1, 1e-1, 1e-2, 1e-2])
    P = np.einsum("nik,njk,i,j->nij", A, A, sd, sd)
    P = P.astype(np.float32).astype(np.float64)
    p = (rng.normal(size=(n, 6)) * 0.1 + np.array([1, 0, 0.5, 0.3, 0.1, 1.3])).astype(np.float32)
    iu, iv = (1, 0) if disk else (1, 2)
    # V set so that the larger of S_ii / V_ii is `shrink`
    var = np.stack([P[:, iu, iu], P[:, iv, iv]], 1) / shrink * rng.uniform(1, 1.3, (n, 2))
    var = var.astype(np.float32)
    z = (p[:, 2] + rng.normal(size=n) * 0.1).astype(np.float32)
    one = torch.ones(n, device="cuda")
    t = lambda a: torch.as_tensor(np.ascontiguousarray(a), device="cuda")  # noqa: E731
    hits = tkf.DeviceHits(one, 0 * one, t(z), t(var[:, 0]), t(var[:, 1]),
                          torch.full((n,), L - 1, dtype=torch.int32, device="cuda"),
                          torch.tensor([0, n], dtype=torch.int32, device="cuda"))
    ids = np.full((n, L), -1, dtype=np.int32)
    ids[:, L - 1] = np.arange(n)
    cfg = dict(radius=(40.0,) * L, disk_z=[8.0 * (l + 1) for l in range(L)]) if disk else {}
    ctx = tkf.Context(tkf.default_config(precision=tkf.MIXED, **cfg))
    init = device_tracks(p.astype(np.float64), P, np.zeros(n), np.full(n, 9), ids, precision=tkf.MIXED)
    out = tkf.DeviceTracks.empty(n, L, tkf.MIXED)
    ctx.fit(hits, init, L - 1, L - 1, out)
    ctx.sync_status()
    ctx.close()
    assert torch.all(out.nhits == 10)

    p = p.astype(np.float64)
    H = np.zeros((2, 6))
    H[0, iu], H[1, iv] = 1, 1
    u = -p[:, 1]
    v = 1 - p[:, 0] if disk else z.astype(np.float64) - p[:, 2]
    r = np.stack([u, v], 1).astype(np.float32).astype(np.float64)
    S = H @ P @ H.T + np.stack([np.diag(d) for d in var.astype(np.float64)])
    K = P @ H.T @ np.linalg.inv(S)
    IKH = np.eye(6) - K @ H
    V = S - H @ P @ H.T
    ref = IKH @ P @ IKH.transpose(0, 2, 1) + K @ V @ K.transpose(0, 2, 1)
    sig = np.sqrt(np.einsum("nii->ni", P))
    got = unpack_cov(out.cov.double().cpu().numpy())
    rho2 = S[:, 0, 1] ** 2 / (S[:, 0, 0] * S[:, 1, 1])
    made_of = sig[:, :, None] * sig[:, None, :] / (1 - rho2)[:, None, None]
    # numpy's own inverse and products: 2^-49 of the same elements
    bound = 2.0 ** -24 * np.abs(ref) + 2.0 ** -42 * made_of
    worst = np.max(np.abs(got - ref) / bound)
    assert worst <= 1.0, worst
    step = np.abs(K * r[:, None, :]).sum(2)
    new = p + (K @ r[:, :, None])[:, :, 0]
    d = out.par.double().cpu().numpy().T - new
    d[:, 4] = (d[:, 4] + np.pi) % (2 * np.pi) - np.pi
    assert np.all(np.abs(d) <= 2.0 ** -22 * (np.abs(p) + step + 7))
    chi2 = np.einsum("ni,nij,nj->n", r, np.linalg.inv(S), r)
    assert np.all(np.abs(out.chi2.double().cpu().numpy() - chi2) <= 2.0 ** -23 * chi2 + 2.0 ** -40 * (r ** 2).sum(1) / np.linalg.eigvalsh(S)[:, 0])
