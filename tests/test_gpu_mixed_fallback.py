"""The mixed-precision Kalman update where a variance shrinks by more than 2^16: it runs in double, which the test
of the update on pairs of floats does not tell from the pairs (its bound is theirs).  Here each covariance
element is the exact update's within half a unit of its last place plus 2^-49 of the elements it is made of (16
roundings of double); the pairs' own arithmetic, done on the host, misses that."""
import os
import shutil
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1702_06359_gb300", "csrc")
L, N = 10, 777
TRI = [(i, j) for i in range(6) for j in range(i + 1)]

PROGRAM = r"""
#include <cstdio>
#include "pair_f32.cuh"
using namespace tkf;
int main()
{  // P - K B on pairs for a hit with tangent direction (0, 1) on a cylinder: rows of P's triangle, V
    float t[21], vu, vv;
    auto at = [&](int i, int j) { return i > j ? t[i * (i + 1) / 2 + j] : t[j * (j + 1) / 2 + i]; };
    for (;;) {
        for (float &x : t)
            if (std::scanf("%a", &x) != 1) return 0;
        if (std::scanf("%a %a", &vu, &vv) != 2) return 1;
        const pair32 Suu = two_sum(at(1, 1), vu), Svv = two_sum(at(2, 2), vv), Suv = {at(1, 2), 0.f};
        const pair32 uv2 = mul(Suv, Suv), det = add(mul(Suu, Svv), pair32{-uv2.h, -uv2.l}), id = recip(det);
        const pair32 i00 = mul(Svv, id), i11 = mul(Suu, id), m01 = mul(Suv, id), i01 = {-m01.h, -m01.l};
        for (int i = 0; i < 6; ++i) {
            const pair32 B0 = {at(1, i), 0.f}, B1 = {at(2, i), 0.f};
            const pair32 K0 = add(mul(B0, i00), mul(B1, i01)), K1 = add(mul(B0, i01), mul(B1, i11));
            for (int j = 0; j <= i; ++j) std::printf("%a\n", minus_products(at(i, j), K0, at(1, j), K1, at(2, j)));
        }
    }
}
"""


def _inputs(disk, shrink):
    rng = np.random.default_rng(int(np.log10(shrink)))
    A = rng.normal(size=(N, 6, 6)) + 2.0 * np.eye(6)
    sd = np.array([1e-2, 1e-2, 1e-1, 1e-1, 1e-2, 1e-2])
    P = np.einsum("nik,njk,i,j->nij", A, A, sd, sd).astype(np.float32)
    iu, iv = (1, 0) if disk else (1, 2)
    var = (np.stack([P[:, iu, iu], P[:, iv, iv]], 1) / shrink * rng.uniform(1, 1.3, (N, 2))).astype(np.float32)
    return rng, P, var, iu, iv


def _exact(P, var, iu, iv):
    """P - B^T S^-1 B in the host's extended precision, and the bound."""
    P, var = P.astype(np.longdouble), var.astype(np.longdouble)
    Suu, Svv, Suv = P[:, iu, iu] + var[:, 0], P[:, iv, iv] + var[:, 1], P[:, iu, iv]
    det = Suu * Svv - Suv * Suv
    B0, B1 = P[:, iu, :], P[:, iv, :]
    K0 = (B0 * Svv[:, None] - B1 * Suv[:, None]) / det[:, None]
    K1 = (B1 * Suu[:, None] - B0 * Suv[:, None]) / det[:, None]
    # as (I - K H) P (I - K H)^T + K V K^T: no cancellation of the size of P
    IKH = np.tile(np.eye(6, dtype=np.longdouble), (N, 1, 1))
    IKH[:, :, iu] -= K0
    IKH[:, :, iv] -= K1
    T = sum(IKH[:, :, k, None] * P[:, None, k, :] for k in range(6))
    ref = sum(T[:, :, k, None] * IKH[:, None, :, k] for k in range(6))
    ref = ref + K0[:, :, None] * K0[:, None, :] * var[:, 0, None, None] + K1[:, :, None] * K1[:, None, :] * var[:, 1, None, None]
    sig = np.sqrt(np.einsum("nii->ni", P))
    made_of = sig[:, :, None] * sig[:, None, :] / (1 - Suv ** 2 / (Suu * Svv))[:, None, None]
    return ref, np.longdouble(2) ** -24 * np.abs(ref) + np.longdouble(2) ** -49 * made_of


@pytest.mark.parametrize("shrink", [1e6, 1e9])
def test_the_bound_is_beyond_pairs_of_floats(tmp_path, shrink):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("needs g++")
    (tmp_path / "u.cpp").write_text(PROGRAM)
    inc = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "include")
    subprocess.check_call([gxx, "-O1", "-std=c++17", "-ffp-contract=off", "-I", CSRC, "-I", inc, str(tmp_path / "u.cpp"), "-o",
                           str(tmp_path / "u")])
    _, P, var, iu, iv = _inputs(False, shrink)
    rows = "\n".join(" ".join(float(x).hex() for x in [*(P[n, i, j] for i, j in TRI), *var[n]]) for n in range(N))
    out = subprocess.run([str(tmp_path / "u")], input=rows, capture_output=True, text=True, check=True).stdout.split()
    got = np.array([float.fromhex(x) for x in out]).reshape(N, 21)
    ref, bound = _exact(P, var, iu, iv)
    worst = max(float(np.max(np.abs(got[:, k] - ref[:, i, j]) / bound[:, i, j])) for k, (i, j) in enumerate(TRI))
    assert worst > 1.0, worst  # what the update on the device is held to


@pytest.mark.gpu
@pytest.mark.parametrize("disk", [False, True], ids=["cylinder", "disk"])
@pytest.mark.parametrize("shrink", [1e6, 1e9])
def test_large_shrinks_are_updated_in_double(disk, shrink):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from _gpu import device_tracks, unpack_cov
    from paper_1702_06359_gb300 import tkf
    rng, P, var, iu, iv = _inputs(disk, shrink)
    p = (rng.normal(size=(N, 6)) * 0.1 + np.array([1, 0, 0.5, 0.3, 0.1, 1.3])).astype(np.float32)
    z = (p[:, 2] + rng.normal(size=N) * 0.1).astype(np.float32)
    one = torch.ones(N, device="cuda")
    t = lambda a: torch.as_tensor(np.ascontiguousarray(a), device="cuda")  # noqa: E731
    hits = tkf.DeviceHits(one, 0 * one, t(z), t(var[:, 0]), t(var[:, 1]), torch.full((N,), L - 1, dtype=torch.int32, device="cuda"),
                          torch.tensor([0, N], dtype=torch.int32, device="cuda"))
    ids = np.full((N, L), -1, dtype=np.int32)
    ids[:, L - 1] = np.arange(N)
    cfg = dict(radius=(40.0,) * L, disk_z=[8.0 * (l + 1) for l in range(L)]) if disk else {}
    ctx = tkf.Context(tkf.default_config(precision=tkf.MIXED, **cfg))
    init = device_tracks(p.astype(np.float64), P.astype(np.float64), np.zeros(N), np.full(N, 9), ids, precision=tkf.MIXED)
    out = tkf.DeviceTracks.empty(N, L, tkf.MIXED)
    ctx.fit(hits, init, L - 1, L - 1, out)
    ctx.sync_status()
    ctx.close()
    assert torch.all(out.nhits == 10)
    ref, bound = _exact(P, var, iu, iv)
    got = unpack_cov(out.cov.double().cpu().numpy())
    worst = float(np.max(np.abs(got - ref) / bound))
    assert worst <= 1.0, worst
