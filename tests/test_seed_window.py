"""The azimuth windows of the seeding search (csrc/seed_window.cuh), compiled as host C++: circles of the allowed
curvatures and distances, with their hits on either branch, lie in them wherever they pass the chord cuts."""
import ctypes as C
import os
import shutil
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1702_06359_gb300", "csrc")

PROGRAM = r"""
#include "seed_window.cuh"
using namespace tkf;
extern "C" {
int size() { return (int)sizeof(SeedWindows); }
void make(const double *radius, double dr, double kmax, double d0, double w3, SeedWindows *g) { *g = seed_windows(radius, dr, kmax, d0, w3); }
void layer1(const SeedWindows *g, float rhi, int n, const float *ra, float *half)
{
    for (int i = 0; i < n; ++i) half[i] = half_layer1(*g, rhi, ra[i]);
}
void layer2(const SeedWindows *g, int n, const float *ra, const float *rb, const float *k01, float *half, float *mid)
{
    for (int i = 0; i < n; ++i) half[i] = half_layer2(*g, ra[i], rb[i], k01[i], mid[i]);
}
void layer3(const SeedWindows *g, int n, const float *k, const float *d0, float *half)
{
    for (int i = 0; i < n; ++i) half[i] = half_layer3(*g, k[i], d0[i]);
}
}
"""


@pytest.fixture(scope="module")
def win(tmp_path_factory):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("needs g++")
    d = tmp_path_factory.mktemp("win")
    (d / "win.cpp").write_text(PROGRAM)
    inc = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "include")
    subprocess.check_call([gxx, "-O1", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, "-I", inc, str(d / "win.cpp"), "-o",
                           str(d / "libwin.so")])
    return C.CDLL(str(d / "libwin.so"))


def _ptr(a):
    return a.ctypes.data_as(C.c_void_p)


def _wrap(x):
    return (x + np.pi) % (2 * np.pi) - np.pi


def _outside(win, radius, dr, kmax, d0, w3, n, rng):
    """Hits outside their windows on layers 1, 2 and 3, and how many were held by a window of less than a row."""
    R = np.array(radius, float)
    g = np.zeros(win.size(), np.uint8)
    win.make(_ptr(R), C.c_double(dr), C.c_double(kmax), C.c_double(d0), C.c_double(w3), _ptr(g))
    lim = 2 * np.diff(R)
    edge = lambda lo, p: np.where(rng.random(n) < p, rng.choice([lo, 1.0], n), rng.uniform(lo, 1, n))  # noqa: E731
    k, d = np.maximum(kmax * edge(0.0, 0.3), 1e-7), d0 * edge(-1.0, 0.3)
    rho = 1 / k
    u2 = rho * rho + 2 * rho * d  # the centre's distance squared
    real = u2 > 0
    u = np.sqrt(np.where(real, u2, 1))

    def hit(l, off=0.0):  # at f = off from the circle, the azimuth from the centre's direction
        r = R[l] + dr * edge(-1.0, 0.3)
        c = (r * r + u2 - rho * rho - 2 * rho * off) / (2 * r * u)
        return r, np.arccos(np.clip(c, -1, 1)) * rng.choice([-1, 1], n), np.abs(c) <= 1
    (ra, ha, ga), (rb, hb, gb), (rc, hc, gc) = (hit(l) for l in range(3))
    re, he, ge = hit(3, w3 * edge(-1.0, 0.3))
    chord = lambda p, hp, q, hq: np.sqrt(p * p + q * q - 2 * p * q * np.cos(hp - hq))  # noqa: E731
    ab = chord(ra, ha, rb, hb)
    k01 = 2 * np.sin(hb - ha) / ab
    pair = real & ga & gb & (ab <= lim[0]) & (np.abs(k01) <= kmax)
    trip = pair & gc & (chord(rb, hb, rc, hc) <= lim[1])
    conf = trip & ge & (chord(rc, hc, re, he) <= lim[2])
    f32 = lambda a: np.ascontiguousarray(a, np.float32)  # noqa: E731
    half1, half2, mid, half3 = np.zeros((4, n), np.float32)
    win.layer1(_ptr(g), C.c_float(R[1] + dr), n, _ptr(f32(ra)), _ptr(half1))
    win.layer2(_ptr(g), n, _ptr(f32(ra)), _ptr(f32(rb)), _ptr(f32(k01)), _ptr(half2), _ptr(mid))
    win.layer3(_ptr(g), n, _ptr(f32(k)), _ptr(f32(d)), _ptr(half3))
    cross = np.arccos(np.clip((R[3] ** 2 + u2 - rho * rho) / (2 * R[3] * u), -1, 1))
    near = np.where(np.abs(_wrap(hc - cross)) <= np.abs(_wrap(hc + cross)), cross, -cross)
    out = 0
    held = []
    for ok, off, half in ((pair, _wrap(hb - ha), half1), (trip, _wrap(hc - ha - mid), half2), (conf, _wrap(he - near), half3)):
        out += int((ok & (np.abs(off) > half)).sum())
        held.append(int((ok & (half < 3.9)).sum()))
    return out, held


RADII = [(4, 8, 12, 16), (4, 8, 20, 24), (3, 6, 16, 25), (3, 10, 13, 17), (2, 9, 30, 40), (3.1, 6.8, 10.5, 16), (4, 5, 6, 7),
         (1, 2, 4, 8), (8, 9, 20, 60)]


@pytest.mark.parametrize("radius", RADII, ids=lambda r: "-".join(map(str, r)))
@pytest.mark.parametrize("d0", [0.02, 0.08, 0.5, 1.5])
def test_windows_hold_every_circle_the_cuts_allow(win, radius, d0):
    rng = np.random.default_rng(int(100 * d0) + int(10 * sum(radius)))
    total = np.zeros(3, int)
    for pt in (0.05, 0.1, 0.2, 0.5, 2.0):
        for dr in (0.0, 0.45 * min(min(np.diff(radius)), radius[0])):
            for w3 in (0.1, 1.0):
                out, held = _outside(win, radius, dr, 0.00299792458 * 3.8 / pt * 1.15, d0, w3, 20000, rng)
                assert out == 0, (pt, dr, w3)
                total += held
    if radius == (4, 8, 12, 16):  # not by whole rows: layers of equal steps have windows at every d0 here
        assert (total > 2000).all()


def test_default_cuts_have_windows_for_every_pair_and_triplet(win):
    R, g = np.array([4.0, 8.0, 12.0, 16.0]), np.zeros(win.size(), np.uint8)
    kmax = 0.00299792458 * 3.8 / 0.5 * 1.15
    for dr in (0.0, 0.5):
        win.make(_ptr(R), C.c_double(dr), C.c_double(kmax), C.c_double(0.08), C.c_double(0.1), _ptr(g))
        half, mid = np.zeros(2, np.float32), np.zeros(2, np.float32)
        one = lambda x: _ptr(np.full(2, x, np.float32))  # noqa: E731
        win.layer2(_ptr(g), 2, one(4 - dr), one(8 + dr), one(kmax), _ptr(half), _ptr(mid))
        assert (half < 0.05).all()
        win.layer3(_ptr(g), 2, one(kmax), one(0.08), _ptr(half))
        assert (half < 0.05).all()
