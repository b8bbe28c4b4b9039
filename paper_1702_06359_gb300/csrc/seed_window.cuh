// Where the hits of a seed can lie in azimuth: the windows of the seeding search (tkf_seeding.cu), shared
// with a host test that samples circles.
//
// Notation: a circle of signed curvature k whose signed distance from the beam line is d0 (the origin's
// power divided by the diameter) crosses the radius r at an angle chi to the radial direction with sin chi =
// k r / 2 - d0 / r, so |sin chi| <= S(r) = |k| r / 2 + |d0| / r, which is convex in r.  While S < 1 it crosses
// every radius twice, once on each of its two branches, and moves outwards along a branch.
//
// Branches.  Two points of one circle on different branches, at radii p and q, are at least opposite(p, q)
// apart: the azimuth of a branch from the direction of the circle's centre is at least acos(S / m), where
// m^2 = 1 - 2 |k d0| bounds the centre's distance from below.  Where that exceeds the chord limit, the
// chord cut leaves one branch.
//
// Layer 2.  Let ab be the chord of the first two hits.  The circles through both are a pencil with one
// parameter t, k = 2 sin(t) / ab, and the power of any point p over the diameter is
// (pa pb / ab) sin(t - t_p): for the origin, d0 = (ra rb / ab) sin(t - t01), with t01 the circle through the
// beam line.  So |d0| <= D means |t - t01| <= asin(u), u = D ab / (ra rb), and k is within 2 asin(u) / ab of
// k01.  The point at radius r moves by (pa pb / ab) / (r cos chi) in azimuth per unit of t, and on one branch
// pa <= (r - ra) / C, pb <= (r - rb) / C with C the smallest cos chi on the way: the crossing of layer
// 2 lies within D (r - ra) (r - rb) / (ra rb r) (asin(u) / u) / C^3 of that of the circle through the beam line.
//
// Layer 3.  The triplet's circle is known; in the angle h from its centre's direction f = k r U (cos h0 -
// cos h) for a point at radius r (U the centre's distance, h0 the crossing), so |f| <= w means
// |h - h0| <= w / (r k U sin), sin the smallest on the way.
#pragma once

#include <cuda_runtime.h>
#include <math.h>

namespace tkf {

// Limits of the windows, made by seed_windows; a k limit below 0: always the whole row.
struct SeedWindows {
    float hit_dr, kmax, d0, w3;
    float R2, R3, inv_lo[2];  // radii of layers 2 and 3; 1 / (R - hit_dr)
    float s0;                 // d0 over the smallest radius of layer 0
    float k2, k3;             // largest curvature for which layer 2's and layer 3's windows hold
    int one_branch;           // whether layer 1's does
    float ic2;                // 1 / C of layer 2 at kmax, where that is small; 0: by each pair's curvature
};

constexpr float kWholeRow = 4.f;  // half width of a window that is the whole row

#ifdef __CUDACC__
#define TKF_WIN __host__ __device__ __forceinline__
#else
#define TKF_WIN inline
#endif

// asin(x) for a window's centre: the series to x^7 is within 4e-6 below 0.35
TKF_WIN float asin_near(float x)
{
    const float q = x * x;
    return fabsf(x) < 0.35f ? x * (1.f + q * (1.f / 6.f + q * (3.f / 40.f + q * (15.f / 336.f)))) : asinf(x);
}

TKF_WIN float win_rsqrt(float x)
{
#ifdef __CUDA_ARCH__
    return rsqrtf(x);
#else
    return 1.f / sqrtf(x);
#endif
}

// Half width of the layer-1 window around the azimuth of a first hit at radius ra; rhi: the layer's outer radius.
TKF_WIN float half_layer1(const SeedWindows &g, float rhi, float ra)
{
    const float s = g.kmax * rhi * 0.5f;
    return g.one_branch && s < 1.f ? asinf(s) - asinf(g.kmax * ra * 0.5f) + 2e-3f : kWholeRow;
}

// The layer-2 window of a pair at radii ra, rb with curvature k01 through the beam line: half width, and
// its centre relative to the first hit's azimuth.  The factors 1.1 and 0.75 are 1 (times asin(u) / u, below 1.05
// here) and 0.5 in exact arithmetic; the roundings of the azimuths and of the centre are below 2e-5 rad.
TKF_WIN float half_layer2(const SeedWindows &g, float ra, float rb, float k01, float &mid)
{
    mid = 0.f;
    const float inv = 1.f / (ra * rb), hi = g.R2 + g.hit_dr, lever = (hi - ra) * (hi - rb) * inv;
    float ic = g.ic2;
    if (ic == 0.f) {
        const float k = fminf(g.kmax, fabsf(k01) + 2.1f * g.d0 * inv);  // 2.1: 2 asin(u) / u
        if (!(k <= g.k2)) return kWholeRow;
        const float s = 0.5f * k * hi + g.s0;  // at least S between the first hit and layer 2
        ic = win_rsqrt(1.f - s * s);
    }
    mid = asin_near(k01 * g.R2 * 0.5f) - asin_near(k01 * ra * 0.5f);
    return (1.1f * g.d0 * lever * (ic * ic * ic) + 0.002f) * g.inv_lo[0] + 0.75f * g.hit_dr * fabsf(k01) * ic + 1e-4f;
}

// Half width of the layer-3 window around the crossing of the triplet's circle (curvature k > 0, signed
// distance d0) with layer 3.
TKF_WIN float half_layer3(const SeedWindows &g, float k, float d0)
{
    if (!(k <= g.k3)) return kWholeRow;
    const float hi = g.R3 + g.hit_dr, lo = g.inv_lo[1];
    const float iu = win_rsqrt(1.f + 2.f * k * d0);  // 1 / (k U)
    const float s = (0.5f * k * hi + (fabsf(d0) + g.w3) * lo) * iu, ic = win_rsqrt(1.f - s * s) * iu;
    return (1.25f * g.w3 * ic + 0.005f) * lo + g.hit_dr * ic * (0.75f * k + 1.25f * fabsf(d0) * lo * lo) + 3e-4f;
}

// radius: of layers 0 .. 3.
inline SeedWindows seed_windows(const double *radius, double hit_dr, double kmax, double d0, double w3)
{
    SeedWindows g{};
    g.hit_dr = (float)hit_dr;
    g.kmax = (float)kmax;
    g.d0 = (float)d0;
    g.w3 = (float)w3;
    g.R2 = (float)radius[2];
    g.R3 = (float)radius[3];
    g.inv_lo[0] = (float)(1.0 / (radius[2] - hit_dr));
    g.inv_lo[1] = (float)(1.0 / (radius[3] - hit_dr));
    g.s0 = (float)(d0 / (radius[0] - hit_dr));
    double lim[3];
    for (int l = 0; l < 3; ++l) lim[l] = 2.0 * (radius[l + 1] - radius[l]);
    // whether points of one circle (curvature up to k, distance up to d, passing within w of the outer one) on
    // layers l and l + 1 are on one branch if their chord is within the limit, crossing at S <= 0.9
    auto one_branch = [&](int l, double k, double d, double w) {
        const double m2 = 1.0 - 2.0 * k * (d + w);
        if (!(m2 > 0.0)) return false;
        for (int i = 0; i <= 8; ++i)
            for (int j = 0; j <= 8; ++j) {
                const double p = radius[l] + hit_dr * (i - 4) / 4.0, q = radius[l + 1] + hit_dr * (j - 4) / 4.0;
                const double sp = (0.5 * k * p + d / p) / sqrt(m2), sq = (0.5 * k * q + (d + w) / q) / sqrt(m2);
                if (!(sp <= 0.9 && sq <= 0.9)) return false;
                const double far = p * p + q * q + 2.0 * p * q * (sqrt((1.0 - sp * sp) * (1.0 - sq * sq)) - sp * sq);
                if (!(far > 1.01 * lim[l] * lim[l])) return false;
            }
        return true;
    };
    auto largest = [&](auto holds) {  // curvature up to kmax (holds: for every smaller one as well)
        if (!holds(0.0)) return -1.f;
        if (holds(kmax)) return g.kmax;
        double lo = 0.0, hi = kmax;
        for (int i = 0; i < 40; ++i) {
            const double mid = 0.5 * (lo + hi);
            (holds(mid) ? lo : hi) = mid;
        }
        return (float)lo * 0.999f;
    };
    g.one_branch = one_branch(0, kmax, 0.0, 0.0);
    // (asin(u) <= 1.05 u, and the pencil's parameters of two allowed circles less than pi apart)
    const bool small = d0 * lim[0] <= 0.5 * (radius[0] - hit_dr) * (radius[1] - hit_dr);
    g.k2 = largest([&](double k) {
        return small && 0.5 * k * lim[0] <= 0.95 && 0.5 * k * (radius[2] + hit_dr) + d0 / (radius[0] - hit_dr) <= 0.95 &&
               one_branch(0, k, d0, 0.0) && one_branch(1, k, d0, 0.0);
    });
    const double s2 = 0.5 * kmax * (radius[2] + hit_dr) + d0 / (radius[0] - hit_dr);
    if (g.k2 == g.kmax && s2 < 0.3) g.ic2 = (float)(1.0 / sqrt(1.0 - s2 * s2));
    g.k3 = largest([&](double k) { return one_branch(2, k, d0, w3); });
    return g;
}
#undef TKF_WIN

}  // namespace tkf
