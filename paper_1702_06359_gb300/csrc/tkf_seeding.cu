// Seeding from hit triplets on layers 0, 1, 2 with a confirmation hit on layer 3 (the seeding
// stage of Sec. 2, which the paper names without specifying): tkf_find_seeds.
//
// For each layer-0 hit the search takes the layer-1 cells of the hit index (eta row, phi sixteenths)
// that a circle from the beam line through the hit can reach with |curvature| <= kappa_max and a
// z-vertex within z_vertex; for every pair that passes, the layer-2 window around the pair's
// extrapolation; for every triplet that passes, the layer-3 window around the triplet circle's
// crossing.  The windows on layers 2 and 3 are read from grids of their own (k_seed_grid).  The
// windows only choose which hits are read; every hit in them is tested against the exact cuts, so
// the seeds are those of a scan over all hits of the layers.  A warp shares its first hits' work out
// over its lanes through queues in shared memory (k_seed_find); the lane of each layer-0 hit keeps
// that hit's triplet of smallest score.  Seeds are then compacted in the index order of their first
// hits (event by event, eta-phi cell by cell), which keeps a warp's seeds near one another for the
// building that follows.
//
// Circle quantities are evaluated in the frame of the first hit a: with b' = b - a and
// c' = c - a, the circle through a, b, c has centre a + w / (2 det) (det = b' x c',
// w = (c'_y |b'|^2 - b'_y |c'|^2, b'_x |c'|^2 - c'_x |b'|^2)), curvature 2 |det| / |w| and unit
// normal n = sign(det) w / |w|, and a point p lies at f(p) = kappa |p - a|^2 / 2 - (p - a) . n
// from it (the point's power divided by the diameter).  None of these subtracts two numbers
// of the size of the radius, so they keep FP32 accuracy for the straight tracks of high pT.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <string>

#include "internal.h"
#include "kf_math.cuh"
#include "seed_window.cuh"

using namespace tkf;

namespace {

constexpr int kSeedThreads = 256;
constexpr int kFindThreads = 128;
constexpr float kInf = 3.0e38f;

struct SeedGeom {
    int L, n_eta, n_phi, n_bins, n_events;
    float R[4];           // radii of layers 0..3
    float eta_min, inv_eta_w, phi_scale;
    float kmax;           // curvature limit
    float zv, d0, dz, w3, z3;
    float lim01, lim12, lim23;  // transverse chord limits 2 (R_{l+1} - R_l)
    float hit_dr;
    SeedWindows win;
    float aspect[2];  // z extent of a layer-2 / layer-3 window over its phi extent
    int confirm;
};

// a b + c d with the first product fused: written out where the cuts and the score are formed, so
// that no decision depends on how the compiler would contract the sum in the code around it
__device__ __forceinline__ float dot2(float a, float b, float c, float d) { return fmaf(a, b, __fmul_rn(c, d)); }

__device__ __forceinline__ int seed_find_event(const int *off, int n_events, int i)
{  // largest e with off[e] <= i
    int lo = 0, hi = n_events;
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (__ldg(&off[mid]) <= i) lo = mid; else hi = mid;
    }
    return lo;
}

// eta bins [b0, b1] of z in [z_lo, z_hi] on the cylinder of radius R (eta = asinh(z / R)), with
// 1e-3 of slack in eta for the index's own rounding
__device__ __forceinline__ void eta_bins(const SeedGeom &g, float R, float z_lo, float z_hi, int &b0, int &b1)
{
    auto eta = [&](float z) {
        const float t = z / R, at = fabsf(t);
        return copysignf(fast_log(at + sqrtf(at * at + 1.f)), t);
    };
    b0 = (int)floorf((eta(z_lo) - 1e-3f - g.eta_min) * g.inv_eta_w);
    b1 = (int)floorf((eta(z_hi) + 1e-3f - g.eta_min) * g.inv_eta_w);
    b0 = max(0, min(b0, g.n_eta - 1));
    b1 = max(0, min(b1, g.n_eta - 1));
}

// The phi window [phi - half, phi + half] as at most two runs of consecutive (phi bin, phi
// sixteenth) cells of an eta row (two when it wraps around phi = +-pi): run r covers cells
// lo[r] .. hi[r], a cell numbered bin * kSubBins + sixteenth (hi < lo: empty).
struct PhiWin {
    int lo[2], hi[2];
};

__device__ __forceinline__ PhiWin phi_window(const SeedGeom &g, float phi, float half)
{
    PhiWin w;
    w.lo[1] = 0;
    w.hi[1] = -1;
    const float tp = 2.f * (float)kPi;
    phi -= tp * floorf((phi + (float)kPi) / tp);  // into [-pi, pi)
    const float c_lo = (phi - half + (float)kPi) * g.phi_scale, c_hi = (phi + half + (float)kPi) * g.phi_scale;
    const int nphi = g.n_phi, last = nphi * kSubBins - 1;
    if (!(c_hi - c_lo < (float)(nphi - 1)) || !(c_lo > (float)-nphi) || !(c_hi < (float)(2 * nphi))) {
        w.lo[0] = 0;  // the whole row
        w.hi[0] = last;
        return w;
    }
    const int k0 = (int)floorf(c_lo), k1 = (int)floorf(c_hi);
    const int s0 = min(max((int)floorf((c_lo - (float)k0) * (float)kSubBins), 0), kSubBins - 1);
    const int s1 = min(max((int)floorf((c_hi - (float)k1) * (float)kSubBins), 0), kSubBins - 1);
    if (k0 < 0) {
        w.lo[0] = (k0 + nphi) * kSubBins + s0;
        w.hi[0] = last;
        w.hi[1] = k1 * kSubBins + s1;
    } else if (k1 >= nphi) {
        w.lo[0] = k0 * kSubBins + s0;
        w.hi[0] = last;
        w.hi[1] = (k1 - nphi) * kSubBins + s1;
    } else {
        w.lo[0] = k0 * kSubBins + s0;
        w.hi[0] = k1 * kSubBins + s1;
    }
    return w;
}

// start of phi sixteenth t (1 <= t < kSubBins) of a bin from its packed bin_sub word (byte t - 1)
__device__ __forceinline__ int sixteenth_start(const uint4 w, int t)
{
    const unsigned word = t <= 4 ? w.x : (t <= 8 ? w.y : (t <= 12 ? w.z : w.w));
    return (int)((word >> (8 * ((t - 1) & 3))) & 0xFFu);
}

// the positions of one run of cells lo .. hi of the phi window in eta row eb of segment seg
__device__ __forceinline__ int2 run_range(const SeedGeom &g, const int *bin_off, const uint4 *bin_sub, int seg, int eb,
                                          int lo, int hi)
{
    const int row = seg * g.n_bins + eb * g.n_phi;
    const int ps0 = lo & (kSubBins - 1), ps1 = hi & (kSubBins - 1);
    const int ba = row + lo / kSubBins, bb = row + hi / kSubBins;
    const int oa = __ldg(&bin_off[ba]), ob = __ldg(&bin_off[bb]), ob1 = __ldg(&bin_off[bb + 1]);
    const uint4 wa = __ldg(&bin_sub[ba]), wb = __ldg(&bin_sub[bb]);
    return make_int2(oa + ((ps0 <= 0 || wa.w == 0xFFFFFFFFu) ? 0 : sixteenth_start(wa, ps0)),
                     ob + ((ps1 >= kSubBins - 1 || wb.w == 0xFFFFFFFFu) ? ob1 - ob : sixteenth_start(wb, ps1 + 1)));
}

// ------------------------------------------------------------------ seeding grids of layers 2 and 3
//
// The hits of one (event, layer) ordered by a grid of their own: rows of equal height in z, cells
// of equal width in phi inside a row.  The windows there are a few tenths of a cm tall and a few
// hundredths of a radian wide, far smaller than the hit index's eta bins (1.2 cm at layer 2), so
// reading them from the index meant reading every hit of those bins to fail its z cut.  A grid has
// up to four cells per hit; its rows are as many windows tall as its cells are wide.
struct SeedCells {
    float z0, inv_dz, scale;  // row = (z - z0) inv_dz, cell = (phi + pi) scale, both clamped
    int nz, nphi, tab, pad0, pad1;  // tab: first entry of the cell table (nz nphi + 1 entries)
};
constexpr int kCellsPerHit = 4;  // 160-event batch: 2.34 ms at 2, 2.18 at 4, 2.16 at 8
constexpr int kMinCells = 64;
constexpr int kMaxCells = 49152;  // the counters of a block: 192 KB of shared memory
constexpr int kGridThreads = 1024;

__host__ __device__ __forceinline__ int grid_cells(int hits)
{
    return hits < kMinCells / kCellsPerHit ? kMinCells : hits > kMaxCells / kCellsPerHit ? kMaxCells : kCellsPerHit * hits;
}
__device__ __forceinline__ int clamp_cell(float v, int n) { return max(0, min(__float2int_rd(v), n - 1)); }

// First-hit and cell-table offsets of the events (one block): first[e] = layer-0 hits of the
// events before e, cells[2 e + k].tab = cells of the grids before layer 2 + k of event e.
__global__ void __launch_bounds__(1024) k_seed_plan(const SeedGeom g, const int *bin_off, int *first, SeedCells *cells,
                                                    int *queue)
{
    __shared__ int s_a[32], s_b[32];
    __shared__ int carry_a, carry_b;
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    allow_next();
    if (tid == 0) carry_a = carry_b = *queue = 0;
    __syncthreads();
    for (int base = 0; base < g.n_events; base += blockDim.x) {
        const int e = base + tid;
        int n0 = 0, c2 = 0, c3 = 0;
        if (e < g.n_events) {
            const size_t b = (size_t)e * g.L * g.n_bins;
            n0 = bin_off[b + g.n_bins] - bin_off[b];
            const int h2 = bin_off[b + 3 * (size_t)g.n_bins] - bin_off[b + 2 * (size_t)g.n_bins];
            const int h3 = bin_off[b + 4 * (size_t)g.n_bins] - bin_off[b + 3 * (size_t)g.n_bins];
            c2 = grid_cells(h2);
            c3 = grid_cells(h3);
        }
        int a = n0, c = c2 + c3 + 2;  // each table has one entry past its cells
        if (e >= g.n_events) c = 0;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int ta = __shfl_up_sync(0xffffffffu, a, o), tc = __shfl_up_sync(0xffffffffu, c, o);
            if (lane >= o) {
                a += ta;
                c += tc;
            }
        }
        if (lane == 31) {
            s_a[w] = a;
            s_b[w] = c;
        }
        __syncthreads();
        int pa = carry_a, pb = carry_b;
        for (int k = 0; k < w; ++k) {
            pa += s_a[k];
            pb += s_b[k];
        }
        a += pa;
        c += pb;
        if (e < g.n_events) {
            first[e] = a - n0;
            cells[2 * e].tab = c - (c2 + c3 + 2);
            cells[2 * e + 1].tab = c - (c3 + 1);
        }
        __syncthreads();
        if (tid == blockDim.x - 1) {
            carry_a = a;
            carry_b = c;
        }
        __syncthreads();
    }
    if (tid == 0) first[g.n_events] = carry_a;
}

// The grid of layer 2 + blockIdx.y of event blockIdx.x, one block: the z extent, counts per cell
// in shared memory, their scan into the cell table, and the hits (x, y, z, r) with their
// event-local ids in cell order, at the positions the index gives the layer.  The order inside a
// cell is that of the atomics; no result depends on it.
__global__ void __launch_bounds__(kGridThreads, 1)
k_seed_grid(const SeedGeom g, const float4 *__restrict__ hxyzi, const int *__restrict__ bin_off, SeedCells *cells,
            int *__restrict__ tab, float4 *__restrict__ gxyzr, int *__restrict__ gid)
{
    after_previous();
    extern __shared__ int s_cnt[];
    __shared__ float s_lo[32], s_hi[32];
    __shared__ int s_part[32];
    const int e = blockIdx.x, k = blockIdx.y, tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    const unsigned full = 0xffffffffu;
    const size_t b = ((size_t)e * g.L + 2 + k) * g.n_bins;
    const int h0 = bin_off[b], h1 = bin_off[b + g.n_bins];
    float lo = 1e6f, hi = -1e6f;  // hits beyond (and NaNs) take the edge rows
    for (int i = h0 + tid; i < h1; i += kGridThreads) {
        const float z = hxyzi[i].z;
        if (fabsf(z) < 1e6f) {
            lo = fminf(lo, z);
            hi = fmaxf(hi, z);
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        lo = fminf(lo, __shfl_xor_sync(full, lo, o));
        hi = fmaxf(hi, __shfl_xor_sync(full, hi, o));
    }
    if (lane == 0) {
        s_lo[w] = lo;
        s_hi[w] = hi;
    }
    __syncthreads();
    lo = s_lo[lane];
    hi = s_hi[lane];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        lo = fminf(lo, __shfl_xor_sync(full, lo, o));
        hi = fmaxf(hi, __shfl_xor_sync(full, hi, o));
    }
    const int most = grid_cells(h1 - h0);
    const float span = fmaxf(hi - lo, 1e-3f);
    // height : width of a cell as of the layer's window; nz nphi <= most
    const float width = sqrtf(span * 2.f * (float)kPi / (g.aspect[k] * (float)most));
    SeedCells c;
    c.nz = max(1, min(__float2int_rd(span / (g.aspect[k] * width)), most / 8));
    c.nphi = most / c.nz;
    c.z0 = lo;
    c.inv_dz = (float)c.nz / span;
    c.scale = (float)c.nphi / (2.f * (float)kPi);
    c.tab = cells[2 * e + k].tab;
    c.pad0 = c.pad1 = 0;
    const int n = c.nz * c.nphi;
    for (int i = tid; i < n; i += kGridThreads) s_cnt[i] = 0;
    __syncthreads();
    auto cell_of = [&](const float4 &q) {
        return clamp_cell((q.z - c.z0) * c.inv_dz, c.nz) * c.nphi +
               clamp_cell((atan2f(q.y, q.x) + (float)kPi) * c.scale, c.nphi);
    };
    for (int i = h0 + tid; i < h1; i += kGridThreads) atomicAdd(&s_cnt[cell_of(hxyzi[i])], 1);
    __syncthreads();
    // exclusive scan: thread t owns a contiguous chunk
    const int per = (n + kGridThreads - 1) / kGridThreads, c0 = min(tid * per, n), c1 = min(c0 + per, n);
    int sum = 0;
    for (int i = c0; i < c1; ++i) sum += s_cnt[i];
    int incl = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int t = __shfl_up_sync(full, incl, o);
        if (lane >= o) incl += t;
    }
    if (lane == 31) s_part[w] = incl;
    __syncthreads();
    int run = h0 + incl - sum;
    for (int i = 0; i < w; ++i) run += s_part[i];
    for (int i = c0; i < c1; ++i) {
        const int m = s_cnt[i];
        s_cnt[i] = run;
        run += m;
    }
    __syncthreads();
    for (int i = tid; i < n; i += kGridThreads) tab[c.tab + i] = s_cnt[i];
    if (tid == 0) {
        tab[c.tab + n] = h1;
        cells[2 * e + k] = c;
    }
    __syncthreads();
    for (int i = h0 + tid; i < h1; i += kGridThreads) {
        const float4 q = hxyzi[i];
        const int pos = atomicAdd(&s_cnt[cell_of(q)], 1);
        gxyzr[pos] = make_float4(q.x, q.y, q.z, sqrtf(dot2(q.x, q.x, q.y, q.y)));
        gid[pos] = __float_as_int(q.w);
    }
}

// A window of a grid: rows z0 .. z1, in each the cells lo[r] .. hi[r] of up to two runs (two when
// the window wraps around phi = +-pi; hi < lo: none).
struct GridWin {
    int r0, r1, lo0, hi0, hi1;  // the second run, if any, starts at cell 0
    int back;                   // r0, for the second run
};

__device__ __forceinline__ GridWin grid_window(const SeedCells &c, float z, float wz, float phi, float half)
{
    GridWin w;
    // a slack of 2e-3 rows and cells covers the rounding of both coordinates
    const float zr = (z - c.z0) * c.inv_dz, wr = wz * c.inv_dz + 2e-3f;
    w.r0 = clamp_cell(zr - wr, c.nz);
    w.r1 = clamp_cell(zr + wr, c.nz);
    w.back = w.r0;
    const float mid = (phi + (float)kPi) * c.scale, wc = half * c.scale + 2e-3f, n = (float)c.nphi;
    const float a = mid - wc, b = mid + wc;
    w.lo0 = __float2int_rd(a);
    w.hi0 = __float2int_rd(b);
    w.hi1 = -1;
    if (!(a >= 0.f && b < n)) {  // reaches phi = +-pi: two runs, or the whole row
        if (!(b - a < n - 1.f) || !(a > -n) || !(b < 2.f * n)) {
            w.lo0 = 0;
            w.hi0 = c.nphi - 1;
        } else {
            const int sh = a < 0.f ? c.nphi : (a >= n ? -c.nphi : 0);
            const int i0 = w.lo0 + sh, i1 = w.hi0 + sh;  // 0 <= i0 < nphi
            w.lo0 = i0;
            w.hi0 = min(i1, c.nphi - 1);
            w.hi1 = i1 - c.nphi;  // negative: no second run
        }
    }
    return w;
}

// The hits of cells lo .. hi of rows r and r + 1 (r + 1 <= r1; one row if r = r1), as one sequence.
struct RowPair {
    int p0, n0, p1, n;  // the first row's positions p0 .. p0 + n0 - 1; sequence index i >= n0 is at p1 + i
    bool second;
    __device__ __forceinline__ int at(int i) const { return i + (i < n0 ? p0 : p1); }
};
__device__ __forceinline__ RowPair row_pair(const int *__restrict__ tab, const SeedCells &c, int r, int r1, int lo, int hi)
{
    const int *row = tab + c.tab + r * c.nphi;
    const int step = r < r1 ? c.nphi : 0;
    RowPair w;
    w.p0 = __ldg(&row[lo]);
    w.p1 = __ldg(&row[step + lo]);
    w.n0 = __ldg(&row[hi + 1]) - w.p0;
    w.n = w.n0 + (step ? __ldg(&row[step + hi + 1]) - w.p1 : 0);
    w.p1 -= w.n0;
    w.second = false;
    return w;
}

// Ranges of layer-1 positions a lane has ahead of it, refilled kRanges at a time.
constexpr int kRanges = 10;
// Queues of one warp: layer-2 hits within a pair's chord and z cuts waiting for the circle through
// the three, passing triplets waiting for their confirmation scan.  `slot` is the lane of the
// pair's first hit.
constexpr int kQueueT = 64;   // both are rings: appended to at most 31 + 32 of 64,
constexpr int kQueueF = 128;  // and 31 + 64 of 128
struct WarpQueues {
    float4 a[32];  // x, y, z, r of the slot's first hit
    int4 f[kQueueF];          // slot, layer-1 position, layer-2 grid position, dz
    int4 t[kQueueT];          // slot, layer-1 position, layer-2 grid position, score
    float4 circle[kQueueT];   // its circle: curvature, normal, d0
    int2 range[kRanges][32];
    int grid[32];  // 2 event
    int4 win[32];  // the layer-1 window's two runs of cells
    int3 rows[32]; // its next eta row, last row, and whether the second run is next
};

__device__ __forceinline__ SeedCells load_cells(const SeedCells *p)
{
    const float4 a = __ldg((const float4 *)p);
    const int2 b = __ldg((const int2 *)p + 2);
    SeedCells c;
    c.z0 = a.x;
    c.inv_dz = a.y;
    c.scale = a.z;
    c.nz = __float_as_int(a.w);
    c.nphi = b.x;
    c.tab = b.y;
    return c;
}

// The search.  G consecutive lanes share a first hit, each walking every G-th eta row of its layer-1
// window (G > 1 when there are too few first hits to fill the GPU).  In every step each lane takes
// the next layer-1 hit of its rows, makes the pair's cuts, and reads the pair's window of the
// layer-2 grid, two hits at a time; the hits within the chord and z cuts are queued and go through
// the circle cuts 32 at a time, the passing triplets through the layer-3 confirmation 32 at a time,
// each result folded into the best triplet of its first hit's lane.  Warps take tiles of 32 / G
// first hits from a queue.  Every lane reaches the warp-wide operations: the loops around them are
// warp-uniform, and the lanes without work carry their flags through them.
//
// What bounds it: instruction issue and the latency of gathered 16-byte reads together (55 % issue
// active, half of the L1 sectors hit).  On the 160-event batch (880 k first hits, 48 M passing
// pairs) it takes 2.3 M steps of about 480 instructions; reading the layer-2 windows from the hit
// index took 2.9 G instructions, this 1.1 G: 4.13 -> 1.83 ms, 640 events 16.0 -> 7.0 ms, one
// event of 3000 tracks 169 -> 57 us.  5 blocks of 128 threads per SM (88 registers): 4 blocks 2.13
// ms, 6 1.95 ms (the L1 that is left to the hits shrinks with the queues' shared memory); a pair's
// hit loaded one step ahead 1.91 ms.
constexpr int kFindBlocksPerSM = 5;
template <int G>
__global__ void __launch_bounds__(kFindThreads, kFindBlocksPerSM)
k_seed_find(const SeedGeom g, const float4 *__restrict__ hxyzi, const int *__restrict__ bin_off,
            const uint4 *__restrict__ bin_sub, const int *__restrict__ ev_off, const int *__restrict__ first,
            const SeedCells *__restrict__ cells, const int *__restrict__ tab, const float4 *__restrict__ gxyzr,
            const int *__restrict__ gid, int *queue, int *__restrict__ res_b, int *__restrict__ res_c,
            float *__restrict__ res_s)
{
    __shared__ WarpQueues s_q[kFindThreads / 32];
    const unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const unsigned below = (1u << lane) - 1u;
    WarpQueues &q = s_q[threadIdx.x >> 5];
    const int n_first = __ldg(&first[g.n_events]);
    const float lim12sq = g.lim12 * g.lim12;

    while (true) {
        int tile = 0;
        if (lane == 0) tile = atomicAdd(queue, 1);
        tile = __shfl_sync(full, tile, 0);
        const int t0 = tile * (32 / G);
        if (t0 >= n_first || t0 < 0) return;
        const int t = t0 + lane / G;

        // this lane's first hit
        bool valid = false;
        int e = 0;
        float ax = 0.f, ay = 0.f, az = 0.f, ra = 1.f, pha = 0.f;
        if (t < n_first) {
            e = seed_find_event(first, g.n_events, t);
            const int seg0 = e * g.L;
            const float4 A = hxyzi[__ldg(&bin_off[(size_t)seg0 * g.n_bins]) + t - __ldg(&first[e])];
            ax = A.x; ay = A.y; az = A.z;
            ra = sqrtf(dot2(ax, ax, ay, ay));
            valid = ra > 1e-6f;  // a hit on the beam line starts no seed
            if (!valid) ra = 1.f;
            pha = atan2f(ay, ax);
        }
        q.a[lane] = make_float4(ax, ay, az, ra);
        q.grid[lane] = 2 * e;
        const SeedCells c2 = load_cells(&cells[2 * e]);
        float best_s = kInf;
        int best_b = 0x7fffffff, best_c = 0x7fffffff;

        // layer-1 window: circles from the beam line through a with |kappa| <= kmax, z-vertex cut
        int row = 0, row_end = -1;
        if (valid) {
            const float R1 = g.R[1];
            const float rlo = R1 - g.hit_dr, rhi = R1 + g.hit_dr;
            const float zpad = 1e-3f + 1e-5f * fabsf(az);
            const float zc_lo = fminf(az * rlo / ra - g.zv * (rlo / ra - 1.f), az * rhi / ra - g.zv * (rhi / ra - 1.f));
            const float zc_hi = fmaxf(az * rlo / ra + g.zv * (rlo / ra - 1.f), az * rhi / ra + g.zv * (rhi / ra - 1.f));
            eta_bins(g, R1, zc_lo - zpad, zc_hi + zpad, row, row_end);
            const PhiWin w1 = phi_window(g, pha, half_layer1(g.win, rhi, ra));
            q.win[lane] = make_int4(w1.lo[0], w1.hi[0], w1.lo[1], w1.hi[1]);
            row += lane % G;
        }
        q.rows[lane] = make_int3(row, row_end, 0);
        int j = 0, jend = 0, n_r = 0, i_r = 0;  // the range being read; ranges held, ranges taken
        __syncwarp();

        // queued layer-2 candidates and triplets and the heads of their rings (warp-uniform)
        int n_f = 0, n_t = 0, h_f = 0, h_t = 0;

        // the confirmation scan of the first cnt queued triplets, one per lane, folded into the
        // best triplet of each slot (held by the slot's lane)
        auto confirm = [&](int cnt) {
            const bool has = lane < cnt;
            int ts = 0, b_id = 0, c_id = 0;
            float s = kInf;
            if (has) {
                const int k = (h_t + lane) & (kQueueT - 1);
                const int4 T = q.t[k];
                ts = T.x;
                const float s2 = __int_as_float(T.w);
                const float4 B = hxyzi[T.y], Cc = gxyzr[T.z];
                b_id = __float_as_int(B.w);
                c_id = __ldg(&gid[T.z]);
                if (!g.confirm) {
                    s = s2;
                } else {
                    const float4 A = q.a[ts];
                    const float kap = q.circle[k].x, nx = q.circle[k].y, ny = q.circle[k].z, d0 = q.circle[k].w;
                    const float rb = sqrtf(dot2(B.y, B.y, B.x, B.x)), rc = Cc.w;
                    if (rc != rb) {
                        const float slope23 = (Cc.z - B.z) / (rc - rb);
                        const float half = half_layer3(g.win, kap, d0), R3 = g.R[3];
                        float ph3 = 0.f;
                        if (half < kWholeRow) {
                            // where the circle crosses r = R3 nearest to c: its centre is U = a + rho n, and
                            // the crossing lies along U at (R3^2 + 2 rho d0) / (2 |U|) (|U|^2 - rho^2 = 2 rho d0)
                            const float rho = 1.f / kap;
                            const float ux = A.x + rho * nx, uy = A.y + rho * ny;
                            const float D = sqrtf(ux * ux + uy * uy);
                            const float along = (R3 * R3 + 2.f * rho * d0) / (2.f * D);
                            const float h = sqrtf(fmaxf(R3 * R3 - along * along, 0.f)), ex = ux / D, ey = uy / D;
                            const float px1 = along * ex - h * ey, py1 = along * ey + h * ex;
                            const float px2 = along * ex + h * ey, py2 = along * ey - h * ex;
                            const bool near1 = (px1 - Cc.x) * (px1 - Cc.x) + (py1 - Cc.y) * (py1 - Cc.y) <=
                                               (px2 - Cc.x) * (px2 - Cc.x) + (py2 - Cc.y) * (py2 - Cc.y);
                            ph3 = atan2f(near1 ? py1 : py2, near1 ? px1 : px2);
                        }
                        const float zc3 = B.z + slope23 * (R3 - rb);
                        const float wz = g.z3 + 1e-3f + 1e-5f * fabsf(zc3) + g.hit_dr * fabsf(slope23);
                        const SeedCells c3 = load_cells(&cells[q.grid[ts] + 1]);
                        const GridWin w3 = grid_window(c3, zc3, wz, ph3, half);
                        float c3s = kInf;
                        for (int r = w3.r0; r <= w3.r1; r += 2) {
                            RowPair rp = row_pair(tab, c3, r, w3.r1, w3.lo0, w3.hi0);
                            for (int i = 0;; ++i) {
                                if (i >= rp.n) {  // the window's second run, if it has one
                                    if (w3.hi1 < 0 || rp.second) break;
                                    rp = row_pair(tab, c3, r, w3.r1, 0, w3.hi1);
                                    rp.second = true;
                                    i = -1;
                                    continue;
                                }
                                const float4 E = gxyzr[rp.at(i)];
                                const float d23x = E.x - Cc.x, d23y = E.y - Cc.y;
                                if (!(sqrtf(d23x * d23x + d23y * d23y) <= g.lim23)) continue;
                                const float qx = E.x - A.x, qy = E.y - A.y;
                                const float f3 = kap * dot2(qx, qx, qy, qy) * 0.5f - dot2(qx, nx, qy, ny);
                                const float re = E.w;
                                const float dz3 = E.z - (B.z + slope23 * (re - rb));
                                if (!(fabsf(f3) <= g.w3) || !(fabsf(dz3) <= g.z3)) continue;
                                const float pu = f3 / g.w3, pv = dz3 / g.z3;
                                c3s = fminf(c3s, dot2(pu, pu, pv, pv));
                            }
                        }
                        if (c3s < kInf) s = s2 + c3s;
                    }
                }
            }
            unsigned m = __ballot_sync(full, s < kInf);
            while (m) {
                const int k = __ffs(m) - 1;
                m &= m - 1u;
                const int ks = __shfl_sync(full, ts, k), kb = __shfl_sync(full, b_id, k), kc = __shfl_sync(full, c_id, k);
                const float kv = __shfl_sync(full, s, k);
                if (lane == ks && (kv < best_s || (kv == best_s && (kb < best_b || (kb == best_b && kc < best_c))))) {
                    best_s = kv;
                    best_b = kb;
                    best_c = kc;
                }
            }
            h_t += cnt;
            n_t -= cnt;
            __syncwarp();
        };

        // the circle through the first cnt queued candidates (a, b, c), one per lane: curvature and
        // d0 cuts and the score without confirmation; passing triplets join the triplet queue
        auto circle = [&](int cnt) {
            const bool has = lane < cnt;
            int fs = 0, fb = 0, fc = 0;
            float dz = 0.f;
            if (has) {
                const int4 F = q.f[(h_f + lane) & (kQueueF - 1)];
                fs = F.x; fb = F.y; fc = F.z; dz = __int_as_float(F.w);
            }
            const float best_fs = __shfl_sync(full, best_s, fs);
            bool pass = false;
            float s2 = 0.f, kap = 0.f, nx = 0.f, ny = 0.f, d0 = 0.f;
            if (has) {
                const float4 A = q.a[fs], B = hxyzi[fb], Cc = gxyzr[fc];
                const float bx = B.x - A.x, by = B.y - A.y, cx = Cc.x - A.x, cy = Cc.y - A.y;
                const float det = dot2(bx, cy, -by, cx);
                if (det != 0.f) {
                    const float bb2 = dot2(bx, bx, by, by), cc2 = dot2(cx, cx, cy, cy);
                    const float wx = dot2(cy, bb2, -by, cc2), wy = dot2(bx, cc2, -cx, bb2);
                    const float wn = sqrtf(dot2(wx, wx, wy, wy));
                    kap = 2.f * fabsf(det) / wn;
                    const float sg = det > 0.f ? 1.f : -1.f;
                    nx = sg * wx / wn;
                    ny = sg * wy / wn;
                    d0 = kap * dot2(A.x, A.x, A.y, A.y) * 0.5f + dot2(A.x, nx, A.y, ny);
                    if (kap <= g.kmax && fabsf(d0) <= g.d0) {
                        const float u = d0 / g.d0, v = dz / g.dz;
                        s2 = dot2(u, u, v, v);
                        pass = !(s2 > best_fs);  // the confirmation term only adds
                    }
                }
            }
            const unsigned m = __ballot_sync(full, pass);
            if (pass) {
                const int k = (h_t + n_t + __popc(m & below)) & (kQueueT - 1);
                q.t[k] = make_int4(fs, fb, fc, __float_as_int(s2));
                q.circle[k] = make_float4(kap, nx, ny, d0);
            }
            n_t += __popc(m);
            h_f += cnt;
            n_f -= cnt;
            __syncwarp();
            if (n_t >= 32) confirm(32);
        };

        while (true) {
            if (j >= jend && i_r < n_r) {
                const int2 r = q.range[i_r++][lane];
                j = r.x;
                jend = r.y;
            }
            if (!__any_sync(full, j < jend)) {
                // every lane's ranges are read: the next kRanges non-empty ones of each
                int row = q.rows[lane].x, part = q.rows[lane].z;
                const int row_end = q.rows[lane].y;
                if (!__any_sync(full, row <= row_end)) break;
                const int4 w1 = q.win[lane];
                n_r = i_r = 0;
                while (__any_sync(full, row <= row_end && n_r < kRanges)) {
                    if (row <= row_end && n_r < kRanges) {
                        const int lo = part ? w1.z : w1.x, hi = part ? w1.w : w1.y;
                        if (hi >= lo) {
                            const int2 r = run_range(g, bin_off, bin_sub, (q.grid[lane] >> 1) * g.L + 1, row, lo, hi);
                            if (r.y > r.x) q.range[n_r++][lane] = r;
                        }
                        part = !part && w1.w >= w1.z;
                        if (!part) row += G;
                    }
                }
                q.rows[lane].x = row;
                q.rows[lane].z = part;
                continue;
            }
            // the next pair of this lane
            bool pass = false;
            float4 B = make_float4(0.f, 0.f, 0.f, 0.f);
            float rb = 0.f, k01 = 0.f, slope = 0.f;
            const int jb = j;
            if (j < jend) {
                ++j;
                B = hxyzi[jb];
                const float bx = B.x - ax, by = B.y - ay;
                const float chord01 = sqrtf(bx * bx + by * by);
                if (chord01 <= g.lim01 && chord01 != 0.f) {
                    rb = sqrtf(dot2(B.x, B.x, B.y, B.y));
                    k01 = 2.f * (ax * B.y - ay * B.x) / (ra * rb * chord01);
                    if (fabsf(k01) <= g.kmax && rb != ra) {
                        slope = (B.z - az) / (rb - ra);
                        pass = fabsf(az - ra * slope) <= g.zv;
                    }
                }
            }
            // its layer-2 window: z along the r-z line of a and b, phi around the crossing of the circle
            // through the beam line, a and b
            GridWin w2;
            w2.r0 = 0; w2.r1 = -1; w2.lo0 = 0; w2.hi0 = 0; w2.hi1 = -1; w2.back = 0;
            if (pass) {
                const float R2 = g.R[2];
                const float zc = az + slope * (R2 - ra);
                const float wz = g.dz + 1e-3f + 1e-5f * fabsf(zc) + g.hit_dr * fabsf(slope);
                float mid;
                const float half = half_layer2(g.win, ra, rb, k01, mid);
                w2 = grid_window(c2, zc, wz, pha + mid, half);
            }
            // two rows at a time, the few hits of both in one sequence
            while (__any_sync(full, w2.r0 <= w2.r1)) {
                RowPair rp{0, 0, 0, 0, false};
                if (w2.r0 <= w2.r1) rp = row_pair(tab, c2, w2.r0, w2.r1, w2.lo0, w2.hi0);
                auto near_z = [&](int pos, float &dz) {
                    const float4 Cc = gxyzr[pos];
                    const float d12x = Cc.x - B.x, d12y = Cc.y - B.y;
                    const float rc = Cc.w;
                    dz = Cc.z - (az + slope * (rc - ra));
                    return d12x * d12x + d12y * d12y <= lim12sq && fabsf(dz) <= g.dz;
                };
                for (int i = 0; __any_sync(full, i < rp.n); i += 2) {
                    bool k0 = false, k1 = false;
                    float dz0 = 0.f, dz1 = 0.f;
                    const int jc0 = rp.at(i), jc1 = rp.at(i + 1);
                    if (i < rp.n) k0 = near_z(jc0, dz0);
                    if (i + 1 < rp.n) k1 = near_z(jc1, dz1);
                    const unsigned m0 = __ballot_sync(full, k0), m1 = __ballot_sync(full, k1);
                    if (!(m0 | m1)) continue;
                    if (k0)
                        q.f[(h_f + n_f + __popc(m0 & below)) & (kQueueF - 1)] =
                            make_int4(lane, jb, jc0, __float_as_int(dz0));
                    n_f += __popc(m0);
                    if (k1)
                        q.f[(h_f + n_f + __popc(m1 & below)) & (kQueueF - 1)] =
                            make_int4(lane, jb, jc1, __float_as_int(dz1));
                    n_f += __popc(m1);
                    __syncwarp();
                    while (n_f >= 32) circle(32);
                }
                // the window's second run, if it wraps around phi = +-pi, after the first
                w2.r0 += 2;
                if (w2.r0 > w2.r1 && w2.hi1 >= 0) {
                    w2.r0 = w2.back;
                    w2.lo0 = 0;
                    w2.hi0 = w2.hi1;
                    w2.hi1 = -1;
                }
            }
        }
        if (n_f > 0) circle(n_f);
        if (n_t > 0) confirm(n_t);
        // the best of the G lanes of a first hit (smallest score, then ids)
#pragma unroll
        for (int o = G / 2; o > 0; o >>= 1) {
            const float os = __shfl_xor_sync(full, best_s, o);
            const int ob = __shfl_xor_sync(full, best_b, o), oc = __shfl_xor_sync(full, best_c, o);
            if (os < best_s || (os == best_s && (ob < best_b || (ob == best_b && oc < best_c)))) {
                best_s = os;
                best_b = ob;
                best_c = oc;
            }
        }
        if (t < n_first && lane % G == 0) {
            if (best_s < kInf) {
                const int base = __ldg(&ev_off[q.grid[lane] >> 1]);
                res_b[t] = base + best_b;
                res_c[t] = base + best_c;
                res_s[t] = best_s;
            } else {
                res_b[t] = -1;
            }
        }
        __syncwarp();  // the queues are the next tile's
    }
}

// Compaction of the first hits' results in their order: block b takes the b-th of gridDim.x equal
// chunks.  First the seeds per chunk, then every block adds up the chunks before its own.
constexpr int kCompactBlocks = 512;
__device__ __forceinline__ int2 chunk_of(int n)
{
    const int per = (n + gridDim.x - 1) / gridDim.x;
    const int a = (int)min((long long)blockIdx.x * per, (long long)n);
    return make_int2(a, min(a + per, n));
}
__device__ __forceinline__ int block_sum(int v, int *s_part)
{
    v = __reduce_add_sync(0xffffffffu, v);
    if ((threadIdx.x & 31) == 0) s_part[threadIdx.x >> 5] = v;
    __syncthreads();
    v = 0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) v += s_part[w];
    __syncthreads();
    return v;
}

__global__ void __launch_bounds__(kSeedThreads) k_seed_count(const int *res_b, const int *n_first, int *count)
{
    after_previous();
    allow_next();
    __shared__ int s_part[kSeedThreads / 32];
    const int2 c = chunk_of(*n_first);
    int v = 0;
    for (int t = c.x + threadIdx.x; t < c.y; t += blockDim.x) v += res_b[t] >= 0;
    v = block_sum(v, s_part);
    if (threadIdx.x == 0) count[blockIdx.x] = v;
}

__global__ void __launch_bounds__(kSeedThreads)
k_seed_scatter(const SeedGeom g, const float4 *hxyzi, const int *bin_off, const int *ev_off, const int *first,
               const int *res_b, const int *res_c, const float *res_s, const int *count, int max_seeds, int *seed_hits,
               int *seed_event, float *seed_score, int *total)
{
    after_previous();
    __shared__ int s_part[kSeedThreads / 32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    int before = 0;
    for (int b = threadIdx.x; b < (int)blockIdx.x; b += blockDim.x) before += count[b];
    int pos0 = block_sum(before, s_part);
    if (blockIdx.x == gridDim.x - 1 && threadIdx.x == 0) *total = pos0 + count[blockIdx.x];
    if (max_seeds == 0) return;
    const int2 c = chunk_of(__ldg(&first[g.n_events]));
    for (int t0 = c.x; t0 < c.y; t0 += blockDim.x) {
        const int t = t0 + threadIdx.x;
        const bool has = t < c.y && res_b[t] >= 0;
        const unsigned m = __ballot_sync(0xffffffffu, has);
        if (lane == 0) s_part[w] = __popc(m);
        __syncthreads();
        int pos = pos0 + __popc(m & ((1u << lane) - 1u));
        for (int k = 0; k < (int)(blockDim.x >> 5); ++k) {
            if (k < w) pos += s_part[k];
            pos0 += s_part[k];
        }
        __syncthreads();
        if (!has || pos >= max_seeds) continue;
        const int e = seed_find_event(first, g.n_events, t);
        const int at = __ldg(&bin_off[(size_t)e * g.L * g.n_bins]) + t - __ldg(&first[e]);
        seed_hits[pos] = __ldg(&ev_off[e]) + __float_as_int(hxyzi[at].w);
        seed_hits[(size_t)max_seeds + pos] = res_b[t];
        seed_hits[2 * (size_t)max_seeds + pos] = res_c[t];
        seed_event[pos] = e;
        if (seed_score) seed_score[pos] = res_s[t];
    }
}

int seed_fail(tkf_ctx *ctx, int code, const std::string &msg)
{
    ctx->err = msg;
    return code;
}

int seed_cuda(tkf_ctx *ctx, cudaError_t e, const char *what)
{
    return seed_fail(ctx, e == cudaErrorMemoryAllocation ? TKF_ERR_NOMEM : TKF_ERR_CUDA,
                     std::string(what) + ": " + cudaGetErrorString(e));
}

}  // namespace

namespace tkf {
void seed_scratch_free(tkf_ctx *ctx)
{
    cudaFree(ctx->seed_mem);
    ctx->seed_mem = nullptr;
    ctx->seed_b = ctx->seed_c = ctx->seed_id = ctx->seed_first = ctx->seed_tab = ctx->seed_cnt = nullptr;
    ctx->seed_s = nullptr;
    ctx->seed_xyzr = ctx->seed_cells = nullptr;
    ctx->seed_cap = ctx->seed_cap_events = ctx->seed_cap_tab = 0;
}
}  // namespace tkf

extern "C" void tkf_default_seed_cuts(tkf_seed_cuts *c)
{
    if (!c) return;
    c->pt_min = 0.5;
    c->kappa_slack = 0.15;
    c->z_vertex = 4.0;
    c->d0_max = 0.08;
    c->dz_max = 0.08;
    c->conf_rphi = 0.1;
    c->conf_z = 0.1;
    c->confirm = 1;
    c->reserved = 0;
}

extern "C" int tkf_find_seeds(tkf_ctx *ctx, const tkf_hit_index *idx, const tkf_seed_cuts *cuts, int32_t max_seeds,
                              int32_t *seed_hits, int32_t *seed_event, float *seed_score, int32_t *n_found,
                              tkf_stream stream)
{
    if (!ctx) return TKF_ERR_INVALID;
    if (!idx || !cuts || !n_found || max_seeds < 0 || (max_seeds > 0 && (!seed_hits || !seed_event)))
        return seed_fail(ctx, TKF_ERR_INVALID, "find_seeds: null argument or negative max_seeds");
    const tkf_config &c = ctx->cfg;
    if (c.n_layers < 4 || idx->n_layers != c.n_layers || idx->n_bins != c.n_eta_bins * c.n_phi_bins)
        return seed_fail(ctx, TKF_ERR_INVALID,
                         "find_seeds: needs an index of at least 4 layers built with this context's bins");
    for (int l = 0; l < 4; ++l)
        if (c.disk_z[l] > 0.0) return seed_fail(ctx, TKF_ERR_INVALID, "find_seeds: layers 0..3 must be cylinders");
    if (!(cuts->pt_min > 0) || !(cuts->kappa_slack >= 0) || !(cuts->z_vertex > 0) || !(cuts->d0_max > 0) ||
        !(cuts->dz_max > 0) || !(cuts->conf_rphi > 0) || !(cuts->conf_z > 0))
        return seed_fail(ctx, TKF_ERR_INVALID, "find_seeds: cuts must be positive");
    if (!(c.radius[0] > 0) || !(c.radius[1] > c.radius[0]) || !(c.radius[2] > c.radius[1]) ||
        !(c.radius[3] > c.radius[2]))
        return seed_fail(ctx, TKF_ERR_INVALID, "find_seeds: layers 0..3 must have increasing radii");
    cudaStream_t s = (cudaStream_t)stream;
    const int n = idx->n;
    const size_t ne = (size_t)idx->n_events;
    // every grid has at most kCellsPerHit cells per hit, kMinCells if that is more, and one entry more
    const size_t n_tab = std::min((size_t)kCellsPerHit * n + 2 * ne * (kMinCells + 1), 2 * ne * (kMaxCells + 1));
    if ((size_t)n > ctx->seed_cap || ne > ctx->seed_cap_events || n_tab > ctx->seed_cap_tab) {
        // one allocation for all of it (each takes some ten microseconds of a first call)
        const size_t cap = std::max<size_t>(std::max(n, 1), ctx->seed_cap), evs = std::max(ne, ctx->seed_cap_events),
                     tab = std::max(n_tab, ctx->seed_cap_tab);
        seed_scratch_free(ctx);
        size_t bytes = 0;
        auto part = [&](size_t count, size_t size) {
            const size_t at = bytes;
            bytes += (count * size + 255) / 256 * 256;
            return at;
        };
        const size_t xyzr = part(cap, sizeof(float4)), cells = part(2 * evs, sizeof(SeedCells)),
                     id = part(cap, sizeof(int)), res_b = part(cap, sizeof(int)), res_c = part(cap, sizeof(int)),
                     res_s = part(cap, sizeof(float)), first = part(evs + 1, sizeof(int)),
                     tabs = part(tab, sizeof(int)), cnt = part(kCompactBlocks + 1, sizeof(int));
        cudaError_t e = cudaMalloc(&ctx->seed_mem, bytes);
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(k_seed_grid, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     kMaxCells * (int)sizeof(int));
        if (e != cudaSuccess) {
            seed_scratch_free(ctx);
            return seed_cuda(ctx, e, "find_seeds: scratch");
        }
        char *m = (char *)ctx->seed_mem;
        ctx->seed_xyzr = m + xyzr;
        ctx->seed_cells = m + cells;
        ctx->seed_id = (int *)(m + id);
        ctx->seed_b = (int *)(m + res_b);
        ctx->seed_c = (int *)(m + res_c);
        ctx->seed_s = (float *)(m + res_s);
        ctx->seed_first = (int *)(m + first);
        ctx->seed_tab = (int *)(m + tabs);
        ctx->seed_cnt = (int *)(m + cnt);
        ctx->seed_cap = cap;
        ctx->seed_cap_events = evs;
        ctx->seed_cap_tab = tab;
    }
    if (n == 0) {
        cudaError_t e = cudaMemsetAsync(n_found, 0, sizeof(int32_t), s);
        return e == cudaSuccess ? TKF_OK : seed_cuda(ctx, e, "find_seeds: memset");
    }
    SeedGeom g{};
    g.L = c.n_layers;
    g.n_eta = c.n_eta_bins;
    g.n_phi = c.n_phi_bins;
    g.n_bins = c.n_eta_bins * c.n_phi_bins;
    g.n_events = idx->n_events;
    for (int l = 0; l < 4; ++l) g.R[l] = (float)c.radius[l];
    g.eta_min = (float)c.eta_min;
    g.inv_eta_w = (float)(1.0 / c.eta_bin_w);
    g.phi_scale = (float)(c.n_phi_bins / (2.0 * kPi));
    g.kmax = (float)(0.00299792458 * c.bz / cuts->pt_min * (1.0 + cuts->kappa_slack));
    g.zv = (float)cuts->z_vertex;
    g.d0 = (float)cuts->d0_max;
    g.dz = (float)cuts->dz_max;
    g.w3 = (float)cuts->conf_rphi;
    g.z3 = (float)cuts->conf_z;
    g.lim01 = (float)(2.0 * (c.radius[1] - c.radius[0]));
    g.lim12 = (float)(2.0 * (c.radius[2] - c.radius[1]));
    g.lim23 = (float)(2.0 * (c.radius[3] - c.radius[2]));
    g.hit_dr = (float)c.hit_dr;
    g.confirm = cuts->confirm != 0;
    // z extent over phi extent of the nominal windows (the grids' cells are shaped like them)
    const double lever = (c.radius[2] - c.radius[0]) * (c.radius[2] - c.radius[1]) / (c.radius[0] * c.radius[1]);
    g.win = seed_windows(c.radius, c.hit_dr, g.kmax, cuts->d0_max, cuts->conf_rphi);
    g.aspect[0] = (float)((cuts->dz_max + 1e-3) / ((1.25 * cuts->d0_max * lever + 0.005) / c.radius[2] + 3e-4));
    g.aspect[1] = (float)((cuts->conf_z + 1e-3) / ((1.25 * cuts->conf_rphi + 0.005) / c.radius[3] + 3e-4));
    SeedCells *cells = (SeedCells *)ctx->seed_cells;
    float4 *xyzr = (float4 *)ctx->seed_xyzr;
    int *queue = ctx->seed_cnt + kCompactBlocks;
    k_seed_plan<<<1, 1024, 0, s>>>(g, idx->bin_off, ctx->seed_first, cells, queue);
    cudaError_t e = launch_next(k_seed_grid, dim3((unsigned)ne, 2), kGridThreads, grid_cells(n) * sizeof(int), s, g,
                                idx->hxyzi, idx->bin_off, cells, ctx->seed_tab, xyzr, ctx->seed_id);
    // Lanes per first hit, by the tiles of 32 first hits (a layer holds about n / L hits) for each
    // warp the GPU holds.  Measured with 1 / 2 / 4 / 8 lanes: 36 tiles a warp 7.00 / 7.08 / 8.09 /
    // 10.1 ms, 9 tiles 1.86 / 1.83 / 2.04 / 2.52 ms, 0.9 tiles 507 / 306 / 288 / 308 us, a sixth of a
    // tile 150 / 102 / 82 / 81 us, a 24th 122 / 81 / 64 / 57 us.
    const long long warps = (long long)ctx->sm_count * kFindBlocksPerSM * (kFindThreads / 32);
    const long long tiles = (long long)n / c.n_layers / 32;
    auto find = [&](auto kern) {
        kern<<<ctx->sm_count * kFindBlocksPerSM, kFindThreads, 0, s>>>(
            g, idx->hxyzi, idx->bin_off, idx->bin_sub, idx->ev_off, ctx->seed_first, cells, ctx->seed_tab, xyzr,
            ctx->seed_id, queue, ctx->seed_b, ctx->seed_c, ctx->seed_s);
    };
    if (tiles >= 16 * warps)
        find(k_seed_find<1>);
    else if (tiles >= warps)
        find(k_seed_find<2>);
    else if (tiles >= warps / 8)
        find(k_seed_find<4>);
    else
        find(k_seed_find<8>);
    if (e == cudaSuccess)
        e = launch_next(k_seed_count, kCompactBlocks, kSeedThreads, 0, s, ctx->seed_b, ctx->seed_first + ne, ctx->seed_cnt);
    if (e == cudaSuccess)
        e = launch_next(k_seed_scatter, kCompactBlocks, kSeedThreads, 0, s, g, idx->hxyzi, idx->bin_off, idx->ev_off,
                        ctx->seed_first, ctx->seed_b, ctx->seed_c, ctx->seed_s, ctx->seed_cnt, max_seeds, seed_hits,
                        seed_event, seed_score, n_found);
    if (e == cudaSuccess) e = cudaGetLastError();
    return e == cudaSuccess ? TKF_OK : seed_cuda(ctx, e, "find_seeds: launch");
}
