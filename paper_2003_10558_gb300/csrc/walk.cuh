// walk.cuh -- the candidate triangles of a tile: every triangle of the grid
// (TriGrid) whose cap may reach the tile's view cone, found by one CTA.
//
// A fragment of triangle t at pixel direction G needs G inside the miter cap
// enlarged by the ramp half-width (the gbpxstep test of the miter plane,
// Sec. 1.1.1 / 1.1.2).  With alpha the tile's half-angle, h its widest ramp
// half-width and rho a level's largest cap radius, the caps of that level
// that reach the tile have their centres within gamma = alpha + rho + h of
// the tile's axis: cos(beta) = cos(rho) - h sin(rho) >= cos(rho + h) while
// rho + h <= pi/2, so beta <= rho + h.  (Per-fragment pixel step: rho + 4h,
// see pstep_cap.)  Walk: the rows of each level's grid within gamma of the
// axis, in each row the cells within the cap's width at that row, then the
// list; the candidates are numbered over these ranges and tested one per
// thread and step, with coalesced loads where a range is long.
#pragma once

#include "vsr_internal.cuh"

constexpr int WALK_THREADS = 128;   // threads of a walking CTA
constexpr int WALK_RANGES = 128;    // row ranges of a tile (half-angle about 0.5 rad); a wider tile takes every entry
constexpr int WALK_BLOCK = 1024;    // candidates of a block: its hits fit the CTA's list

// cells of row `row` of a grid of nlat rows: 2 nlat at the equator, falling
// towards the poles about as the row's circumference (1 + 2 (nlat^2 - x^2) /
// nlat by a 22-bit reciprocal: the same integer wherever it is computed)
__device__ __forceinline__ int grid_ncol(int nlat, int row)
{
    const uint32_t inv = nlat == 192 ? 21845u : (nlat == 96 ? 43690u : (nlat == 48 ? 87381u : 349525u));
    const int x = 2 * row + 1 - nlat;
    return max(4, min(2 * nlat, 1 + (int)(((uint32_t)(2 * (nlat * nlat - x * x)) * inv) >> 22)));
}
__device__ __forceinline__ int grid_row(float lat, int nlat)
{
    return min(nlat - 1, max(0, (int)floorf((lat + 0.5f * IDX_PI) * ((float)nlat / IDX_PI))));
}
// level l's rows / first word by a run-time level (selects, no memory)
__device__ __forceinline__ int grid_nlat_of(int l) { return l == 0 ? 192 : (l == 1 ? 96 : (l == 2 ? 48 : 12)); }
__device__ __forceinline__ int grid_base_of(int l)
{
    return l == 0 ? grid_base(0) : (l == 1 ? grid_base(1) : (l == 2 ? grid_base(2) : grid_base(3)));
}
// latitude and longitude of a cap centre for its place in the grid, by the
// polynomials 4.4.45 (arccos, error 7e-5) and 4.4.47 (arctan, error 1e-5) of
// Abramowitz and Stegun: the walk's margin of 3e-4 rad covers both errors
__device__ __forceinline__ float grid_lat(float y)
{
    const float a = fminf(1.0f, fabsf(y));
    const float t = 1.0f - a;
    const float p = fmaf(a, fmaf(a, fmaf(a, -0.0187293f, 0.0742610f), -0.2121144f), 1.5707288f);
    const float c = t > 0.0f ? t * rsqrtf(t) * p : 0.0f;  // arccos(a)
    return copysignf(0.5f * IDX_PI - c, y);
}
__device__ __forceinline__ float grid_lon(float x, float z)
{
    const float ax = fabsf(x), az = fabsf(z);
    const float hi = fmaxf(ax, az);
    const float r = hi > 0.0f ? __fdividef(fminf(ax, az), hi) : 0.0f;
    const float r2 = r * r;
    float t = fmaf(r2, fmaf(r2, fmaf(r2, fmaf(r2, 0.0208351f, -0.0851330f), 0.1801410f), -0.3302995f), 0.9998660f) * r;
    t = ax > az ? 0.5f * IDX_PI - t : t;
    t = z < 0.0f ? IDX_PI - t : t;
    return copysignf(t, x);
}

struct WalkShared {
    // range i: (its first candidate, first entry, entries before it wraps,
    // entry of candidate k past the wrap less k); ranges past the last: ~0
    uint4 rng[WALK_RANGES + 1];
    uint32_t total;  // candidates
    int groups;      // ranges, in groups of 32
};

// The tile's ranges, by one warp (all lanes).  g: its geometry (half-angle,
// latitude, longitude of the axis, h; h < 0: no valid pixel); ay: the axis'
// y = sin(latitude).  Fast trigonometry (errors of 1e-6) under the margins.
__device__ __forceinline__ void walk_ranges(const WalkIndex& wi, int T, const float4& g, float ay, WalkShared& ws)
{
    const unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const bool none = !(g.w >= 0.0f);
    uint32_t n = (uint32_t)T;
    float gam = 0.0f;
    int r0 = 0, before = 0, R = 0;
    if (!wi.direct) {
        // lanes 0 .. 3: their level's reach and rows
        const unsigned bits = lane < GRID_LEVELS ? wi.hdr[GRID_H_MAX + lane] : (lane == 31 ? wi.hdr[GRID_H_N] : 0u);
        n = min(__shfl_sync(FULL, bits, 31), (uint32_t)T);
        const int nlat = grid_nlat_of(lane);
        int nr = 0;
        if (lane < GRID_LEVELS && bits && !none) {
            // rho <= sin(rho) (1 + sin^2(rho) 0.19) up to 30 degrees
            const float sr = fminf(0.5f, __uint_as_float(bits));
            const float rho = sr * fmaf(sr * sr, 0.19f, 1.00001f);
            gam = g.w <= 1.0f ? g.x + rho + (wi.pstep ? 4.0f : 1.0f) * g.w + 3e-4f : 4.0f;
            r0 = gam < IDX_PI ? grid_row(g.y - gam, nlat) : 0;
            nr = (gam < IDX_PI ? grid_row(g.y + gam, nlat) : nlat - 1) - r0 + 1;
        }
        int incl = nr;
#pragma unroll
        for (int o = 1; o < GRID_LEVELS; o <<= 1) {
            const int y = __shfl_up_sync(FULL, incl, o);
            if (lane >= o) incl += y;
        }
        before = incl - nr;
        R = __shfl_sync(FULL, incl, GRID_LEVELS - 1) + 1;  // and the list
    }
    if (none || wi.direct || R > WALK_RANGES) {
        ws.rng[lane] = make_uint4(lane > 0 ? 0xffffffffu : 0u, 0u, n, 0u);
        if (lane == 0) ws.rng[32] = make_uint4(0xffffffffu, 0u, 0u, 0u);
        if (lane == 0) {
            ws.total = none ? 0u : n;
            ws.groups = 1;
        }
        return;
    }
    const int p1 = __shfl_sync(FULL, before, 1), p2 = __shfl_sync(FULL, before, 2), p3 = __shfl_sync(FULL, before, 3);
    const float clat = sqrtf(fmaxf(0.0f, fmaf(-ay, ay, 1.0f)));
    uint32_t carry = 0;
#pragma unroll 1
    for (int b = 0; b < WALK_RANGES; b += 32) {
        const int i = b + lane;
        const int l = (i >= p1) + (i >= p2) + (i >= p3);
        const float gl = __shfl_sync(FULL, gam, l);
        const int row = __shfl_sync(FULL, r0, l) + i - __shfl_sync(FULL, before, l);
        uint32_t a0 = 0, len0 = 0, a1 = 0, len1 = 0;
        if (i < R - 1) {
            const int nlat = grid_nlat_of(l);
            const int ncol = grid_ncol(nlat, row);
            const uint32_t* st = wi.start + grid_base_of(l) + row * (2 * nlat + 1);
            int c0 = 0, c1 = ncol - 1;
            if (fabsf(g.y) + gl < 0.5f * IDX_PI - 0.1f) {
                // the cap's longitude half-width over this row: at the
                // latitude of its widest point (sin = sin(lat) / cos(gamma)),
                // or the row's nearest edge
                const float cell = __fdividef(IDX_PI, (float)nlat), lo = fmaf((float)row, cell, -0.5f * IDX_PI);
                const float wide = grid_lat(__fdividef(ay, __cosf(gl)));
                const float phi = fminf(lo + cell, fmaxf(lo, wide));
                const float sg = __sinf(0.5f * gl), sd = __sinf(0.5f * (phi - g.y));
                const float q = __fdividef(sg * sg - sd * sd, __cosf(phi) * clat);  // sin^2 of half of it
                // the sines' errors (4e-7) and the filed latitudes' (7e-5) over cos(phi) clat >= 0.01
                const float sq = fminf(1.0f, fmaxf(0.0f, fmaf(4e-4f, sg, q)));
                // arcsin by the arccos polynomial (error 7e-5)
                const float dl = 2.0f * grid_lat(sq * rsqrtf(fmaxf(sq, 1e-30f))) + 5e-4f;
                const float k = (float)ncol * (0.5f / IDX_PI);
                const int f0 = (int)floorf((g.z - dl + IDX_PI) * k), f1 = (int)floorf((g.z + dl + IDX_PI) * k);
                if (f1 - f0 + 1 < ncol) {
                    c0 = f0 < 0 ? f0 + ncol : f0;
                    c1 = f1 >= ncol ? f1 - ncol : f1;
                }
            }
            c0 = min(max(c0, 0), ncol - 1);
            c1 = min(max(c1, 0), ncol - 1);
            // one range, or two where the window wraps across longitude +-pi
            const bool wraps = c0 > c1;
            const uint32_t e0 = min(st[wraps ? ncol : c1 + 1], n);
            a0 = min(st[c0], n);
            len0 = e0 > a0 ? e0 - a0 : 0u;
            if (wraps) {
                a1 = min(st[0], n);
                const uint32_t e1 = min(st[c1 + 1], n);
                len1 = e1 > a1 ? e1 - a1 : 0u;
            }
        } else if (i == R - 1) {
            a0 = min(wi.start[GRID_LIST], n);
            const uint32_t e0 = min(wi.start[GRID_LIST + 1], n);
            len0 = e0 > a0 ? e0 - a0 : 0u;
        }
        uint32_t incl = len0 + len1;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(FULL, incl, o);
            if (lane >= o) incl += y;
        }
        const uint32_t first = carry + incl - (len0 + len1);
        ws.rng[i] = i < R ? make_uint4(first, a0, len0, a1 - len0) : make_uint4(0xffffffffu, 0u, 0u, 0u);
        carry += __shfl_sync(FULL, incl, 31);
        if (b + 32 >= R) {
            if (lane == 0) {
                ws.rng[b + 32] = make_uint4(0xffffffffu, 0u, 0u, 0u);
                ws.total = carry;
                ws.groups = b / 32 + 1;
            }
            break;
        }
    }
}

// The walk as one thread sees it, after the barrier that follows walk_ranges.
struct Walk {
    float ax, ay, az, ca, sa, h;  // the tile's cone and widest ramp
    float2 ramp;                  // pixel step: pstep_ramp(h)
    uint32_t ex0;                 // first candidate of range `lane`

    __device__ __forceinline__ void init(const WalkIndex& wi, const Cone& c, const WalkShared& ws)
    {
        const int lane = threadIdx.x & 31;
        ax = c.c0.x;
        ay = c.c0.y;
        az = c.c0.z;
        ca = c.c0.w;
        sa = c.c1.x;
        h = c.c1.y;
        ramp = wi.pstep ? pstep_ramp(h) : make_float2(1.0f, 0.0f);
        ex0 = ws.rng[lane].x;
    }

    // A candidate as read: its cap (centre, cos and sin of its radius) and triangle.
    struct Cand {
        float4 q;
        float sr;
        uint32_t t;
        bool ok;
    };

    // candidate idx < total (one per thread, consecutive within a warp;
    // `in`: whether this thread's exists -- all lanes call)
    __device__ __forceinline__ Cand read(const WalkIndex& wi, const float4* rec, int T,
                                         const WalkShared& ws, uint32_t idx, bool in) const
    {
        Cand c{make_float4(0.0f, 0.0f, 0.0f, 0.0f), 0.0f, 0u, in};
        if (wi.direct) {
            c.t = idx;
            if (in) {
                const F8 cap = ld_f8(rec + rec_at((size_t)T, idx, RF_CAP));
                c.q = cap.a;
                c.sr = cap.b.x;
                c.ok = cap.b.w != 0.0f;
            }
        } else {
            // the range of the warp's first candidate by a vote per group of
            // ranges (one, but for wide tiles), then each lane moves on to its own
            const unsigned FULL = 0xffffffffu;
            const uint32_t lane = threadIdx.x & 31, first = idx - lane;
            int o = __popc(__ballot_sync(FULL, ex0 <= first)) - 1;
            for (int g = 1; g < ws.groups; ++g) o += __popc(__ballot_sync(FULL, ws.rng[32 * g + lane].x <= first));
            if (in) {
                while (ws.rng[o + 1].x <= idx) ++o;
                const uint4 r = ws.rng[o];
                const uint32_t k = idx - r.x;
                const uint32_t e = k < r.z ? r.y + k : r.w + k;
                const F8 ent = ld_f8(wi.ent + 2 * (size_t)e);
                c.q = ent.a;
                c.sr = ent.b.x;
                c.t = __float_as_uint(ent.b.y);
            }
        }
        return c;
    }

    // whether the cap may reach the tile's cone
    __device__ __forceinline__ bool reaches(const WalkIndex& wi, const Cand& c) const
    {
        const float4& q = c.q;
        const float sr = c.sr;
        float cb, sb;
        if (wi.pstep) {
            const float2 c4 = pstep_cap(q.w, sr, ramp);
            cb = c4.x;
            sb = c4.y;
        } else {
            cb = fmaf(-h, sr, q.w);
            const float s2 = fmaxf(fmaf(-cb, cb, 1.0f), 1e-30f);
            sb = s2 * rsqrtf(s2);
        }
        // angle(S, axis) <= alpha + beta (always when alpha + beta >= pi); the
        // margin covers the FP32 rounding of the products
        const float cg = fmaf(q.x, ax, fmaf(q.y, ay, q.z * az));
        return c.ok && (cb + ca <= 2e-6f || cg >= fmaf(ca, cb, -sa * sb) - 2e-6f);
    }
};

// The hits of candidates [i0, i1), at most WALK_BLOCK, appended to ids (*n of
// them so far, both in shared memory).  Called by every thread of the CTA; the
// caller synchronizes on both sides.  A thread reads two candidates before it
// tests either (1M triangles from inside: 427.5 -> 421.5 us a frame; the pixel
// step at 1280 x 720: 119.5 -> 115.9 us).  Prefetching the hits' records as
// they are found changed nothing (421.3, 116.4 us).
__device__ __forceinline__ void walk_hits(const Walk& w, const WalkIndex& wi, const float4* rec, int T,
                                          const WalkShared& ws, uint32_t i0, uint32_t i1, uint32_t* ids, uint32_t* n)
{
    const unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const uint32_t lt = (1u << lane) - 1u;
    for (uint32_t i = i0; i < i1; i += 2 * WALK_THREADS) {
        const uint32_t ia = i + threadIdx.x, ib = ia + WALK_THREADS;
        const bool two = i + WALK_THREADS < i1;
        const Walk::Cand a = w.read(wi, rec, T, ws, ia, ia < i1);
        Walk::Cand b{};
        if (two) b = w.read(wi, rec, T, ws, ib, ib < i1);
        const bool ha = w.reaches(wi, a), hb = two && w.reaches(wi, b);
        const unsigned ma = __ballot_sync(FULL, ha), mb = __ballot_sync(FULL, hb);
        if (!(ma | mb)) continue;
        uint32_t at = 0;
        if (lane == 0) at = atomicAdd(n, (uint32_t)(__popc(ma) + __popc(mb)));
        at = __shfl_sync(FULL, at, 0);
        if (ha) ids[at + (uint32_t)__popc(ma & lt)] = a.t;
        if (hb) ids[at + (uint32_t)(__popc(ma) + __popc(mb & lt))] = b.t;
    }
}
