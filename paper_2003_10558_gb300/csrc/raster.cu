// raster.cu -- per-tile coverage / depth / visibility kernel.
//
// One CTA of 128 threads per 16x16 tile; warp w covers the 8x8 pixel block
// (w & 1, w >> 1) of the tile and each lane two pixels of it, (x, y) and
// (x, y + 4), so every shared-memory load, vote and branch per triangle
// serves two pixels.  For every pixel G (unit direction, global delta) and
// every triangle t of the tile's bin the kernel evaluates the four plane
// distances of the rasterization equation (Sec. 1.1.2):
//   g_1..3 = G.n_i                   edge planes through the eye (Sec. 1.1)
//   g_4    = (G.S-hat - cos rho)/sin rho   miter cap, in the same angular
//            units as the edge distances, computed in the chord form
//            (4 sin^2(rho/2) - |G - S-hat|^2 + |G|^2 - 1) / (2 sin rho),
//            which keeps its accuracy for caps far below a pixel
// then   fragment   iff min g_i > -1/(2 delta) and r > 0   (gbpxstep)
//        m^f        = clamp(delta min g_i + 1/2, 0, 1)       (gpstep)
//        r          = (A'.N-hat)/(G.N-hat)                    (Sec. 1.1.4)
//        centre-inside iff g_1..3 >= 0 (tie rule via the normal's sign)
// and merges front to back (Sec. 1.4).  The merge
//   m^fc = min(m^f, 1 - m^b),  m^b = m^b + m^fc
// equals m^b = min(1, sum m^f) by induction, independent of the order, so
// each pixel keeps a saturating 2^-22 fixed-point sum and the 64-bit key
// (bits(r) << 32 | t) of its nearest centre-inside triangle.
//
// Accuracy in FP32: every distance is re-centred on the tile's cone axis a,
//   G.n = a.n + (G - a).n,
// with a.n formed once per (tile, triangle) from the FP32-pair normals in a
// compensated dot product.  The per-pixel part is a plain 3-term FMA chain
// on |G - a| <= the tile's angular radius, so its rounding error in units of
// the ramp is ~(tile size in pixels) x 2^-23, a few 1e-6 of coverage.
//
// Work culling (the paper's low-resolution region mask, Sec. 1.1.3, at the
// granularity of a warp's 8x8 pixels): the triangles of a staged chunk are
// first tested lane-parallel (lane j <-> triangle j) against each warp's
// view cone, cap and edge planes alike; the survivors are then evaluated for
// all 64 pixels, one triangle per step for the whole warp.  A culled pair is
// never a fragment, and both the coverage sum and the visibility key are
// order-free, so the result does not depend on the cull.
#include <type_traits>

#include "raster_walk.cuh"

namespace {

// One lane's two pixels as the evaluation sees them.
struct PixPair {
    float2 dgx, dgy, dgz;  // G - a (tile axis) of both pixels; 0 at an invalid pixel
    float2 eg;             // |G|^2 - 1
    float delta[PPT];      // global delta (0: invalid pixel)
    float lim[PPT];        // fragment iff min distance > lim (-1/(2 delta); +inf if invalid)
    uint32_t acc[PPT];     // coverage, 2^-22 fixed point (not meaningful at an invalid pixel)
    unsigned long long key[PPT];  // ((bits(r) - 1) << 32) | t of the nearest centre-inside fragment, or KEY_NONE
    int32_t cnt_in[PPT];   // centre-inside fragments (statistics)
};
// Evaluate staged slot j at the lane's two pixels and merge the fragments into the pixels' coverage and keys.
// Called by all 32 lanes of a warp together (warp votes).
//
// Issue-bound, the compares and selects (ALU pipe, half rate) above all.  So:
// the coverage of a lane without a fragment is added too (its ramp value
// rounds to 0 in the 2^-22 fixed point: gm <= -1/(2 delta) rounded leaves at
// most 2^-25 after the 1/2); the depth test is folded into the key, whose
// high word is bits(r) - 1; and everything rare -- a distance exactly on an
// edge plane (tie rule), a plane distance too small for the plain reciprocal
// -- is one warp-uniform decision to run the general copy.
template <bool STATS>
__device__ __forceinline__ void eval_slot(const Stage& st, int j, PixPair& q, uint32_t& cnt_alg)
{
    // the four distances of both pixels in packed FP32x2 arithmetic; the miter
    // in chord form, G - S-hat = (G - a) - (S-hat - a): both differences are at
    // most the tile radius, so their rounding costs ~1e-9 rad where it matters
    const float4 b = st.s1[j];
    const float4 e = st.s6[j];
    const float2 g4p = miter_distance2(q.dgx, q.dgy, q.dgz, e, b, q.eg);
    const float2 g1p = plane_distance2(q.dgx, q.dgy, q.dgz, st.s2[j]);
    const float2 g2p = plane_distance2(q.dgx, q.dgy, q.dgz, st.s3[j]);
    const float2 g3p = plane_distance2(q.dgx, q.dgy, q.dgz, st.s4[j]);
    const float g4[PPT] = {g4p.x, g4p.y};
    const float g3m[PPT] = {fminf(fminf(g1p.x, g2p.x), g3p.x), fminf(fminf(g1p.y, g2p.y), g3p.y)};
    float gm[PPT];
    bool frag[PPT], anyf = false;
#pragma unroll
    for (int p = 0; p < PPT; ++p) {
        if (STATS) cnt_alg += g4[p] > q.lim[p];
        gm[p] = fminf(g3m[p], g4[p]);
        frag[p] = gm[p] > q.lim[p];  // gbpxstep on all four distances; never on invalid pixels
        anyf |= frag[p];
    }
    if (!__any_sync(0xffffffffu, anyf)) return;
    const float2 Dp = plane_distance2(q.dgx, q.dgy, q.dgz, st.s5[j]);
    const float D[PPT] = {Dp.x, Dp.y};
    auto post = [&](auto rare_t) {
        constexpr bool RARE = decltype(rare_t)::value;
        uint32_t rq[PPT];
        bool inn[PPT];
#pragma unroll
        for (int p = 0; p < PPT; ++p) {
            const float r = RARE ? __fdividef(b.w, D[p]) : __fmul_rn(b.w, rcp_fast(D[p]));
            rq[p] = __float_as_uint(r) - 1u;
            const float m = __saturatef(fmaf(gm[p], q.delta[p], 0.5f));
            if (rq[p] < DEPTH_LIM) q.acc[p] += cov_fixed(m);
            // centre-inside: all three edge distances >= 0; an exact zero
            // takes the tie rule on the three distances, recomputed from
            // the staged planes (the scalar form gives the packed values
            // bit for bit), so they need not stay live in registers here
            inn[p] = frag[p] && g3m[p] > 0.0f;
            if (RARE && frag[p] && g3m[p] == 0.0f) {
                const float dx = p ? q.dgx.y : q.dgx.x, dy = p ? q.dgy.y : q.dgy.x, dz = p ? q.dgz.y : q.dgz.x;
                inn[p] = centre_inside(plane_distance(dx, dy, dz, st.s2[j]), plane_distance(dx, dy, dz, st.s3[j]),
                                       plane_distance(dx, dy, dz, st.s4[j]), g3m[p], __float_as_uint(st.s0[j].w));
            }
            if (STATS) q.cnt_in[p] += inn[p] && rq[p] < DEPTH_LIM;
        }
        // the visibility keys only where some lane of the warp has a
        // centre-inside fragment
        if (__any_sync(0xffffffffu, inn[0] || inn[1])) {
#pragma unroll
            for (int p = 0; p < PPT; ++p) {
                const unsigned long long k = ((unsigned long long)rq[p] << 32) | __float_as_uint(e.w);
                q.key[p] = inn[p] && k < q.key[p] ? k : q.key[p];
            }
        }
    };
    const float tiny = fminf(fminf(fabsf(g3m[0]), fabsf(g3m[1])), fminf(fabsf(D[0]), fabsf(D[1])));
    if (__any_sync(0xffffffffu, tiny < 1.17549435e-38f))
        post(std::true_type{});
    else
        post(std::false_type{});
}

// The pixel pair's loop state from its directions (xyz, delta) and the tile
// axis; invalid pixels (delta 0) evaluate at the axis and never pass.
__device__ __forceinline__ void pix_pair(PixPair& q, const float4& g0, const float4& g1, float ax, float ay, float az)
{
    const bool v0 = g0.w > 0.0f, v1 = g1.w > 0.0f;
    q.dgx = make_float2(v0 ? g0.x - ax : 0.0f, v1 ? g1.x - ax : 0.0f);
    q.dgy = make_float2(v0 ? g0.y - ay : 0.0f, v1 ? g1.y - ay : 0.0f);
    q.dgz = make_float2(v0 ? g0.z - az : 0.0f, v1 ? g1.z - az : 0.0f);
    const float2 eg = norm2_minus_one2(make_float2(g0.x, g1.x), make_float2(g0.y, g1.y), make_float2(g0.z, g1.z));
    q.eg = make_float2(v0 ? eg.x : 0.0f, v1 ? eg.y : 0.0f);
    q.delta[0] = g0.w;
    q.delta[1] = g1.w;
    q.lim[0] = v0 ? -(0.5f / g0.w) : INFINITY;
    q.lim[1] = v1 ? -(0.5f / g1.w) : INFINITY;
#pragma unroll
    for (int p = 0; p < PPT; ++p) {
        q.acc[p] = 0u;
        q.key[p] = KEY_NONE;
        q.cnt_in[p] = 0;
    }
}

// Coverage of a finished pixel: saturated, 0 at an invalid pixel.
__device__ __forceinline__ uint32_t final_acc(const PixPair& q, int p)
{
    return q.lim[p] < INFINITY ? min(q.acc[p], COV_ONE) : 0u;
}

// The pixels' loop state, and the warp's own view cone; returns whether the
// warp has a valid pixel.
__device__ __forceinline__ bool start_pixels(const float4 (&g)[PPT], const float4& axis, PixPair& q, WarpCones& wc)
{
    pix_pair(q, g[0], g[1], axis.x, axis.y, axis.z);
    const float gx[PPT] = {g[0].x, g[1].x}, gy[PPT] = {g[0].y, g[1].y}, gz[PPT] = {g[0].z, g[1].z};
    const bool pv[PPT] = {g[0].w > 0.0f, g[1].w > 0.0f};
    const float h[PPT] = {pv[0] ? -q.lim[0] : 0.0f, pv[1] ? -q.lim[1] : 0.0f};
    float4 c0, c1;
    block_cone(gx, gy, gz, h, pv, c0, c1);
    if ((threadIdx.x & 31) == 0) {
        wc.c[threadIdx.x >> 5][0] = c0;
        wc.c[threadIdx.x >> 5][1] = c1;
    }
    __syncwarp();
    return c1.z > 0.0f;
}

// The n staged triangles of a chunk at the warp's pixels: a lane-parallel cull
// of 32 triangles at a time against the warp's cone, then the survivors one by
// one.
template <bool STATS>
__device__ __forceinline__ void eval_chunk(const Stage& st, int n, const WarpCones& wc, bool count_alg, PixPair& q,
                                           uint32_t& cnt_alg, uint32_t& cnt_exec)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int gbase = 0; gbase < n; gbase += 32) {
        const float4 wc0 = wc.c[warp][0], wc1 = wc.c[warp][1];
        bool keep = false;
        const int jj = gbase + lane;
        if (jj < n && __float_as_uint(st.s6[jj].w) != STAGE_EMPTY)
            keep = cone_may_hit(st.s0[jj], st.s1[jj], st.s2[jj], st.s3[jj], st.s4[jj], wc0, wc1, count_alg);
        unsigned mask = __ballot_sync(0xffffffffu, keep);
        while (mask) {
            const int k = 31 - __clz(mask);  // any order: from the top, one instruction less than from the bottom
            mask ^= 1u << k;
            if (STATS) ++cnt_exec;
            eval_slot<STATS>(st, gbase + k, q, cnt_alg);
        }
    }
}

// The global step for the walking raster.
struct GlobalStep {
    static constexpr int CTAS = VSR_RASTER_CTAS_PER_SM, FEW_BLOCK = WALK_BLOCK / 4;
    static constexpr bool SATURATES = true, HOST_OUT = true, SKIPS = false;
    static constexpr int FEW_FROM = 2, SHARE_FROM = 1;
    using Pix = PixPair;
    using Cones = WarpCones;
    struct In {};
    struct Raw {
        float4 g[PPT];
    };
    __device__ __forceinline__ static void load(const RasterView& view, const In&, const TilePos& tp, Raw& r)
    {
        load_pixels(view, tp, r.g);
    }
    __device__ __forceinline__ static bool start(const Raw& r, const float4& axis, Pix& q, Cones& wc)
    {
        return start_pixels(r.g, axis, q, wc);
    }
    __device__ __forceinline__ static bool cull(const Stage& st, int j, const Cones& wc, int warp)
    {
        return cone_may_hit(st.s0[j], st.s1[j], st.s2[j], st.s3[j], st.s4[j], wc.c[warp][0], wc.c[warp][1], false);
    }
    __device__ __forceinline__ static void eval(const WalkCtx<In>&, const Stage& st, int j, Pix& q)
    {
        uint32_t unused = 0;
        eval_slot<false>(st, j, q, unused);
    }
    __device__ __forceinline__ static uint32_t final_acc(const Pix& q, int p) { return ::final_acc(q, p); }
    __device__ __forceinline__ static void group(const WalkCtx<In>&, int, Pix&) {}
    __device__ __forceinline__ static bool skip(const In&, int) { return false; }
    __device__ __forceinline__ static void clamp(Pix& q)
    {
#pragma unroll
        for (int p = 0; p < PPT; ++p) q.acc[p] = min(q.acc[p], COV_ONE);
    }
    template <bool ROWS>
    __device__ __forceinline__ static void finish(const WalkCtx<In>& cx, const TilePos& tp, const Pix& q, int*)
    {
        write_tile<ROWS>(cx.view, tp, q);
    }
};

// One 16x16 tile of one view over its stored bin.  Called by every thread of a
// CTA of RT threads; `st` is the CTA's staging area (reusable across calls:
// every use is fenced by the barriers of the chunk loop).
template <bool STATS, bool ROWS = false>
__device__ __forceinline__ void raster_tile(const RasterView& view, int tile, Stage& st, bool count_alg,
                                            uint32_t& cnt_alg, uint32_t& cnt_exec, int32_t* __restrict__ n_inside,
                                            int* __restrict__ status, int range_lo = 0, int range_hi = -1,
                                            int split_slot = -1, int nsplit = 1, SplitAcc split = SplitAcc{})
{
    const uint32_t* ids = view.ids;
    const uint32_t cap = view.cap;
    const TilePos tp(tile, view.tiles_x);
    const Cone tc = view.tiles[tile];
    PixPair q;
    __shared__ WarpCones wc;
    float4 g[PPT];
    load_pixels(view, tp, g);
    const bool warp_active = start_pixels(g, tc.c0, q, wc);

    uint32_t b0 = 0, b1 = 0;
    if (tc.c1.z > 0.0f) {
        b0 = view.offsets[tile];
        b1 = view.ends ? view.ends[tile] : view.offsets[tile + 1];
        if (b1 > cap) {
            if (threadIdx.x == 0 && b0 <= cap) raise_status(status, VSR_ERR_BIN_OVERFLOW);  // (as the binning, once)
            b1 = cap;
            b0 = min(b0, cap);
        }
        if (range_hi >= 0) {  // one item of a split tile
            const uint32_t lo = b0 + (uint32_t)range_lo, hi = b0 + (uint32_t)range_hi;
            b0 = min(lo, b1);
            b1 = min(hi, b1);
        }
    }
    static_assert(PPT == 2, "packed pairs hold the thread's two pixels");

    for (uint32_t base = b0; base < b1; base += CHUNK) {
        const int n = (int)min((uint32_t)CHUNK, b1 - base);
        // saturate once per chunk: at most CHUNK terms of <= COV_ONE each were added since
#pragma unroll
        for (int p = 0; p < PPT; ++p) q.acc[p] = min(q.acc[p], COV_ONE);
        __syncthreads();
        if ((int)threadIdx.x < n) stage_checked(view.rec, view.T, ids[base + threadIdx.x], tc.c0, st, threadIdx.x, status);
        __syncthreads();
        if (warp_active) eval_chunk<STATS>(st, n, wc, count_alg, q, cnt_alg, cnt_exec);
    }

#pragma unroll
    for (int p = 0; p < PPT; ++p) q.acc[p] = final_acc(q, p);
    if (split_slot >= 0 && !merge_slot(split, split_slot, tp, q, 1u, (uint32_t)nsplit)) return;
    write_tile<ROWS>(view, tp, q);
    if (STATS && n_inside) {
#pragma unroll
        for (int p = 0; p < PPT; ++p)
            if (tp.px < view.W && tp.py + 4 * p < view.H)
                n_inside[(size_t)(tp.py + 4 * p) * view.W + tp.px] = q.cnt_in[p];
    }
}

template <bool STATS>
__global__ void __launch_bounds__(RT, 7) raster_kernel(RasterView view, unsigned long long* __restrict__ n_alg,
                                                        unsigned long long* __restrict__ n_exec,
                                                        int32_t* __restrict__ n_inside, int* __restrict__ status)
{
    __shared__ Stage st;
    __shared__ unsigned long long red[2][RT / 32];
    uint32_t cnt_alg = 0, cnt_exec = 0;
    raster_tile<STATS>(view, blockIdx.x, st, n_alg != nullptr, cnt_alg, cnt_exec, n_inside, status);
    if (STATS && (n_alg || n_exec)) {
        const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
        // cnt_exec counts warp-level evaluations: one per (warp, triangle) for 64 pixels
        unsigned long long va = cnt_alg, ve = lane == 0 ? (unsigned long long)cnt_exec * (32ull * PPT) : 0ull;
        for (int o = 16; o; o >>= 1) {
            va += __shfl_xor_sync(0xffffffffu, va, o);
            ve += __shfl_xor_sync(0xffffffffu, ve, o);
        }
        if (lane == 0) {
            red[0][warp] = va;
            red[1][warp] = ve;
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            unsigned long long sa = 0, se = 0;
            for (int w = 0; w < RT / 32; ++w) {
                sa += red[0][w];
                se += red[1][w];
            }
            if (n_alg) atomicAdd(n_alg, sa);
            if (n_exec) atomicAdd(n_exec, se);
        }
    }
}

// Raster over work items, one CTA each.  Items 0 .. n_tiles-1 are the tiles
// themselves (the first item of a split tile); the further items of split
// tiles are listed in `extra` as (tile, k).  CTAs past the end of the list
// return at once.
template <bool ROWS>
__global__ void __launch_bounds__(RT, VSR_RASTER_CTAS_PER_SM) raster_items_kernel(RasterView view, uint32_t n_tiles,
                                                              const uint32_t* nsplit_of,
                                                              const int32_t* split_slot,
                                                              const uint2* extra,
                                                              const uint32_t* n_extra, int split_max,
                                                              SplitAcc split, int* __restrict__ status)
{
    grid_wait();
    grid_go();
    __shared__ Stage st;
    uint32_t u, k = 0;
    if (blockIdx.x < n_tiles) {
        u = blockIdx.x;
    } else {
        const uint32_t e = blockIdx.x - n_tiles;
        if (e >= *n_extra) return;
        const uint2 uk = extra[e];
        if (uk.x == 0xffffffffu) return;
        u = uk.x;
        k = uk.y;
    }
    const int nsplit = (int)nsplit_of[u];
    uint32_t ca = 0, ce = 0;
    if (nsplit == 1)
        raster_tile<false, ROWS>(view, (int)u, st, false, ca, ce, nullptr, status);
    else
        raster_tile<false, ROWS>(view, (int)u, st, false, ca, ce, nullptr, status, (int)k * split_max,
                           (int)(k + 1) * split_max, split_slot[u], nsplit, split);
}

// The work items of several views in one persistent launch: each CTA takes
// the next item of a shared queue (an atomic counter over the views' item
// ranges, item_start[v] .. item_start[v + 1]: the view's tiles, then room
// for its extra items) until none is left, and rasterizes it exactly as
// raster_items_kernel does.  The views' items must have been assigned
// (items_kernel) on the launching stream before.
__global__ void __launch_bounds__(RT, VSR_RASTER_CTAS_PER_SM) raster_pool_kernel(const PoolView* __restrict__ views,
                                                                                 const uint32_t* __restrict__ item_start,
                                                                                 int nviews, uint32_t* __restrict__ queue,
                                                                                 int split_max, int* __restrict__ status)
{
    __shared__ Stage st;
    __shared__ uint32_t s_item;
    const uint32_t total = item_start[nviews];
    for (;;) {
        __syncthreads();  // the previous item is done with the shared memory
        if (threadIdx.x == 0) s_item = atomicAdd(queue, 1u);
        __syncthreads();
        const uint32_t it = s_item;
        if (it >= total) return;
        int v = 0;  // the last view whose items start at or before `it`
        for (int hi = nviews - 1; v < hi;) {
            const int mid = (v + hi + 1) >> 1;
            if (item_start[mid] <= it)
                v = mid;
            else
                hi = mid - 1;
        }
        const PoolView& pv = views[v];
        const uint32_t e = it - item_start[v];
        uint32_t u, k = 0;
        if (e < pv.n_tiles) {
            u = e;
        } else {
            const uint32_t x = e - pv.n_tiles;
            if (x >= *pv.n_extra) continue;
            const uint2 uk = pv.extra[x];
            if (uk.x == 0xffffffffu) continue;
            u = uk.x;
            k = uk.y;
        }
        const int nsplit = (int)pv.nsplit_of[u];
        uint32_t ca = 0, ce = 0;
        if (nsplit == 1)
            raster_tile<false>(pv.view, (int)u, st, false, ca, ce, nullptr, status);
        else
            raster_tile<false>(pv.view, (int)u, st, false, ca, ce, nullptr, status, (int)k * split_max,
                               (int)(k + 1) * split_max, pv.split_slot[u], nsplit,
                               SplitAcc{pv.acc, pv.key, pv.done});
    }
}

// Dense reference of the same rasterization: every pixel of a tile against
// every triangle of the scene, with no binning and no cull.  As in the
// oracle, the miter distance is evaluated first: a triangle whose enlarged
// cap holds none of the warp's 64 pixels is skipped after it (a warp vote),
// else the coverage kernel's own evaluation follows.  The outputs equal the
// binned path's bit for bit (the same arithmetic per pair, and the merge is
// order-free); its cost is that of W x H x T pair tests.
__global__ void __launch_bounds__(RT) raster_dense_kernel(RasterView view, int* __restrict__ status)
{
    __shared__ Stage st;
    const int T = view.T;
    const TilePos tp(blockIdx.x, view.tiles_x);
    const Cone tc = view.tiles[blockIdx.x];
    const float ax = tc.c0.x, ay = tc.c0.y, az = tc.c0.z;
    PixPair q;
    float4 g[PPT];
    load_pixels(view, tp, g);
    pix_pair(q, g[0], g[1], ax, ay, az);
    const bool active = tc.c1.z > 0.0f;
    const size_t TT = (size_t)T;
    uint32_t unused = 0;
    for (int base = 0; active && base < T; base += CHUNK) {
        const int n = min(CHUNK, T - base);
#pragma unroll
        for (int p = 0; p < PPT; ++p) q.acc[p] = min(q.acc[p], COV_ONE);
        __syncthreads();
        if ((int)threadIdx.x < n) {
            const uint32_t t = (uint32_t)(base + threadIdx.x);
            if (view.rec[rec_at(TT, t, RF_CAP2)].w == 0.0f)  // culled at set-up
                st.s6[threadIdx.x] = make_float4(0.0f, 0.0f, 0.0f, __uint_as_float(STAGE_EMPTY));
            else
                stage_triangle(view.rec, TT, t, ax, ay, az, st, threadIdx.x);
        }
        __syncthreads();
        for (int j = 0; j < n; ++j) {
            const float4 e = st.s6[j];
            if (__float_as_uint(e.w) == STAGE_EMPTY) continue;
            const float2 g4 = miter_distance2(q.dgx, q.dgy, q.dgz, e, st.s1[j], q.eg);
            if (!__any_sync(0xffffffffu, g4.x > q.lim[0] || g4.y > q.lim[1])) continue;
            eval_slot<false>(st, j, q, unused);
        }
    }
#pragma unroll
    for (int p = 0; p < PPT; ++p) q.acc[p] = final_acc(q, p);
    write_tile<false>(view, tp, q);
}

// Work items per tile: ceil(bin / split_max) when a split slot and room in
// the extra list are free, else 1 (the tile runs in one CTA).
__global__ void items_kernel(const uint32_t* offsets, const uint32_t* ends,
                             uint32_t n_tiles, int split_max, uint32_t* __restrict__ nsplit_of,
                             int32_t* __restrict__ split_slot, uint32_t* __restrict__ counters /* n_split, n_extra */,
                             uint32_t split_cap, uint2* __restrict__ extra, uint32_t extra_cap)
{
    grid_wait();
    grid_go();
    const uint32_t u = blockIdx.x * blockDim.x + threadIdx.x;
    if (u >= n_tiles) return;
    const uint32_t c = (ends ? ends[u] : offsets[u + 1]) - offsets[u];
    uint32_t n = 1;
    int32_t slot = -1;
    if (c > (uint32_t)split_max) {
        const uint32_t want = (c + split_max - 1) / split_max;
        const uint32_t sl = atomicAdd(&counters[0], 1u);
        const uint32_t pos = atomicAdd(&counters[1], want - 1);
        const bool ok = sl < split_cap && pos + (want - 1) <= extra_cap;
        for (uint32_t q = 1; q < want && pos + q - 1 < extra_cap; ++q)
            extra[pos + q - 1] = ok ? make_uint2(u, q) : make_uint2(0xffffffffu, 0u);
        if (ok) {
            n = want;
            slot = (int32_t)sl;
        }
    }
    nsplit_of[u] = n;
    split_slot[u] = slot;
}

}  // namespace

vsr_status launch_raster(const float4* map, int W, int H, const Cone* tiles, const float4* rec, int T,
                         const uint32_t* offsets, const uint32_t* ids, uint32_t cap, uint32_t* id, float* depth,
                         float* cov, unsigned long long* n_alg, unsigned long long* n_exec, int32_t* n_inside,
                         int* status, cudaStream_t st, const uint32_t* ends)
{
    const int tx = (W + TILE - 1) / TILE, ty = (H + TILE - 1) / TILE;
    const RasterView v{map, W, H, tiles, tx, rec, T, offsets, ids, cap, id, depth, cov, ends};
    if (n_alg || n_exec || n_inside)
        raster_kernel<true><<<tx * ty, RT, 0, st>>>(v, n_alg, n_exec, n_inside, status);
    else
        raster_kernel<false><<<tx * ty, RT, 0, st>>>(v, nullptr, nullptr, nullptr, status);
    VSR_CUDA_TRY(cudaGetLastError());
    return VSR_OK;
}

int raster_split_items(int split_max) { return split_max < CHUNK ? CHUNK : (split_max / CHUNK) * CHUNK; }

uint32_t raster_extra_cap(uint32_t cap, const RasterWork& w, int split_max)
{
    // enough extra items for every pair of the bins, bounded by the list
    const uint64_t bound = (uint64_t)cap / (uint64_t)raster_split_items(split_max) + 1;
    return bound < w.extra_cap ? (uint32_t)bound : w.extra_cap;
}

vsr_status launch_raster_assign(const uint32_t* offsets, uint32_t n_tiles, uint32_t cap, RasterWork w, int split_max,
                                cudaStream_t st, const uint32_t* ends)
{
    if (n_tiles == 0) return VSR_OK;
    VSR_CUDA_TRY(cudaMemsetAsync(w.counters, 0, 2 * sizeof(uint32_t), st));
    VSR_CUDA_TRY(launch_next(items_kernel, (n_tiles + 255) / 256, 256, st, offsets, ends, n_tiles,
                             raster_split_items(split_max), w.nsplit_of, w.split_slot, w.counters, w.split_cap, w.extra,
                             raster_extra_cap(cap, w, split_max)));
    return VSR_OK;
}

vsr_status launch_raster_pool(const PoolView* views_dev, const uint32_t* item_start_dev, int nviews,
                              uint32_t* queue, int split_max, int* status, cudaStream_t st)
{
    if (nviews == 0) return VSR_OK;
    const int sms = sm_count();
    if (sms < 0) return VSR_ERR_CUDA;
    VSR_CUDA_TRY(cudaMemsetAsync(queue, 0, sizeof(uint32_t), st));
    raster_pool_kernel<<<sms * VSR_RASTER_CTAS_PER_SM, RT, 0, st>>>(views_dev, item_start_dev, nviews, queue,
                                                                    raster_split_items(split_max), status);
    VSR_CUDA_TRY(cudaGetLastError());
    return VSR_OK;
}

vsr_status launch_raster_items(const RasterView& view, const uint32_t* offsets, uint32_t n_tiles, uint32_t cap,
                               RasterWork w, int split_max, int* status, cudaStream_t st, bool host_out)
{
    if (n_tiles == 0) return VSR_OK;
    vsr_status s = launch_raster_assign(offsets, n_tiles, cap, w, split_max, st, view.ends);
    if (s != VSR_OK) return s;
    const uint32_t extra_cap = raster_extra_cap(cap, w, split_max);
    split_max = raster_split_items(split_max);
    auto kern = host_out ? raster_items_kernel<true> : raster_items_kernel<false>;
    VSR_CUDA_TRY(launch_next(kern, n_tiles + extra_cap, RT, st, view, n_tiles, w.nsplit_of, w.split_slot, w.extra,
                             w.counters + 1, split_max, SplitAcc{w.acc, w.key, w.done}, status));
    return VSR_OK;
}

vsr_status walk_work_alloc(WalkWork* w, cudaStream_t st)
{
    if (w->mem) return VSR_OK;
    // accumulators | keys | claims | done | nblk | hits | hint, active, begun, ended
    const size_t pix = sizeof(unsigned long long) * TILE_PIX * (size_t)WALK_SLOTS;
    const size_t rest = sizeof(unsigned long long) * WALK_SLOTS + 3 * sizeof(uint32_t) * WALK_SLOTS + 4 * sizeof(uint32_t);
    char* m = nullptr;
    if (cudaMalloc((void**)&m, 2 * pix + rest) != cudaSuccess) {
        cudaGetLastError();
        return VSR_ERR_OOM;
    }
    if (clear_workspace({{m, 0, pix}, {m + pix, 0xff, pix}, {m + 2 * pix, 0, rest}}, st) != VSR_OK) {
        cudaFree(m);
        return VSR_ERR_CUDA;
    }
    w->mem = m;
    return VSR_OK;
}

void walk_work_free(WalkWork* w)
{
    cudaFree(w->mem);
    w->mem = nullptr;
}

vsr_status launch_raster_walk(const RasterView& view, const WalkIndex& wi, const float4* geom, const WalkWork& work,
                              uint32_t* tile_pairs, int* status, cudaStream_t st, bool host_out)
{
    return launch_walk<GlobalStep>(view, GlobalStep::In{}, wi, geom, work, tile_pairs, status, st, host_out);
}

vsr_status launch_raster_dense(const RasterView& view, int* status, cudaStream_t st)
{
    const int n_tiles = view.tiles_x * ((view.H + TILE - 1) / TILE);
    if (n_tiles == 0) return VSR_OK;
    raster_dense_kernel<<<n_tiles, RT, 0, st>>>(view, status);
    VSR_CUDA_TRY(cudaGetLastError());
    return VSR_OK;
}

int raster_threads_per_cta() { return RT; }

vsr_status raster_work_alloc(RasterWork* w, uint32_t n_tiles, cudaStream_t st)
{
    *w = RasterWork{};
    const size_t cap = n_tiles < SPLIT_SLOTS ? n_tiles : SPLIT_SLOTS;
    // one allocation: accumulators | keys | extra items | done | items and slots per tile | counters
    const size_t pix = sizeof(unsigned long long) * TILE_PIX * (cap + 1);
    const size_t extra = sizeof(uint2) * EXTRA_ITEMS, done = sizeof(uint32_t) * (cap + 1);
    const size_t tiles = sizeof(uint32_t) * ((size_t)n_tiles + 1);
    char* m = nullptr;
    if (cudaMalloc((void**)&m, 2 * pix + extra + done + 2 * tiles + 2 * sizeof(uint32_t)) != cudaSuccess) {
        cudaGetLastError();
        return VSR_ERR_OOM;
    }
    w->acc = (unsigned long long*)m;
    w->key = (unsigned long long*)(m + pix);
    w->extra = (uint2*)(m + 2 * pix);
    w->done = (uint32_t*)(m + 2 * pix + extra);
    w->nsplit_of = (uint32_t*)(m + 2 * pix + extra + done);
    w->split_slot = (int32_t*)(m + 2 * pix + extra + done + tiles);
    w->counters = (uint32_t*)(m + 2 * pix + extra + done + 2 * tiles);
    w->split_cap = (uint32_t)cap;
    w->extra_cap = EXTRA_ITEMS;
    if (clear_workspace({{w->acc, 0, pix}, {w->key, 0xff, pix}, {w->done, 0, done}}, st) != VSR_OK) {
        raster_work_free(w);
        return VSR_ERR_CUDA;
    }
    return VSR_OK;
}

void raster_work_free(RasterWork* w)
{
    cudaFree(w->acc);
    *w = RasterWork{};
}
