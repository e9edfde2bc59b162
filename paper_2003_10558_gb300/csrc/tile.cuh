// tile.cuh -- what the tile kernels share: a CTA of 128 threads per 16x16
// tile, two pixels per lane, the warps' view cones, staging, the merge of a
// tile's parts and its outputs (raster.cu, pstep.cu, raster_walk.cuh).
#pragma once

#include "stage.cuh"

constexpr int RT = 128;          // threads per CTA (one 16x16 tile)
constexpr int PPT = 2;           // pixels per thread: (x, y) and (x, y + 4) of the warp's 8x8 block
constexpr int CHUNK = RT;        // triangles staged per pass
static_assert(CHUNK == STAGE_CHUNK, "one staging slot per thread");
static_assert(RT * PPT == TILE_PIX, "one CTA covers one tile");
// resident CTAs per SM the timed kernel is compiled for (its register cap)
#ifndef VSR_RASTER_CTAS_PER_SM
#define VSR_RASTER_CTAS_PER_SM 8
#endif

// Split tiles: a tile whose bin is longer than split_max triangles (a
// multiple of CHUNK) is processed as several work items of at most
// split_max triangles each.  The
// items of one tile add their coverage (2^-22 fixed point) and take the
// minimum of their visibility keys in the tile's accumulator slot with
// atomics -- both are order-free, so the result is exactly that of one item
// -- and the item that arrives last (atomic counter, nothing waits) writes
// the outputs and clears the slot for the next frame.
struct SplitAcc {
    unsigned long long* acc;  // [slot][TILE_PIX], zero between frames (64 bits: many partials)
    unsigned long long* key;  // [slot][TILE_PIX], ~0 between frames
    uint32_t* done;           // [slot], zero between frames
};

// A cone (axis, cos, sin, widest ramp half-width) may hold a fragment of the
// staged triangle (cap a, b; edge normals n1..n3): the cap test, and unless
// counting algorithmic tests (defined by the cap alone) the edge planes.
// Every pixel G of the cone is within alpha of the axis c, so
// G.n <= c.n + sin(alpha) + (1 - cos(alpha)) for a unit normal n; a triangle
// with some edge plane below -h there has no fragment.
__device__ __forceinline__ bool cone_may_hit(const float4& a, const float4& b, const float4& n1, const float4& n2,
                                             const float4& n3, const float4& c0, const float4& c1, bool count_alg)
{
    bool keep = cap_hits_cone(make_float3(a.x, a.y, a.z), 1.0f - 0.5f * b.y, b.x, make_float3(c0.x, c0.y, c0.z),
                              c0.w, c1.x, c1.y);
    const float lim = -(c1.y + c1.x + (1.0f - c0.w) + 1e-6f);
    return keep && (count_alg || (fmaf(c0.x, n1.x, fmaf(c0.y, n1.y, c0.z * n1.z)) > lim &&
                                  fmaf(c0.x, n2.x, fmaf(c0.y, n2.y, c0.z * n2.z)) > lim &&
                                  fmaf(c0.x, n3.x, fmaf(c0.y, n3.y, c0.z * n3.z)) > lim));
}

// View cone of the warp's 8x8 block from its valid pixels: axis = normalised
// sum, cos alpha = min G.axis less a margin, h = the widest ramp half-width;
// a block without a valid pixel gets valid = 0, a degenerate sum the whole
// sphere.  The cone only culls, so the sums may be taken in any order: the
// axis by shuffles, the two extrema by the integer reductions of sm_80+
// (non-negative floats order as their bits; the minimum of G.axis <= 1 + a
// few ulp as the maximum of 2 - G.axis, whose rounding of 1.2e-7 the margin
// covers).
__device__ __forceinline__ void block_cone(const float* gx, const float* gy, const float* gz, const float* h,
                                           const bool* pv, float4& c0, float4& c1)
{
    const unsigned FULL = 0xffffffffu;
    const int cn = __popc(__ballot_sync(FULL, pv[0])) + __popc(__ballot_sync(FULL, pv[1]));
    float sx = 0.0f, sy = 0.0f, sz = 0.0f, hw = 0.0f;
#pragma unroll
    for (int p = 0; p < PPT; ++p)
        if (pv[p]) {
            sx += gx[p];
            sy += gy[p];
            sz += gz[p];
            hw = fmaxf(hw, h[p]);
        }
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        sx += __shfl_xor_sync(FULL, sx, o);
        sy += __shfl_xor_sync(FULL, sy, o);
        sz += __shfl_xor_sync(FULL, sz, o);
    }
    hw = __uint_as_float(__reduce_max_sync(FULL, __float_as_uint(hw)));
    const float len2 = fmaf(sx, sx, fmaf(sy, sy, sz * sz));
    const bool deg = !(len2 > 1e-12f * (float)(cn * cn));
    const float inv = rsqrtf(len2);
    const float ax = deg ? 0.0f : sx * inv, ay = deg ? 0.0f : sy * inv, az = deg ? 1.0f : sz * inv;
    float away = 0.0f;
#pragma unroll
    for (int p = 0; p < PPT; ++p)
        if (pv[p]) away = fmaxf(away, 2.0f - fmaf(gx[p], ax, fmaf(gy[p], ay, gz[p] * az)));
    const float cm = 2.0f - __uint_as_float(__reduce_max_sync(FULL, __float_as_uint(away)));
    float cs = fmaxf(-1.0f, fminf(1.0f, cm - 2e-6f));
    if (deg) cs = -1.0f;
    c0 = make_float4(ax, ay, az, cs);
    c1 = make_float4(sqrtf(fmaxf(0.0f, 1.0f - cs * cs)), hw, cn > 0 ? 1.0f : 0.0f, 0.0f);
}

// A depth 0 < r < inf has bits(r) - 1 < DEPTH_LIM (unsigned; NaN, zeros and
// negative numbers do not), so a key below KEY_NONE is a valid depth's.
constexpr uint32_t DEPTH_LIM = 0x7f7fffffu;
constexpr unsigned long long KEY_NONE = (unsigned long long)DEPTH_LIM << 32;

// 1/x to the precision of the hardware's reciprocal; x neither denormal nor
// above 2^126: the quotient a * rcp_fast(x) is then __fdividef(a, x) bit for
// bit, without the instructions that scale its operands.
__device__ __forceinline__ float rcp_fast(float x)
{
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

// A thread's place in its tile: warp w covers the 8x8 block (w & 1, w >> 1),
// a lane the pixels (lx, ly) and (lx, ly + 4).
struct TilePos {
    int tx, ty, lx, ly, px, py;
    __device__ __forceinline__ TilePos(int tile, int tiles_x)
    {
        const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
        tx = tile % tiles_x;
        ty = tile / tiles_x;
        lx = (warp & 1) * 8 + (lane & 7);
        ly = (warp >> 1) * 8 + (lane >> 3);
        px = tx * TILE + lx;
        py = ty * TILE + ly;
    }
};

// The lane's pixels from the map (zero outside the picture).
__device__ __forceinline__ void load_pixels(const RasterView& view, const TilePos& tp, float4 (&g)[PPT])
{
#pragma unroll
    for (int p = 0; p < PPT; ++p) {
        const int y = tp.py + 4 * p;
        g[p] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        if (tp.px < view.W && y < view.H) g[p] = view.map[(size_t)y * view.W + tp.px];
    }
}

// The warps' view cones (their 8x8 pixels; block_cone), in shared memory: the
// cull reads them once per 32 triangles, and held in registers they would
// spill others out of the evaluation loop.
struct WarpCones {
    float4 c[RT / 32][2];
};

// Stage triangle t into slot j (an index beyond the records -- never left by a
// completed binning or grid -- empties the slot and raises the status).
__device__ __forceinline__ void stage_checked(const float4* rec, int T, uint32_t t, const float4& axis,
                                              Stage& st, int j, int* status)
{
    if (t >= (uint32_t)T) {
        raise_status(status, VSR_ERR_BIN_OVERFLOW);
        st.s6[j] = make_float4(0.0f, 0.0f, 0.0f, __uint_as_float(STAGE_EMPTY));
    } else {
        stage_triangle(rec, (size_t)T, t, axis.x, axis.y, axis.z, st, j);
    }
}

// Merge the lane's pixels into accumulator slot `slot` of a tile processed in
// several parts; the part that brings the count of `done` units to `target`
// gets the tile's result in q, clears the slot and returns true.  Called by
// every thread of the CTA.  SATURATES: the sum is a coverage, at most COV_ONE.
template <bool SATURATES = true, class Pix>
__device__ __forceinline__ bool merge_slot(const SplitAcc& split, int slot, const TilePos& tp, Pix& q,
                                           uint32_t units, uint32_t target)
{
    __shared__ int s_last;
    const int lp0 = tp.lx + TILE * tp.ly;
    unsigned long long* __restrict__ sacc = split.acc + (size_t)slot * TILE_PIX;
    unsigned long long* __restrict__ skey = split.key + (size_t)slot * TILE_PIX;
#pragma unroll
    for (int p = 0; p < PPT; ++p) {
        if (q.acc[p]) atomicAdd(&sacc[lp0 + TILE * 4 * p], (unsigned long long)q.acc[p]);
        if (q.key[p] != KEY_NONE) atomicMin(&skey[lp0 + TILE * 4 * p], q.key[p]);
    }
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) s_last = atomicAdd(&split.done[slot], units) + units == target;
    __syncthreads();
    if (!s_last) return false;
    __threadfence();
#pragma unroll
    for (int p = 0; p < PPT; ++p) {
        const unsigned long long sum = atomicExch(&sacc[lp0 + TILE * 4 * p], 0ull);
        q.acc[p] = (uint32_t)(SATURATES ? min(sum, (unsigned long long)COV_ONE) : sum);
        q.key[p] = min(atomicExch(&skey[lp0 + TILE * 4 * p], ~0ull), KEY_NONE);
    }
    if (threadIdx.x == 0) split.done[slot] = 0u;
    return true;
}

// ROWS: the outputs go through shared memory and leave in whole tile rows
// (pinned host outputs written in place over the host link).
template <bool ROWS, class Pix>
__device__ __forceinline__ void write_tile(const RasterView& view, const TilePos& tp, const Pix& q)
{
    const int W = view.W, H = view.H;
    if constexpr (!ROWS) {
#pragma unroll
        for (int p = 0; p < PPT; ++p) {
            if (tp.px >= W || tp.py + 4 * p >= H) continue;
            const size_t o = (size_t)(tp.py + 4 * p) * W + tp.px;
            const bool hit = q.key[p] != KEY_NONE;
            if (view.out_id) view.out_id[o] = hit ? (uint32_t)(q.key[p] & 0xffffffffull) : 0xffffffffu;
            if (view.out_depth) view.out_depth[o] = hit ? __uint_as_float((uint32_t)(q.key[p] >> 32) + 1u) : INFINITY;
            if (view.out_cov) view.out_cov[o] = (float)q.acc[p] * (1.0f / (float)COV_ONE);
        }
    } else {
        // Through shared memory, so that each warp store covers two whole tile
        // rows (16 pixels, 64 B each) instead of four 8-pixel pieces: over the
        // host link 32-byte pieces cost about a quarter of its bandwidth.
        __shared__ uint32_t s_out[3][TILE_PIX];
#pragma unroll
        for (int p = 0; p < PPT; ++p) {
            const int lp = tp.lx + TILE * (tp.ly + 4 * p);
            const bool hit = q.key[p] != KEY_NONE;
            s_out[0][lp] = hit ? (uint32_t)(q.key[p] & 0xffffffffull) : 0xffffffffu;
            s_out[1][lp] = hit ? (uint32_t)(q.key[p] >> 32) + 1u : __float_as_uint(INFINITY);
            s_out[2][lp] = __float_as_uint((float)q.acc[p] * (1.0f / (float)COV_ONE));
        }
        __syncthreads();
#pragma unroll
        for (int i = threadIdx.x; i < TILE_PIX; i += RT) {
            const int ox = tp.tx * TILE + (i % TILE), oy = tp.ty * TILE + i / TILE;
            if (ox >= W || oy >= H) continue;
            const size_t o = (size_t)oy * W + ox;
            if (view.out_id) view.out_id[o] = s_out[0][i];
            if (view.out_depth) view.out_depth[o] = __uint_as_float(s_out[1][i]);
            if (view.out_cov) view.out_cov[o] = __uint_as_float(s_out[2][i]);
        }
        __syncthreads();  // read before the CTA's next tile writes it
    }
}
