// grad.cu -- the differentiable path: per-pixel fragment lists, the
// front-to-back merge of a shade pass, and its hand-written adjoint.
//
// Forward (vsr_raster_shaded).  The image is the paper's front-to-back mask
// merge (Sec. 1.4) applied to a shade pass, shade_t = c_t |N-hat_t . G|
// (the hard normal of Sec. 1.1.4):
//   over the fragments of a pixel in ascending (r, t):
//     m^fc = min(m^f, 1 - m^b);  I += m^fc shade;  m^b += m^fc
// Unlike coverage, the image depends on the order, so every fragment is
// kept, as the float4 (r, t, m^f, shade), sorted per pixel.  Two launches:
//  * the count (FragCountStep, a walking raster) evaluates every pixel x
//    triangle pair, counts each pixel's fragments, takes the tile's range of
//    the lists with one atomic (so no scan over the pixels runs) and keeps
//    what the second launch needs: the tile's triangles and, per pixel, a bit
//    for each that is a fragment.  Ids and depths are final here.
//  * frag_fill_kernel evaluates only the triangles with a fragment in the
//    warp's block, sorts each pixel's fragments on their way in (shared
//    memory), writes and merges them.
// A tile with more than FRAG_LIST triangles or of several blocks of candidates
// keeps no list: where there are such tiles, a third launch (FragFillStep,
// again a walking raster) walks and evaluates them once more.
//
// Backward (vsr_raster_backward).  Per pixel, with upstream gradients dI,
// dcov, ddepth: the merge takes m^fc = m^f until the first fragment f* with
// m^f > 1 - m^b, which takes 1 - m^b and saturates the pixel, so
//   dI/d shade_f = m^fc_f,
//   dI/d m^f_f   = shade_f - shade_f* (f < f*; shade_f when nothing
//                  saturates), 0 from f* on,
//   dcov/d m^f_f = 1 when nothing saturates, else 0;
// m^f = clamp(delta min_i g_i + 1/2, 0, 1) (gpstep on the four plane
// distances) passes d g_i* = delta dm and d delta = g_i* dm to the
// minimising distance while the clamp is open; g_1..3 = G.n_i, g_4 =
// (G.S-hat - cos rho)/sin rho; depth r = (A'.N-hat)/(G.N-hat).  The
// per-triangle record gradients accumulate with float4 atomics; the
// per-pixel (dG, d delta) go to the map adjoint (map.cu), and the set-up
// adjoint below takes the record gradients to the world vertices.
#include <type_traits>

#include "raster_walk.cuh"

namespace {

static_assert(FRAG_LIST == STAGE_CHUNK && FRAG_LIST == 128, "a tile's list is one chunk, a pixel's bits four words");

__device__ __forceinline__ bool frag_less(const float4& a, const float4& b)
{
    return a.x < b.x || (a.x == b.x && __float_as_uint(a.y) < __float_as_uint(b.y));
}

// A lane's two pixels as the fragment kernels see them.
struct FragPix {
    float2 dgx, dgy, dgz, eg;  // G - a, |G|^2 - 1; 0 at an invalid pixel
    float delta[PPT], lim[PPT];  // as PixPair of raster.cu
};

__device__ __forceinline__ bool frag_start(const float4 (&g)[PPT], const float4& axis, FragPix& q, WarpCones& wc)
{
    float gx[PPT], gy[PPT], gz[PPT], h[PPT];
    bool pv[PPT];
#pragma unroll
    for (int p = 0; p < PPT; ++p) {
        pv[p] = g[p].w > 0.0f;
        gx[p] = g[p].x;
        gy[p] = g[p].y;
        gz[p] = g[p].z;
        h[p] = pv[p] ? 0.5f / g[p].w : 0.0f;
        q.delta[p] = g[p].w;
        q.lim[p] = pv[p] ? -h[p] : INFINITY;
    }
    q.dgx = make_float2(pv[0] ? gx[0] - axis.x : 0.0f, pv[1] ? gx[1] - axis.x : 0.0f);
    q.dgy = make_float2(pv[0] ? gy[0] - axis.y : 0.0f, pv[1] ? gy[1] - axis.y : 0.0f);
    q.dgz = make_float2(pv[0] ? gz[0] - axis.z : 0.0f, pv[1] ? gz[1] - axis.z : 0.0f);
    const float2 eg = norm2_minus_one2(make_float2(gx[0], gx[1]), make_float2(gy[0], gy[1]), make_float2(gz[0], gz[1]));
    q.eg = make_float2(pv[0] ? eg.x : 0.0f, pv[1] ? eg.y : 0.0f);
    float4 c0, c1;
    block_cone(gx, gy, gz, h, pv, c0, c1);
    if ((threadIdx.x & 31) == 0) {
        wc.c[threadIdx.x >> 5][0] = c0;
        wc.c[threadIdx.x >> 5][1] = c1;
    }
    __syncwarp();
    return c1.z > 0.0f;
}

// One staged triangle at the lane's pixels: the coverage kernel's distances
// and classification.
struct FragEval {
    float gm[PPT], r[PPT], D[PPT];
    bool f[PPT];
};
// false (for the whole warp): no fragment
__device__ __forceinline__ bool frag_eval(const Stage& st, int j, const FragPix& q, FragEval& o)
{
    const float4 b = st.s1[j], e = st.s6[j];
    const float2 g4 = miter_distance2(q.dgx, q.dgy, q.dgz, e, b, q.eg);
    const float2 g1 = plane_distance2(q.dgx, q.dgy, q.dgz, st.s2[j]);
    const float2 g2 = plane_distance2(q.dgx, q.dgy, q.dgz, st.s3[j]);
    const float2 g3 = plane_distance2(q.dgx, q.dgy, q.dgz, st.s4[j]);
    const float g3m[PPT] = {fminf(fminf(g1.x, g2.x), g3.x), fminf(fminf(g1.y, g2.y), g3.y)};
    o.gm[0] = fminf(g3m[0], g4.x);
    o.gm[1] = fminf(g3m[1], g4.y);
    const bool f0 = o.gm[0] > q.lim[0], f1 = o.gm[1] > q.lim[1];
    if (!__any_sync(0xffffffffu, f0 || f1)) return false;
    const float2 Dp = plane_distance2(q.dgx, q.dgy, q.dgz, st.s5[j]);
    o.D[0] = Dp.x;
    o.D[1] = Dp.y;
#pragma unroll
    for (int p = 0; p < PPT; ++p) {
        o.r[p] = __fdividef(b.w, o.D[p]);
        o.f[p] = (p ? f1 : f0) && __float_as_uint(o.r[p]) - 1u < DEPTH_LIM;  // 0 < r < inf
    }
    return true;
}

__device__ __forceinline__ float4 frag_record(const FragEval& o, const FragPix& q, int p, uint32_t t, float colour)
{
    return make_float4(o.r[p], __uint_as_float(t), __saturatef(fmaf(o.gm[p], q.delta[p], 0.5f)),
                       colour * fabsf(o.D[p]));
}

// Sorts a pixel's m fragments where they are stored, by (r, t), and merges
// them: the first CAP by insertion of their depths in shared memory (one column
// a thread), then each record into its place along the permutation's cycles;
// what is beyond CAP by insertion among the records.  Insertion of the records
// alone is a chain of dependent loads and stores that needs the lists in the
// L1, which holds those of a few CTAs.  A shaded forward of 1024 x 1024 pixels:
// 5000 triangles, 12 fragments a pixel, 1578 -> 540 us; 50k, 16 a pixel, 2630 ->
// 1055; 20k, 6 a pixel, 328 -> 222.  (Counting the smaller depths instead of
// inserting, with one move a turn for all lanes: 1577 us on the first.)
// OTHERS: other CTAs may have written the records, so the first read of each
// goes past the L1 (and it is stored again); such tiles are few, and insertion
// of the records is the faster one.
template <int CAP>
struct FragKeys {
    float r[CAP][RT];
    unsigned char at[CAP][RT];  // which record
};
template <bool OTHERS, int CAP>
__device__ __forceinline__ void frag_merge(const FragArgs& v, size_t pixel, float4* F, uint32_t m, FragKeys<CAP>& key)
{
    const uint32_t me = threadIdx.x, mk = OTHERS ? 0u : min(m, (uint32_t)CAP);
    for (uint32_t u = 0; u < mk; ++u) {
        const float r = F[u].x;
        uint32_t w = u;
        while (w > 0) {
            const float q = key.r[w - 1][me];
            const unsigned char a = key.at[w - 1][me];
            if (!(r < q || (r == q && __float_as_uint(F[u].y) < __float_as_uint(F[a].y)))) break;
            key.r[w][me] = q;
            key.at[w][me] = a;
            --w;
        }
        key.r[w][me] = r;
        key.at[w][me] = (unsigned char)u;
    }
    for (uint32_t u = 0; u < mk; ++u) {
        uint32_t from = key.at[u][me];
        if (from == u) continue;
        const float4 first = F[u];
        uint32_t to = u;
        while (from != u) {
            F[to] = F[from];
            key.at[to][me] = (unsigned char)to;
            to = from;
            from = key.at[to][me];
        }
        F[to] = first;
        key.at[to][me] = (unsigned char)to;
    }
    for (uint32_t u = mk; u < m; ++u) {
        const float4 x = OTHERS ? __ldcg(F + u) : F[u];
        uint32_t w = u;
        while (w > 0 && frag_less(x, F[w - 1])) {
            F[w] = F[w - 1];
            --w;
        }
        F[w] = x;
    }
    float mb = 0.0f, img = 0.0f;
    for (uint32_t u = 0; u < m && mb < 1.0f; ++u) {
        const float4 x = F[u];
        const float mfc = fminf(x.z, 1.0f - mb);
        img = fmaf(mfc, x.w, img);
        mb += mfc;
    }
    if (v.image) v.image[pixel] = img;
    if (v.cov) v.cov[pixel] = mb;
}

// One staged triangle in the count: as the coverage kernel's evaluation
// (eval_slot of raster.cu), with a count and a bit in place of the coverage.
struct FragCount : FragPix {
    uint32_t acc[PPT], bits[PPT];  // fragments; those of the current group of 32 slots
    unsigned long long key[PPT];   // ((bits(r) - 1) << 32) | t of the nearest centre-inside fragment, or KEY_NONE
};
__device__ __forceinline__ void frag_count(const Stage& st, int j, FragCount& q)
{
    const float4 b = st.s1[j], e = st.s6[j];
    const float2 g4 = miter_distance2(q.dgx, q.dgy, q.dgz, e, b, q.eg);
    const float2 g1 = plane_distance2(q.dgx, q.dgy, q.dgz, st.s2[j]);
    const float2 g2 = plane_distance2(q.dgx, q.dgy, q.dgz, st.s3[j]);
    const float2 g3 = plane_distance2(q.dgx, q.dgy, q.dgz, st.s4[j]);
    const float g3m[PPT] = {fminf(fminf(g1.x, g2.x), g3.x), fminf(fminf(g1.y, g2.y), g3.y)};
    const bool f[PPT] = {fminf(g3m[0], g4.x) > q.lim[0], fminf(g3m[1], g4.y) > q.lim[1]};
    if (!__any_sync(0xffffffffu, f[0] || f[1])) return;
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
            const bool frag = f[p] && rq[p] < DEPTH_LIM;
            q.acc[p] += frag;
            q.bits[p] |= (frag ? 1u : 0u) << (j & 31);
            inn[p] = f[p] && g3m[p] > 0.0f;
            if (RARE && f[p] && g3m[p] == 0.0f) {
                const float dx = p ? q.dgx.y : q.dgx.x, dy = p ? q.dgy.y : q.dgy.x, dz = p ? q.dgz.y : q.dgz.x;
                inn[p] = centre_inside(plane_distance(dx, dy, dz, st.s2[j]), plane_distance(dx, dy, dz, st.s3[j]),
                                       plane_distance(dx, dy, dz, st.s4[j]), g3m[p], __float_as_uint(st.s0[j].w));
            }
        }
        if (__any_sync(0xffffffffu, inn[0] || inn[1])) {
#pragma unroll
            for (int p = 0; p < PPT; ++p) {
                const unsigned long long kk = ((unsigned long long)rq[p] << 32) | __float_as_uint(e.w);
                q.key[p] = inn[p] && kk < q.key[p] ? kk : q.key[p];
            }
        }
    };
    const float tiny = fminf(fminf(fabsf(g3m[0]), fabsf(g3m[1])), fminf(fabsf(D[0]), fabsf(D[1])));
    if (__any_sync(0xffffffffu, tiny < 1.17549435e-38f))
        post(std::true_type{});
    else
        post(std::false_type{});
}

// The count as a step of the walking raster, so tiles of many candidates are
// shared between CTAs here too (see raster_walk_kernel).  A frame with its
// backward: 145 -> 138 us at 1024 x 1024 with 10k triangles, where no tile is
// shared; 3.8 -> 1.4 ms at 128 x 128 with 300k triangles, where all are.
struct FragStep {
    using Cones = WarpCones;
    using In = FragArgs;
    static constexpr int FEW_BLOCK = WALK_BLOCK;  // a tile of one block can keep its list
    static constexpr bool SATURATES = false, HOST_OUT = false;
    __device__ __forceinline__ static bool cull(const Stage& st, int j, const Cones& wc, int warp)
    {
        return cone_may_hit(st.s0[j], st.s1[j], st.s2[j], st.s3[j], st.s4[j], wc.c[warp][0], wc.c[warp][1], false);
    }
};

struct FragCountStep : FragStep {
    static constexpr bool SKIPS = false;
    static constexpr int FEW_FROM = 2, SHARE_FROM = 3;
    static constexpr int CTAS = 8;  // 64 registers; 7: 40.2 us, 6: 44.0 us against 39.4 us
    using Pix = FragCount;
    using Ctx = WalkCtx<FragArgs>;
    struct Raw {
        float4 g[PPT];
    };
    __device__ __forceinline__ static void load(const RasterView& view, const In&, const TilePos& tp, Raw& r)
    {
        load_pixels(view, tp, r.g);
    }
    __device__ __forceinline__ static bool start(const Raw& r, const float4& axis, Pix& q, Cones& wc)
    {
        q.acc[0] = q.acc[1] = q.bits[0] = q.bits[1] = 0u;
        q.key[0] = q.key[1] = KEY_NONE;
        return frag_start(r.g, axis, q, wc);
    }
    __device__ __forceinline__ static bool skip(const In&, int) { return false; }
    __device__ __forceinline__ static void clamp(Pix&) {}
    __device__ __forceinline__ static void eval(const Ctx&, const Stage& st, int j, Pix& q) { frag_count(st, j, q); }
    __device__ __forceinline__ static uint32_t final_acc(const Pix& q, int p) { return q.acc[p]; }
    // does the tile keep a list?  (known with its only block's hits)
    __device__ __forceinline__ static bool list(const Ctx& cx)
    {
        return cx.wt.nblk <= 1u && cx.wt.slot < 0 && cx.wt.n <= (uint32_t)FRAG_LIST;
    }
    __device__ __forceinline__ static void group(const Ctx& cx, int g, Pix& q)
    {
        if (list(cx)) {
            const FragArgs& v = cx.in;
            const TilePos tp(cx.wt.tile, v.tiles_x);
#pragma unroll
            for (int p = 0; p < PPT; ++p)
                if (tp.px < v.W && tp.py + 4 * p < v.H)
                    v.bits[((size_t)g * v.H + tp.py + 4 * p) * v.W + tp.px] = q.bits[p];
        }
        q.bits[0] = q.bits[1] = 0u;
    }
    // the tile's range of the lists, its pixels in thread order
    template <bool ROWS>
    __device__ __forceinline__ static void finish(const Ctx& cx, const TilePos& tp, const Pix& q, int*)
    {
        __shared__ uint32_t s_sum[RT / 32], s_base;
        const FragArgs& v = cx.in;
        const int tile = cx.wt.tile, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
        const uint32_t mine = q.acc[0] + q.acc[1];
        uint32_t incl = mine;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += y;
        }
        if (lane == 31) s_sum[warp] = incl;
        __syncthreads();
        uint32_t before = 0, total = 0;
#pragma unroll
        for (int w = 0; w < RT / 32; ++w) {
            if (w < warp) before += s_sum[w];
            total += s_sum[w];
        }
        const bool keep = list(cx);
        const uint32_t n = cx.wt.n;
        if (threadIdx.x == 0) {
            s_base = total ? atomicAdd(v.cursor, total) : 0u;
            v.tile_n[tile] = keep ? n : 0xffffffffu;
            if (!keep) atomicAdd(v.cursor + 1, 1u);
        }
        if (keep && threadIdx.x < n) v.tile_ids[(size_t)tile * FRAG_LIST + threadIdx.x] = cx.ids[threadIdx.x];
        __syncthreads();
        uint32_t off = s_base + before + incl - mine;
#pragma unroll
        for (int p = 0; p < PPT; ++p) {
            if (tp.px < v.W && tp.py + 4 * p < v.H) {
                const size_t o = (size_t)(tp.py + 4 * p) * v.W + tp.px;
                v.span[o] = make_uint2(off, q.acc[p]);
                const bool hit = q.key[p] != KEY_NONE;
                if (v.out_id) v.out_id[o] = hit ? (uint32_t)(q.key[p] & 0xffffffffull) : 0xffffffffu;
                if (v.out_depth) v.out_depth[o] = hit ? __uint_as_float((uint32_t)(q.key[p] >> 32) + 1u) : INFINITY;
            }
            off += q.acc[p];
        }
    }
};

// The fill of the tiles without a list: walked and evaluated again, fragments
// appended to their pixels' lists in any order (a shared tile's parts take
// their places from the slot's accumulators) and sorted by the part that
// finishes the tile.
struct FragAppend : FragPix {
    uint32_t at[PPT], room[PPT];  // the pixel's list
    uint32_t acc[PPT];            // fragments appended (a shared tile: counted in its slot)
    unsigned long long key[PPT];  // unused
};
struct FragFillStep : FragStep {
    static constexpr bool SKIPS = true;
    // Shared from the seventh block on: in a shared tile every fragment waits
    // for its place from an atomic.  A shaded forward with sharing from the
    // third, seventh, eleventh block: 5000 triangles of 0.3 rad at 64x64 484,
    // 334, 335 us; 50k of 0.1 rad at 256x256 486, 417, 412; 100k small ones at
    // 128x128 652, 578, 575; 300k 1243, 1233, 1514.
    static constexpr int FEW_FROM = 6, SHARE_FROM = 6;
    static constexpr int CTAS = 5;
    using Pix = FragAppend;
    using Ctx = WalkCtx<FragArgs>;
    struct Raw {
        float4 g[PPT];
        uint32_t at[PPT], room[PPT];
    };
    __device__ __forceinline__ static void load(const RasterView& view, const In& v, const TilePos& tp, Raw& r)
    {
        load_pixels(view, tp, r.g);
#pragma unroll
        for (int p = 0; p < PPT; ++p) {
            uint2 s = make_uint2(0u, 0u);
            if (tp.px < v.W && tp.py + 4 * p < v.H) s = v.span[(size_t)(tp.py + 4 * p) * v.W + tp.px];
            r.at[p] = s.x;
            r.room[p] = (uint64_t)s.x + s.y <= v.fcap ? s.y : 0u;  // (finish reports a list cut short)
        }
    }
    __device__ __forceinline__ static bool start(const Raw& r, const float4& axis, Pix& q, Cones& wc)
    {
#pragma unroll
        for (int p = 0; p < PPT; ++p) {
            q.at[p] = r.at[p];
            q.room[p] = r.room[p];
            q.acc[p] = 0u;
            q.key[p] = KEY_NONE;
        }
        return frag_start(r.g, axis, q, wc);
    }
    __device__ __forceinline__ static bool skip(const In& v, int tile) { return v.tile_n[tile] <= (uint32_t)FRAG_LIST; }
    __device__ __forceinline__ static void clamp(Pix&) {}
    __device__ __forceinline__ static void group(const Ctx&, int, Pix&) {}
    __device__ __forceinline__ static uint32_t final_acc(const Pix& q, int p) { return q.acc[p]; }
    __device__ __forceinline__ static void eval(const Ctx& cx, const Stage& st, int j, Pix& q)
    {
        FragEval o;
        if (!frag_eval(st, j, q, o)) return;
        const FragArgs& v = cx.in;
        const uint32_t t = __float_as_uint(st.s6[j].w);
        const float colour = v.colors ? v.colors[t] : 1.0f;
        const int slot = cx.wt.slot;
        const TilePos tp(0, 1);
#pragma unroll
        for (int p = 0; p < PPT; ++p) {
            if (!o.f[p]) continue;
            const uint32_t u = slot < 0 ? q.acc[p]++
                                        : (uint32_t)atomicAdd(&cx.slots.split.acc[(size_t)slot * TILE_PIX + tp.lx +
                                                                                  TILE * (tp.ly + 4 * p)],
                                                              1ull);
            if (u < q.room[p]) v.frags[(size_t)q.at[p] + u] = frag_record(o, q, p, t, colour);
        }
    }
    template <bool ROWS>
    __device__ __forceinline__ static void finish(const Ctx& cx, const TilePos& tp, const Pix& q, int* status)
    {
        using Keys = FragKeys<sizeof(Stage) / (5 * RT)>;
        static_assert(sizeof(Keys) <= sizeof(Stage), "the keys take the triangles' place");
        Keys& key = *(Keys*)&cx.stage;
        const FragArgs& v = cx.in;
        const bool shared = cx.wt.slot >= 0;
        __syncthreads();  // no warp evaluates any more
#pragma unroll 1
        for (int p = 0; p < PPT; ++p) {
            if (tp.px >= v.W || tp.py + 4 * p >= v.H) continue;
            const uint32_t n = p ? q.acc[1] : q.acc[0], room = p ? q.room[1] : q.room[0];
            // spans of another frame, or no room (see FragArgs::early)
            if (n != room && !(v.early && room == 0u)) raise_status(status, VSR_ERR_FRAG_OVERFLOW);
            const size_t o = (size_t)(tp.py + 4 * p) * v.W + tp.px;
            float4* F = v.frags + (p ? q.at[1] : q.at[0]);
            if (shared)
                frag_merge<true>(v, o, F, min(n, room), key);
            else
                frag_merge<false>(v, o, F, min(n, room), key);
        }
    }
};

// fragments of a pixel sorted in shared memory as they are found; a longer list
// is stored and then sorted (frag_merge, its keys in the same memory)
constexpr uint32_t FRAG_SORT = 8;
struct FillBuffers {
    Stage st;
    float4 rec[FRAG_SORT][RT];
};
using FillKeys = FragKeys<sizeof(FillBuffers) / (RT * 5)>;
union __align__(16) FillShared {
    FillBuffers b;
    FillKeys key;
    __device__ FillShared() {}
};

// The fill of the tiles with a list: the evaluations that are fragments, no
// walk and no cull.  Bound by issue with lanes idle (each triangle's step runs
// for the pixels that have it) and by the sort; 1024 x 1024, 10k triangles:
// 28.7 us, 59.7 when every pair was evaluated again and sorted where it was
// stored, 33.8 while one kernel held the walk of the other tiles too (92
// registers instead of 72).
__global__ void __launch_bounds__(RT, 6) frag_fill_kernel(FragArgs v)
{
    grid_wait();
    grid_go();
    __shared__ FillShared sh;
    Stage& st = sh.b.st;
    float4 (&rec)[FRAG_SORT][RT] = sh.b.rec;
    __shared__ float scol[STAGE_CHUNK];
    __shared__ WarpCones wc;
    const unsigned FULL = 0xffffffffu;
    const int tile = blockIdx.x;
    const TilePos tp(tile, v.tiles_x);
    if (tile == 0 && threadIdx.x < 2) v.cursor[threadIdx.x] = 0u;  // for the next frame
    const uint32_t n = v.tile_n[tile];
    if (n > (uint32_t)FRAG_LIST) return;
    const Cone tc = v.tiles[tile];
    if (threadIdx.x < n) {
        const uint32_t t = v.tile_ids[(size_t)tile * FRAG_LIST + threadIdx.x];
        stage_checked(v.rec, v.T, t, tc.c0, st, threadIdx.x, v.status);
        scol[threadIdx.x] = v.colors && t < (uint32_t)v.T ? v.colors[t] : 1.0f;
    }
    float4 gp[PPT];
    uint2 span[PPT] = {};
    bool inimg[PPT];
#pragma unroll
    for (int p = 0; p < PPT; ++p) {
        inimg[p] = tp.px < v.W && tp.py + 4 * p < v.H;
        gp[p] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        if (inimg[p]) {
            gp[p] = v.map[(size_t)(tp.py + 4 * p) * v.W + tp.px];
            span[p] = v.span[(size_t)(tp.py + 4 * p) * v.W + tp.px];
        }
    }
    FragPix q;
    frag_start(gp, tc.c0, q, wc);
    // (beyond the buffer: only before the host has sized it)
    const bool fits = (uint64_t)span[0].x + span[0].y <= v.fcap && (uint64_t)span[1].x + span[1].y <= v.fcap;
    if (!fits) {
        if (!v.early) raise_status(v.status, VSR_ERR_FRAG_OVERFLOW);
        span[0].y = span[1].y = 0u;
    }
    uint4 bits[PPT];
#pragma unroll
    for (int p = 0; p < PPT; ++p) {
        const uint32_t* at = v.bits + (size_t)(tp.py + 4 * p) * v.W + tp.px;
        const size_t pic = (size_t)v.H * v.W;
        const bool some = inimg[p] && span[p].y;
        bits[p].x = some ? at[0] : 0u;
        bits[p].y = some && n > 32u ? at[pic] : 0u;
        bits[p].z = some && n > 64u ? at[2 * pic] : 0u;
        bits[p].w = some && n > 96u ? at[3 * pic] : 0u;
    }
    __syncthreads();
    // (one pixel's list at a time in shared memory: the first pixels of
    // the lanes, then the second)
    unsigned longer = 0u;  // pixels with a longer list
#pragma unroll
    for (int p = 0; p < PPT; ++p) {
        const bool sorted = span[p].y <= FRAG_SORT;
        uint32_t cnt = 0u;
#pragma unroll
        for (int g = 0; g < FRAG_LIST / 32; ++g) {
            const uint32_t b = g == 0 ? bits[p].x : (g == 1 ? bits[p].y : (g == 2 ? bits[p].z : bits[p].w));
            unsigned any = __reduce_or_sync(FULL, b);
            while (any) {
                const int k = 31 - __clz(any);
                any ^= 1u << k;
                const int j = 32 * g + k;
                if (!(b >> k & 1u)) continue;
                // this pixel's distances in scalar form (bit for bit the packed ones)
                const float dx = p ? q.dgx.y : q.dgx.x, dy = p ? q.dgy.y : q.dgy.x, dz = p ? q.dgz.y : q.dgz.x;
                const float4 c = st.s1[j], e = st.s6[j];
                const float g4 = miter_distance(dx, dy, dz, e, c, p ? q.eg.y : q.eg.x);
                const float g3m = fminf(fminf(plane_distance(dx, dy, dz, st.s2[j]), plane_distance(dx, dy, dz, st.s3[j])),
                                        plane_distance(dx, dy, dz, st.s4[j]));
                const float D = plane_distance(dx, dy, dz, st.s5[j]);
                const float4 x = make_float4(__fdividef(c.w, D), e.w, __saturatef(fmaf(fminf(g3m, g4), q.delta[p], 0.5f)),
                                             scol[j] * fabsf(D));
                if (cnt < span[p].y) {  // (else spans of another frame: reported below)
                    uint32_t u = cnt;
                    if (sorted) {
                        while (u > 0 && frag_less(x, rec[u - 1][threadIdx.x])) {
                            rec[u][threadIdx.x] = rec[u - 1][threadIdx.x];
                            --u;
                        }
                        rec[u][threadIdx.x] = x;
                    } else {
                        v.frags[(size_t)span[p].x + u] = x;
                    }
                }
                ++cnt;
            }
        }
        if (!inimg[p]) continue;
        if (fits && cnt != span[p].y) raise_status(v.status, VSR_ERR_FRAG_OVERFLOW);  // spans of another frame
        const size_t o = (size_t)(tp.py + 4 * p) * v.W + tp.px;
        const uint32_t m = min(cnt, span[p].y);
        if (!sorted) {
            span[p].y = m;  // below, with every warp done with the triangles
            longer |= 1u << p;
            continue;
        }
        // the pixel's merge, and its list
        float mb = 0.0f, img = 0.0f;
        for (uint32_t u = 0; u < m; ++u) {
            const float4 x = rec[u][threadIdx.x];
            v.frags[(size_t)span[p].x + u] = x;
            if (mb < 1.0f) {
                const float mfc = fminf(x.z, 1.0f - mb);
                img = fmaf(mfc, x.w, img);
                mb += mfc;
            }
        }
        if (v.image) v.image[o] = img;
        if (v.cov) v.cov[o] = mb;
    }
    if (!__syncthreads_or(longer)) return;
#pragma unroll 1
    for (int p = 0; p < PPT; ++p)
        if (longer >> p & 1u)
            frag_merge<false>(v, (size_t)(tp.py + 4 * p) * v.W + tp.px, v.frags + (p ? span[1].x : span[0].x),
                              p ? span[1].y : span[0].y, sh.key);
}

// ---------------------------------------------------------------------------
// Backward, per pixel.

struct BackView {
    const float4* map;
    int W, H;
    const float4* rec;
    int T;
    const float* colors;
    const uint2* span;
    const float4* frags;
    const uint32_t* id;
    const float* dimage;
    const float* dcov;
    const float* ddepth;
    float4* grad;  // GF_COUNT x T, field-major
    float4* dmap;  // per pixel (dG, d delta)
};

__device__ __forceinline__ float dot3f(float ax, float ay, float az, const float4& b)
{
    return fmaf(ax, b.x, fmaf(ay, b.y, az * b.z));
}

__global__ void __launch_bounds__(TILE_PIX) frag_backward_kernel(BackView v)
{
    grid_wait();
    grid_go();
    const int i = blockIdx.x * TILE + (threadIdx.x % TILE);
    const int j = blockIdx.y * TILE + (threadIdx.x / TILE);
    if (i >= v.W || j >= v.H) return;
    const size_t o = (size_t)j * v.W + i;
    const float4 g = v.map[o];
    float4 dG = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    if (!(g.w > 0.0f)) {
        v.dmap[o] = dG;
        return;
    }
    const size_t TT = (size_t)v.T;
    const float dI = v.dimage ? v.dimage[o] : 0.0f;
    const float dC = v.dcov ? v.dcov[o] : 0.0f;
    const float dD = v.ddepth ? v.ddepth[o] : 0.0f;
    const uint2 span = v.span[o];
    const uint32_t n = span.y;
    const float4* F = v.frags + span.x;

    // the saturating fragment, replaying the forward merge's arithmetic
    uint32_t fstar = n;
    float sstar = 0.0f, mb = 0.0f;
    for (uint32_t q = 0; q < n; ++q) {
        const float4 x = F[q];
        if (x.z > 1.0f - mb) {
            fstar = q;
            sstar = x.w;
            break;
        }
        mb += x.z;
    }
    const float beta = fstar < n ? -dI * sstar : dC;
    const uint32_t last = fstar < n ? fstar + 1 : n;
    mb = 0.0f;
    for (uint32_t q = 0; q < last; ++q) {
        const float4 x = F[q];
        const uint32_t t = __float_as_uint(x.y);
        float dm, dsh;
        if (q == fstar) {
            dm = 0.0f;
            dsh = dI * (1.0f - mb);
        } else {
            dm = fmaf(dI, x.w, beta);
            dsh = dI * x.z;
            mb += x.z;
        }
        if (dm != 0.0f && x.z > 0.0f && x.z < 1.0f) {
            // the minimising distance (any one of equal minima is a valid
            // subgradient); the forward's g_min from its own m^f
            const float4 n1 = v.rec[rec_at(TT, t, RF_N1)], n2 = v.rec[rec_at(TT, t, RF_N2)], n3 = v.rec[rec_at(TT, t, RF_N3)];
            const float4 cp = v.rec[rec_at(TT, t, RF_CAP)], cp2 = v.rec[rec_at(TT, t, RF_CAP2)];
            const float g1 = dot3f(g.x, g.y, g.z, n1), g2 = dot3f(g.x, g.y, g.z, n2), g3 = dot3f(g.x, g.y, g.z, n3);
            const float mx = g.x - cp.x, my = g.y - cp.y, mz = g.z - cp.z;
            const float g4 = (cp2.y - fmaf(mx, mx, fmaf(my, my, mz * mz))) * cp2.z;
            int is = 0;
            float gmin = g1;
            if (g2 < gmin) { gmin = g2; is = 1; }
            if (g3 < gmin) { gmin = g3; is = 2; }
            if (g4 < gmin) { gmin = g4; is = 3; }
            const float gm = (x.z - 0.5f) / g.w;
            const float dg = dm * g.w;
            dG.w = fmaf(dm, gm, dG.w);
            if (is < 3) {
                const float4 nn = is == 0 ? n1 : (is == 1 ? n2 : n3);
                atomicAdd(&v.grad[(GF_N1 + is) * TT + t], make_float4(dg * g.x, dg * g.y, dg * g.z, 0.0f));
                dG.x = fmaf(dg, nn.x, dG.x);
                dG.y = fmaf(dg, nn.y, dG.y);
                dG.z = fmaf(dg, nn.z, dG.z);
            } else {
                const float sr = cp2.x, c = cp.w;
                const float q4 = dg / sr;
                atomicAdd(&v.grad[GF_CAP * TT + t],
                          make_float4(q4 * g.x, q4 * g.y, q4 * g.z, q4 * fmaf(g4 / sr, c, -1.0f)));
                dG.x = fmaf(q4, cp.x, dG.x);
                dG.y = fmaf(q4, cp.y, dG.y);
                dG.z = fmaf(q4, cp.z, dG.z);
            }
        }
        if (dsh != 0.0f) {
            const float4 pl = v.rec[rec_at(TT, t, RF_PL)];
            const float u = dot3f(g.x, g.y, g.z, pl);
            const float col = v.colors ? v.colors[t] : 1.0f;
            const float du = u > 0.0f ? dsh * col : (u < 0.0f ? -dsh * col : 0.0f);
            atomicAdd(&v.grad[GF_PL * TT + t], make_float4(du * g.x, du * g.y, du * g.z, dsh * fabsf(u)));
            dG.x = fmaf(du, pl.x, dG.x);
            dG.y = fmaf(du, pl.y, dG.y);
            dG.z = fmaf(du, pl.z, dG.z);
        }
    }
    if (dD != 0.0f && v.id) {
        const uint32_t t = v.id[o];
        if (t < (uint32_t)v.T) {
            const float4 pl = v.rec[rec_at(TT, t, RF_PL)];
            const float u = dot3f(g.x, g.y, g.z, pl);
            const float r = pl.w / u;
            const float dGN = -dD * r / u;
            atomicAdd(&v.grad[GF_PL * TT + t], make_float4(dGN * g.x, dGN * g.y, dGN * g.z, 0.0f));
            atomicAdd(&v.grad[GF_D * TT + t].x, dD / u);
            dG.x = fmaf(dGN, pl.x, dG.x);
            dG.y = fmaf(dGN, pl.y, dG.y);
            dG.z = fmaf(dGN, pl.z, dG.z);
        }
    }
    v.dmap[o] = dG;
}

// ---------------------------------------------------------------------------
// Set-up adjoint, per triangle: record gradients -> world vertices.
//   n_e = sigma x/|x|, x = P' x Q'  =>  dx = sigma (dn - x^ (x^.dn))/|x|,
//                                       dP' += Q' x dx, dQ' += dx x P'
//   S-hat = S/|S|, c = |S|          =>  dS = (dS^ - S^ (S^.dS^))/|S| + S^ dc
//   S = midpoint or (Os A^ + Ot B^ + Op C^)/(Os + Ot + Op) of the unit
//   vertices U = V/|V| (Sec. 1.1.2), differentiated through the squared
//   chords a^2, b^2, c^2
//   N-hat = N/|N|, N = (A' - B') x (C' - B'), d' = A'.N-hat
//   X' = M (X - O)                  =>  dX = M^T dX'
// Plain FP32 throughout: the forward quantities are recomputed from the
// world vertices, sigma is read off the stored normal.

struct F3 {
    float x, y, z;
};
__device__ __forceinline__ F3 f3(float x, float y, float z) { return F3{x, y, z}; }
__device__ __forceinline__ F3 operator+(F3 a, F3 b) { return f3(a.x + b.x, a.y + b.y, a.z + b.z); }
__device__ __forceinline__ F3 operator-(F3 a, F3 b) { return f3(a.x - b.x, a.y - b.y, a.z - b.z); }
__device__ __forceinline__ F3 operator*(float s, F3 a) { return f3(s * a.x, s * a.y, s * a.z); }
__device__ __forceinline__ float dot(F3 a, F3 b) { return fmaf(a.x, b.x, fmaf(a.y, b.y, a.z * b.z)); }
__device__ __forceinline__ F3 cross(F3 a, F3 b)
{
    return f3(a.y * b.z - a.z * b.y, a.z * b.x - a.x * b.z, a.x * b.y - a.y * b.x);
}
__device__ __forceinline__ F3 xyz(float4 a) { return f3(a.x, a.y, a.z); }
// gradient of u = x/|x| pulled back to x
__device__ __forceinline__ F3 unit_back(F3 u, float len, F3 du) { return (1.0f / len) * (du - dot(u, du) * u); }

struct CamF {
    float O[3];
    float M[9];
};

__global__ void __launch_bounds__(128) setup_backward_kernel(const float* tris, int T, CamF cam,
                                                              const float4* rec,
                                                              float4* __restrict__ grad,
                                                              float* __restrict__ dtris, float* __restrict__ dcolors)
{
    grid_wait();
    grid_go();
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= T) return;
    const size_t TT = (size_t)T;
    const float4 cp2 = rec[rec_at(TT, t, RF_CAP2)];
    float* out = dtris ? dtris + (size_t)t * 9 : nullptr;
    // The record's gradient, cleared for the next backward where it holds
    // anything: most fields of most triangles are zero already (hidden, or no
    // pixel at that edge), and a store between the loads makes them a chain.  A
    // backward to the vertices of 1M triangles, 640x480: 334 us with a load and
    // a store per field, 214 with the stores after the loads, 103 like this (140
    // with a memset per call instead); of 10k, 1024x1024: 25.9, 25.1, 25.0 us.
    float4 gr[GF_COUNT];
#pragma unroll
    for (int q = 0; q < GF_COUNT; ++q) gr[q] = grad[q * TT + t];
#pragma unroll
    for (int q = 0; q < GF_COUNT; ++q)
        if (gr[q].x != 0.0f || gr[q].y != 0.0f || gr[q].z != 0.0f || gr[q].w != 0.0f)
            grad[q * TT + t] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    const float4 gpl = gr[GF_PL];
    if (dcolors) dcolors[t] = cp2.w != 0.0f ? gpl.w : 0.0f;
    if (!out) return;
    if (cp2.w == 0.0f) {  // culled at set-up: no fragments, no gradient
#pragma unroll
        for (int q = 0; q < 9; ++q) out[q] = 0.0f;
        return;
    }
    F3 V[3], dV[3];
#pragma unroll
    for (int q = 0; q < 3; ++q) {
        const float d0 = tris[(size_t)t * 9 + 3 * q] - cam.O[0];
        const float d1 = tris[(size_t)t * 9 + 3 * q + 1] - cam.O[1];
        const float d2 = tris[(size_t)t * 9 + 3 * q + 2] - cam.O[2];
        V[q] = f3(fmaf(cam.M[0], d0, fmaf(cam.M[1], d1, cam.M[2] * d2)),
                  fmaf(cam.M[3], d0, fmaf(cam.M[4], d1, cam.M[5] * d2)),
                  fmaf(cam.M[6], d0, fmaf(cam.M[7], d1, cam.M[8] * d2)));
        dV[q] = f3(0.0f, 0.0f, 0.0f);
    }
    // edge normals
    const float4 n1s = rec[rec_at(TT, t, RF_N1)];
    const F3 x0 = cross(V[0], V[1]);
    const float sigma = dot(xyz(n1s), x0) < 0.0f ? -1.0f : 1.0f;
#pragma unroll
    for (int e = 0; e < 3; ++e) {
        const int P = e, Q = e == 2 ? 0 : e + 1;
        const F3 x = cross(V[P], V[Q]);
        const float len = sqrtf(dot(x, x));
        const F3 dn = xyz(gr[GF_N1 + e]);
        const F3 dx = sigma * unit_back((1.0f / len) * x, len, dn);
        dV[P] = dV[P] + cross(V[Q], dx);
        dV[Q] = dV[Q] + cross(dx, V[P]);
    }
    // miter
    const float4 gcap = gr[GF_CAP];
    if (gcap.x != 0.0f || gcap.y != 0.0f || gcap.z != 0.0f || gcap.w != 0.0f) {
        F3 U[3];
        float Ul[3];
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            Ul[q] = sqrtf(dot(V[q], V[q]));
            U[q] = (1.0f / Ul[q]) * V[q];
        }
        const F3 ea = U[1] - U[2], eb = U[2] - U[0], ec = U[0] - U[1];
        const float a2 = dot(ea, ea), b2 = dot(eb, eb), c2 = dot(ec, ec);
        const float Os = a2 * (b2 + c2 - a2), Ot = b2 * (c2 + a2 - b2), Op = c2 * (a2 + b2 - c2);
        F3 S;
        const bool mid = Os <= 0.0f || Ot <= 0.0f || Op <= 0.0f;
        const int ma = Os <= 0.0f ? 1 : (Ot <= 0.0f ? 2 : 0);
        const int mbi = Os <= 0.0f ? 2 : (Ot <= 0.0f ? 0 : 1);
        const float sum = Os + Ot + Op;
        if (mid)
            S = 0.5f * (U[ma] + U[mbi]);
        else
            S = (1.0f / sum) * (Os * U[0] + Ot * U[1] + Op * U[2]);
        const float slen = sqrtf(dot(S, S));
        const F3 Sh = (1.0f / slen) * S;
        const F3 dS = unit_back(Sh, slen, xyz(gcap)) + gcap.w * Sh;
        F3 dU[3] = {f3(0.0f, 0.0f, 0.0f), f3(0.0f, 0.0f, 0.0f), f3(0.0f, 0.0f, 0.0f)};
        if (mid) {
            dU[ma] = 0.5f * dS;
            dU[mbi] = 0.5f * dS;
        } else {
            const float Oq[3] = {Os, Ot, Op};
            float dO[3];
#pragma unroll
            for (int q = 0; q < 3; ++q) {
                dO[q] = dot(dS, U[q] - S) / sum;
                dU[q] = (Oq[q] / sum) * dS;
            }
            const float da2 = dO[0] * (b2 + c2 - 2.0f * a2) + dO[1] * b2 + dO[2] * c2;
            const float db2 = dO[0] * a2 + dO[1] * (c2 + a2 - 2.0f * b2) + dO[2] * c2;
            const float dc2 = dO[0] * a2 + dO[1] * b2 + dO[2] * (a2 + b2 - 2.0f * c2);
            dU[1] = dU[1] + (2.0f * da2) * ea;
            dU[2] = dU[2] - (2.0f * da2) * ea;
            dU[2] = dU[2] + (2.0f * db2) * eb;
            dU[0] = dU[0] - (2.0f * db2) * eb;
            dU[0] = dU[0] + (2.0f * dc2) * ec;
            dU[1] = dU[1] - (2.0f * dc2) * ec;
        }
#pragma unroll
        for (int q = 0; q < 3; ++q) dV[q] = dV[q] + unit_back(U[q], Ul[q], dU[q]);
    }
    // plane: shade uses N-hat, depth r = d'/(G.N-hat) with d' = A'.N-hat
    const float dd = gr[GF_D].x;
    const F3 e1 = V[0] - V[1], e2 = V[2] - V[1];
    const F3 N = cross(e1, e2);
    const float nl = sqrtf(dot(N, N));
    const F3 Nh = (1.0f / nl) * N;
    const F3 dNh = xyz(gpl) + dd * V[0];
    dV[0] = dV[0] + dd * Nh;
    const F3 dN = unit_back(Nh, nl, dNh);
    const F3 de1 = cross(e2, dN), de2 = cross(dN, e1);
    dV[0] = dV[0] + de1;
    dV[2] = dV[2] + de2;
    dV[1] = dV[1] - (de1 + de2);
    // world: dX = M^T dX'
#pragma unroll
    for (int q = 0; q < 3; ++q) {
        out[3 * q + 0] = fmaf(cam.M[0], dV[q].x, fmaf(cam.M[3], dV[q].y, cam.M[6] * dV[q].z));
        out[3 * q + 1] = fmaf(cam.M[1], dV[q].x, fmaf(cam.M[4], dV[q].y, cam.M[7] * dV[q].z));
        out[3 * q + 2] = fmaf(cam.M[2], dV[q].x, fmaf(cam.M[5], dV[q].y, cam.M[8] * dV[q].z));
    }
}

}  // namespace

namespace {
RasterView frag_view(const FragArgs& a)
{
    return RasterView{a.map, a.W, a.H, a.tiles, a.tiles_x, a.rec, a.T, nullptr, nullptr, 0u, nullptr, nullptr, nullptr};
}
}  // namespace

vsr_status launch_frag_count(const FragArgs& a, const WalkWork& work, uint32_t* tile_pairs, cudaStream_t st)
{
    return launch_walk<FragCountStep>(frag_view(a), a, a.wi, a.geom, work, tile_pairs, a.status, st, false);
}

vsr_status launch_frag_fill(const FragArgs& a, cudaStream_t st)
{
    VSR_CUDA_TRY(launch_next(frag_fill_kernel, a.tiles_x * ((a.H + TILE - 1) / TILE), RT, st, a));
    return VSR_OK;
}

vsr_status launch_frag_fill_walk(const FragArgs& a, const WalkWork& work, cudaStream_t st)
{
    return launch_walk<FragFillStep>(frag_view(a), a, a.wi, a.geom, work, nullptr, a.status, st, false);
}

vsr_status launch_frag_backward(const FragArgs& a, const uint32_t* id, const float* dimage, const float* dcov,
                                const float* ddepth, float4* grad, float4* dmap, cudaStream_t st)
{
    BackView v{a.map, a.W, a.H, a.rec, a.T, a.colors, a.span, a.frags, id, dimage, dcov, ddepth, grad, dmap};
    dim3 grid((a.W + TILE - 1) / TILE, (a.H + TILE - 1) / TILE);
    VSR_CUDA_TRY(launch_next(frag_backward_kernel, grid, TILE_PIX, st, v));
    return VSR_OK;
}

vsr_status launch_setup_backward(const float* tris, int T, const float cam[12], const float4* rec, float4* grad,
                                 float* dtris, float* dcolors, cudaStream_t st)
{
    if (T == 0) return VSR_OK;
    CamF c;
    for (int q = 0; q < 3; ++q) c.O[q] = cam[q];
    for (int q = 0; q < 9; ++q) c.M[q] = cam[3 + q];
    VSR_CUDA_TRY(launch_next(setup_backward_kernel, (T + 127) / 128, 128, st, tris, T, c, rec, grad, dtris, dcolors));
    return VSR_OK;
}
