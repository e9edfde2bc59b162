// pstep.cu -- coverage / depth / visibility with the per-fragment pixel
// step (Sec. 1.1.1): each of the four plane distances g of the
// rasterization equation ramps over its own fwidth,
//   w = |d_i g| + |d_j g|,  d g = n . d G  (edges),  (S-hat . d G)/sin(rho)
//   (miter, whose distance carries the same 1/sin(rho)),
// with d_i G, d_j G the map's own central differences (stored with the map),
// instead of the map-wide global delta:
//   fragment iff every g > -w/2 (bpxstep),  m^f = min clamp(g/w + 1/2, 0, 1)
// Everything else -- the walk over the grid, tile-centred distances, the
// order-free merge, the visibility key -- is the coverage kernel's
// (raster_walk.cuh, tile.cuh).
//
// Issue-bound as that one: the widths of a lane's two pixels are formed in
// packed FP32x2 beside the distances, a triangle without a fragment in the
// warp ends after them, and the four ramps take one clamp (it is monotone, so
// it commutes with the minimum).  1280x720, 100k triangles, set-up included:
// 173.6 us with scalar pixels over stored bins, 130 us.
#include <type_traits>

#include "raster_walk.cuh"

namespace {

struct PstepPix {
    float2 dgx, dgy, dgz;     // G - a (tile axis) of both pixels; 0 at an invalid pixel
    float2 eg;                // |G|^2 - 1
    float2 dix, diy, diz;     // d_i G
    float2 djx, djy, djz;     // d_j G
    bool valid[PPT];
    uint32_t acc[PPT];
    unsigned long long key[PPT];
};

struct PstepCones {
    float4 c[RT / 32][2];  // as WarpCones (the widest ramp of any distance for h)
    float2 e[RT / 32];     // pstep_ramp of h
};

// |n . d_i G| + |n . d_j G| of both pixels
__device__ __forceinline__ float2 width2(const PstepPix& q, const float4& n)
{
    const float2 a = __ffma2_rn(bcast2(n.x), q.dix, __ffma2_rn(bcast2(n.y), q.diy, __fmul2_rn(bcast2(n.z), q.diz)));
    const float2 b = __ffma2_rn(bcast2(n.x), q.djx, __ffma2_rn(bcast2(n.y), q.djy, __fmul2_rn(bcast2(n.z), q.djz)));
    return make_float2(__fadd_rn(fabsf(a.x), fabsf(b.x)), __fadd_rn(fabsf(a.y), fabsf(b.y)));
}

// g / w + 1/2 with the hardware's reciprocal (w >= 1e-30: no scaling needed)
__device__ __forceinline__ float ramp(float g, float w) { return __fmaf_rn(g, rcp_fast(fmaxf(w, 1e-30f)), 0.5f); }

struct PstepStep {
    static constexpr int FEW_BLOCK = WALK_BLOCK / 4;
    static constexpr bool SATURATES = true, HOST_OUT = false, SKIPS = false;
    static constexpr int FEW_FROM = 2, SHARE_FROM = 1;
    static constexpr int CTAS = 6;  // 80 registers; 5: 135.3 us, 4: 142.7 us against 130.4 us
    using Pix = PstepPix;
    using Cones = PstepCones;
    struct In {
        const float4* deriv;  // 2 float4 per pixel: d_i G, d_j G
    };
    struct Raw {
        float4 g[PPT], di[PPT], dj[PPT];
    };
    __device__ __forceinline__ static void load(const RasterView& view, const In& in, const TilePos& tp, Raw& r)
    {
#pragma unroll
        for (int p = 0; p < PPT; ++p) {
            const int y = tp.py + 4 * p;
            r.g[p] = r.di[p] = r.dj[p] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
            if (tp.px < view.W && y < view.H) {
                const size_t o = (size_t)y * view.W + tp.px;
                r.g[p] = view.map[o];
                const F8 d = ld_f8(in.deriv + 2 * o);
                r.di[p] = d.a;
                r.dj[p] = d.b;
            }
        }
    }
    __device__ __forceinline__ static bool start(const Raw& r, const float4& axis, Pix& q, Cones& wc)
    {
        bool pv[PPT];
        float h[PPT], gx[PPT], gy[PPT], gz[PPT];
#pragma unroll
        for (int p = 0; p < PPT; ++p) {
            const float4 &a = r.di[p], &b = r.dj[p];
            pv[p] = r.g[p].w > 0.0f;
            gx[p] = r.g[p].x;
            gy[p] = r.g[p].y;
            gz[p] = r.g[p].z;
            // the widest ramp half-width of any distance at this pixel
            h[p] = pv[p] ? 0.5f * (sqrtf(fmaf(a.x, a.x, fmaf(a.y, a.y, a.z * a.z))) +
                                   sqrtf(fmaf(b.x, b.x, fmaf(b.y, b.y, b.z * b.z)))) * 1.000001f
                         : 0.0f;
            q.valid[p] = pv[p];
            q.acc[p] = 0u;
            q.key[p] = KEY_NONE;
        }
        q.dgx = make_float2(pv[0] ? gx[0] - axis.x : 0.0f, pv[1] ? gx[1] - axis.x : 0.0f);
        q.dgy = make_float2(pv[0] ? gy[0] - axis.y : 0.0f, pv[1] ? gy[1] - axis.y : 0.0f);
        q.dgz = make_float2(pv[0] ? gz[0] - axis.z : 0.0f, pv[1] ? gz[1] - axis.z : 0.0f);
        const float2 eg =
            norm2_minus_one2(make_float2(gx[0], gx[1]), make_float2(gy[0], gy[1]), make_float2(gz[0], gz[1]));
        q.eg = make_float2(pv[0] ? eg.x : 0.0f, pv[1] ? eg.y : 0.0f);
        q.dix = make_float2(r.di[0].x, r.di[1].x);
        q.diy = make_float2(r.di[0].y, r.di[1].y);
        q.diz = make_float2(r.di[0].z, r.di[1].z);
        q.djx = make_float2(r.dj[0].x, r.dj[1].x);
        q.djy = make_float2(r.dj[0].y, r.dj[1].y);
        q.djz = make_float2(r.dj[0].z, r.dj[1].z);
        float4 c0, c1;
        block_cone(gx, gy, gz, h, pv, c0, c1);
        if ((threadIdx.x & 31) == 0) {
            const int w = threadIdx.x >> 5;
            wc.c[w][0] = c0;
            wc.c[w][1] = c1;
            wc.e[w] = pstep_ramp(c1.y);
        }
        __syncwarp();
        return c1.z > 0.0f;
    }
    __device__ __forceinline__ static bool cull(const Stage& st, int j, const Cones& wc, int warp)
    {
        const float4 c0 = wc.c[warp][0], c1 = wc.c[warp][1];
        const float2 e = wc.e[warp];
        const float4 a = st.s0[j], b = st.s1[j];
        // the cap widened by the ramp (pstep_cap)
        const float2 cap = pstep_cap(1.0f - 0.5f * b.y, b.x, e);
        const bool keep = cap_hits_cone(make_float3(a.x, a.y, a.z), cap.x, fmaxf(cap.y, 0.0f),
                                        make_float3(c0.x, c0.y, c0.z), c0.w, c1.x, 0.0f);
        const float lim = -(c1.y + c1.x + (1.0f - c0.w) + 1e-6f);
        const float4 n1 = st.s2[j], n2 = st.s3[j], n3 = st.s4[j];
        return keep && fmaf(c0.x, n1.x, fmaf(c0.y, n1.y, c0.z * n1.z)) > lim &&
               fmaf(c0.x, n2.x, fmaf(c0.y, n2.y, c0.z * n2.z)) > lim &&
               fmaf(c0.x, n3.x, fmaf(c0.y, n3.y, c0.z * n3.z)) > lim;
    }
    // staged slot j at the lane's two pixels; all 32 lanes together
    __device__ __forceinline__ static void eval(const WalkCtx<In>&, const Stage& st, int j, Pix& q)
    {
        const float4 a = st.s0[j], b = st.s1[j], e = st.s6[j];
        const float4 n1 = st.s2[j], n2 = st.s3[j], n3 = st.s4[j];
        const float2 g1 = plane_distance2(q.dgx, q.dgy, q.dgz, n1);
        const float2 g2 = plane_distance2(q.dgx, q.dgy, q.dgz, n2);
        const float2 g3 = plane_distance2(q.dgx, q.dgy, q.dgz, n3);
        const float2 g4 = miter_distance2(q.dgx, q.dgy, q.dgz, e, b, q.eg);
        const float2 w1 = width2(q, n1), w2 = width2(q, n2), w3 = width2(q, n3);
        const float2 w4 = __fmul2_rn(width2(q, a), bcast2(2.0f * b.z));
        const float2 k1 = __fmul2_rn(w1, bcast2(-0.5f)), k2 = __fmul2_rn(w2, bcast2(-0.5f)),
                     k3 = __fmul2_rn(w3, bcast2(-0.5f)), k4 = __fmul2_rn(w4, bcast2(-0.5f));
        const bool frag[PPT] = {q.valid[0] && g1.x > k1.x && g2.x > k2.x && g3.x > k3.x && g4.x > k4.x,
                                q.valid[1] && g1.y > k1.y && g2.y > k2.y && g3.y > k3.y && g4.y > k4.y};
        if (!__any_sync(0xffffffffu, frag[0] || frag[1])) return;
        const float2 Dp = plane_distance2(q.dgx, q.dgy, q.dgz, st.s5[j]);
        const float D[PPT] = {Dp.x, Dp.y};
        const float g3m[PPT] = {fminf(fminf(g1.x, g2.x), g3.x), fminf(fminf(g1.y, g2.y), g3.y)};
        const float m[PPT] = {
            __saturatef(fminf(fminf(ramp(g1.x, w1.x), ramp(g2.x, w2.x)), fminf(ramp(g3.x, w3.x), ramp(g4.x, w4.x)))),
            __saturatef(fminf(fminf(ramp(g1.y, w1.y), ramp(g2.y, w2.y)), fminf(ramp(g3.y, w3.y), ramp(g4.y, w4.y))))};
        auto post = [&](auto rare_t) {
            constexpr bool RARE = decltype(rare_t)::value;
            uint32_t rq[PPT];
            bool inn[PPT];
#pragma unroll
            for (int p = 0; p < PPT; ++p) {
                const float r = RARE ? __fdividef(b.w, D[p]) : __fmul_rn(b.w, rcp_fast(D[p]));
                rq[p] = __float_as_uint(r) - 1u;
                if (frag[p] && rq[p] < DEPTH_LIM) q.acc[p] += cov_fixed(m[p]);
                inn[p] = frag[p] && g3m[p] > 0.0f;
                if (RARE && frag[p] && g3m[p] == 0.0f)
                    inn[p] = centre_inside(p ? g1.y : g1.x, p ? g2.y : g2.x, p ? g3.y : g3.x, g3m[p],
                                           __float_as_uint(a.w));
            }
            if (__any_sync(0xffffffffu, inn[0] || inn[1])) {
#pragma unroll
                for (int p = 0; p < PPT; ++p) {
                    const unsigned long long k = ((unsigned long long)rq[p] << 32) | __float_as_uint(e.w);
                    q.key[p] = inn[p] && k < q.key[p] ? k : q.key[p];
                }
            }
        };
        // an exact zero or a denormal plane distance takes the general copy
        const float tiny = fminf(fminf(fabsf(g3m[0]), fabsf(g3m[1])), fminf(fabsf(D[0]), fabsf(D[1])));
        if (__any_sync(0xffffffffu, tiny < 1.17549435e-38f))
            post(std::true_type{});
        else
            post(std::false_type{});
    }
    __device__ __forceinline__ static uint32_t final_acc(const Pix& q, int p) { return min(q.acc[p], COV_ONE); }
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

}  // namespace

vsr_status launch_raster_pstep(const RasterView& view, const float4* deriv, const WalkIndex& wi, const float4* geom,
                               const WalkWork& work, uint32_t* tile_pairs, int* status, cudaStream_t st)
{
    return launch_walk<PstepStep>(view, PstepStep::In{deriv}, wi, geom, work, tile_pairs, status, st, false);
}
