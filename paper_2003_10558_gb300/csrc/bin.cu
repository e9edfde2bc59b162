// bin.cu -- the triangle-major binner of the fixed-array path
// (vsr_raster_noalloc) and the tile index it searches; scans.
//
// A fragment of triangle t at pixel direction G needs G inside the miter
// cap enlarged by the ramp half-width (the gbpxstep test of the miter plane,
// Sec. 1.1.1 / 1.1.2): G.S-hat - cos rho > -h sin rho, h = 1/(2 delta).  The
// binner keeps (tile, t) when that enlarged cap can reach the tile's view
// cone.  The paper's analogue is the low-resolution region mask widened by
// fwidth/2 (getPolygonRegion).
//
// Every triangle visits the cells of the map's tile index within beta +
// alpha_small_max of its cap centre (a few dozen cone tests whatever the map's
// size; no tile is found twice): count (atomic per-tile counters) -> exclusive
// scan -> fill (atomic per-tile cursors).  It needs no memory but the bins and
// one word per tile.  The scenes' own rasters walk the triangle grid instead
// (walk.cuh).
#include <math.h>
#include <stddef.h>

#include <algorithm>
#include <atomic>

#include "vsr_internal.cuh"

namespace {

constexpr float PI_F = IDX_PI;

__device__ __forceinline__ float hist_upper(int b) { return exp2f((float)(b + 1) / 3.0f - 17.0f); }

// ---- tile index -------------------------------------------------------------
//
// Built from the per-tile geometry the map kernels write (TileIndex::geom:
// half-angle, axis latitude / longitude, ramp half-width) by one CTA
// (idx_fused_kernel, maps of up to IDX_FUSED_TILES tiles): the histogram of
// half-angles, the grid plan (a 64-bin walk), the per-cell counts, their
// exclusive scan and the cell-sorted copies of the small tiles' cones.

// the grid plan: cell size from the 99th percentile of the half-angles
__device__ void index_plan(const TileIndexHdr* hdr, TileIndexHdr& h)
{
    const unsigned nvalid = hdr->n_valid;
    const unsigned target = (unsigned)ceilf(0.99f * (float)nvalid);
    unsigned run = 0;
    int b = 0;
    for (; b < IDX_HIST; ++b) {
        run += hdr->hist[b];
        if (run >= target) break;
    }
    const float cut = hist_upper(min(b, IDX_HIST - 1));
    const float cell = fminf(PI_F / 8.0f, fmaxf(PI_F / IDX_NLAT_MAX, cut));
    const int nlat = min(IDX_NLAT_MAX, (int)ceilf(PI_F / cell));
    h.nlat = nlat;
    h.nlon = 2 * nlat;
    h.ncell = 2 * nlat * nlat;
    h.cell = PI_F / nlat;
    h.alpha_cut = cut;
}

// The tile loops of the one-CTA index kernels take IDX_BATCH tiles per
// thread at a time and issue each step for all of them before the next
// (geometry loads, then slots, then cone loads, then stores), so their
// memory latencies overlap instead of adding up tile after tile.
constexpr int IDX_BATCH = 4;

__device__ __forceinline__ void load_geom_batch(const float4* __restrict__ geom, int ntiles, int base, int stride,
                                                float4 (&g)[IDX_BATCH])
{
#pragma unroll
    for (int u = 0; u < IDX_BATCH; ++u) {
        const int i = base + u * stride;
        g[u] = i < ntiles ? geom[i] : make_float4(0.0f, 0.0f, 0.0f, -1.0f);
    }
}

// Exclusive scan of n counts in shared memory, in place, by a CTA of
// NT threads (all of which call it; ends with a barrier); returns the total
// to every thread.  Warp w owns a contiguous segment of cells and walks it 32
// cells at a time, lane l on cell 32 k + l of the step (no bank conflicts),
// with a shuffle scan per step.
template <int NT>
__device__ uint32_t block_scan_smem(uint32_t* s, int n, uint32_t* s_wsum /* NT / 32 words */)
{
    constexpr int NW = NT / 32;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int seg = ((n + NW - 1) / NW + 31) & ~31;
    const int b0 = min(n, warp * seg), b1 = min(n, b0 + seg);
    uint32_t tot = 0;
    for (int c = b0 + lane; c < b1; c += 32) tot += s[c];
    for (int o = 16; o; o >>= 1) tot += __shfl_xor_sync(0xffffffffu, tot, o);
    if (lane == 0) s_wsum[warp] = tot;
    __syncthreads();
    if (warp == 0) {
        uint32_t w = lane < NW ? s_wsum[lane] : 0u;
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, w, o);
            if (lane >= o) w += y;
        }
        if (lane < NW) s_wsum[lane] = w;  // inclusive
    }
    __syncthreads();
    uint32_t carry = warp > 0 ? s_wsum[warp - 1] : 0u;
    const uint32_t total = s_wsum[NW - 1];
    for (int c0 = b0; c0 < b1; c0 += 32) {
        const int c = c0 + lane;
        const uint32_t v = c < b1 ? s[c] : 0u;
        uint32_t x = v;
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += y;
        }
        if (c < b1) s[c] = carry + x - v;
        carry += __shfl_sync(0xffffffffu, x, 31);
    }
    __syncthreads();
    return total;
}

// The whole index in one CTA, for maps of at most IDX_FUSED_TILES tiles:
// the histogram, the per-cell counts and their scan in shared memory
// (IDX_CELLS_MAX counters), steps closed by barriers, and the header written
// once at the end.
constexpr int IDX_FUSED_THREADS = 1024;
constexpr int IDX_FUSED_TILES = 32768;
static_assert(IDX_CELLS_MAX <= 65535, "home cells are kept as 16-bit indices");
constexpr size_t IDX_FUSED_SMEM = sizeof(uint32_t) * IDX_CELLS_MAX + sizeof(uint16_t) * IDX_FUSED_TILES;

__global__ void __launch_bounds__(IDX_FUSED_THREADS) idx_fused_kernel(const Cone* __restrict__ tiles,
                                                                       const float4* __restrict__ geom, int ntiles,
                                                                       TileIndexHdr* __restrict__ hdr,
                                                                       uint32_t* __restrict__ cell_start,
                                                                       Cone* __restrict__ sorted,
                                                                       Cone* __restrict__ big)
{
    extern __shared__ uint32_t s_cell[];  // per-cell counts, then running slots
    // each small tile's home cell (0xffff: big or empty), from step 3 to step 5
    uint16_t* s_tcell = reinterpret_cast<uint16_t*>(s_cell + IDX_CELLS_MAX);
    __shared__ TileIndexHdr s_h;
    __shared__ uint32_t s_wsum[IDX_FUSED_THREADS / 32];
    const int tid = threadIdx.x, lane = tid & 31;
    if (tid == 0) s_h = TileIndexHdr{};
    __syncthreads();
    // 1. histogram of half-angles (one add per group of equal bins in a
    // warp), valid tiles, widest ramp (one atomic per warp)
    uint32_t nv = 0u, hm = 0u, va = 0u;
    for (int base = 0; base < ntiles; base += IDX_FUSED_THREADS * IDX_BATCH) {
        float4 gb[IDX_BATCH];
        load_geom_batch(geom, ntiles, base + tid, IDX_FUSED_THREADS, gb);
#pragma unroll
        for (int u = 0; u < IDX_BATCH; ++u) {
            const float4 g = gb[u];
            const bool ok = g.w >= 0.0f;
            const int bin = ok ? hist_bin(g.x) : -1;
            const unsigned peers = __match_any_sync(0xffffffffu, bin);
            if (ok && lane == __ffs(peers) - 1) atomicAdd(&s_h.hist[bin], (unsigned)__popc(peers));
            nv += ok;
            hm = max(hm, ok ? __float_as_uint(g.w) : 0u);  // non-negative floats order as their bits
            if (ok) va = max(va, view_angle_bits(tiles[base + tid + u * IDX_FUSED_THREADS], g.x));
        }
    }
    for (int o = 16; o; o >>= 1) {
        nv += __shfl_xor_sync(0xffffffffu, nv, o);
        hm = max(hm, __shfl_xor_sync(0xffffffffu, hm, o));
        va = max(va, __shfl_xor_sync(0xffffffffu, va, o));
    }
    if (lane == 0 && nv) {
        atomicAdd(&s_h.n_valid, nv);
        atomicMax(&s_h.h_max, hm);
        atomicMax(&s_h.view_angle, va);
    }
    __syncthreads();
    // 2. the grid plan
    if (tid == 0) index_plan(&s_h, s_h);
    __syncthreads();
    const int ncell = s_h.ncell;
    for (int c = tid; c < ncell; c += IDX_FUSED_THREADS) s_cell[c] = 0u;
    __syncthreads();
    // 3. per-cell counts; big tiles to their own list
    uint32_t am = 0u;
    for (int base = tid; base < ntiles; base += IDX_FUSED_THREADS * IDX_BATCH) {
        float4 gb[IDX_BATCH];
        load_geom_batch(geom, ntiles, base, IDX_FUSED_THREADS, gb);
#pragma unroll
        for (int u = 0; u < IDX_BATCH; ++u) {
            const float4 g = gb[u];
            const int i = base + u * IDX_FUSED_THREADS;
            if (i >= ntiles) continue;
            uint16_t home = 0xffffu;
            if (g.w >= 0.0f) {
                if (g.x > s_h.alpha_cut) {
                    big[atomicAdd(&s_h.n_big, 1u)] = index_entry(tiles[i], i);
                } else {
                    const int c = home_cell_geom(g, s_h);
                    atomicAdd(&s_cell[c], 1u);
                    home = (uint16_t)c;
                    am = max(am, __float_as_uint(g.x));
                }
            }
            s_tcell[i] = home;
        }
    }
    for (int o = 16; o; o >>= 1) am = max(am, __shfl_xor_sync(0xffffffffu, am, o));
    if (lane == 0 && am) atomicMax(&s_h.alpha_small_max, am);
    __syncthreads();
    // 4. exclusive scan of the counts (in place: they become running slots),
    // the starts out (coalesced)
    const uint32_t total = block_scan_smem<IDX_FUSED_THREADS>(s_cell, ncell, s_wsum);
    for (int c = tid; c < ncell; c += IDX_FUSED_THREADS) cell_start[c] = s_cell[c];
    if (tid == 0) cell_start[ncell] = total;
    // 5. cell-sorted copies of the small tiles (slots, then cone loads, then stores)
    for (int base = tid; base < ntiles; base += IDX_FUSED_THREADS * IDX_BATCH) {
        uint32_t slot[IDX_BATCH];
#pragma unroll
        for (int u = 0; u < IDX_BATCH; ++u) {
            const int i = base + u * IDX_FUSED_THREADS;
            const uint16_t c = i < ntiles ? s_tcell[i] : (uint16_t)0xffffu;
            slot[u] = c != 0xffffu ? atomicAdd(&s_cell[c], 1u) : 0xffffffffu;
        }
        Cone cn[IDX_BATCH];
#pragma unroll
        for (int u = 0; u < IDX_BATCH; ++u)
            if (slot[u] < (uint32_t)ntiles) cn[u] = tiles[base + u * IDX_FUSED_THREADS];
#pragma unroll
        for (int u = 0; u < IDX_BATCH; ++u)
            if (slot[u] < (uint32_t)ntiles) sorted[slot[u]] = index_entry(cn[u], base + u * IDX_FUSED_THREADS);
    }
    if (tid == 0) *hdr = s_h;
}

// ---- per-triangle binning ---------------------------------------------------
//
// The candidate tiles of a triangle are the cones of its search window: the
// index rows r0..r1 around the cap centre, each a contiguous range of the
// cell-sorted cones (two ranges where the window wraps across longitude
// +-pi), plus the big tiles.  One warp bins 32 triangles.  Phase 1, one lane
// per triangle: the cap enlarged by the widest ramp and the window.  Phase
// 2: the windows' (triangle, row range) pairs -- the big list cut into
// chunks of BIN_BIG_CHUNK cones counts as further pairs -- are concatenated
// in lane order and handed out one pair per lane per round, so the
// dependent loads of the search run on all lanes at once instead of one
// lane walking its whole window.
//
// count: counts[tile] += 1 per hit (no value returned, so nothing waits);
// fill: the same search, each hit taking slot counts[tile] - 1 by atomic
// decrement and writing ids[offsets[tile] + slot] = triangle.  The counts
// return to zero; the order of ids inside a bin is not fixed and the raster
// kernels' results do not depend on it.

constexpr int BIN_BIG_CHUNK = 16;
// cones per step of the search for grids beyond one resident wave
// The longest cone range of a warp round, in steps of the flattened walk,
// above which the round walks its cones flattened across the warp.
#ifndef VSR_BIN_FLAT_RATIO
#define VSR_BIN_FLAT_RATIO 2
#endif

// triangles per warp of the large-grid shape: 16 (measured on the 1080p
// frame's 220k triangles: bin stage 65.9 us against 73.8 us at 32 and 67.7 us
// at 8) -- the grid is then two resident waves, and each warp's chain of
// dependent loads (window rows, then cones) half as long
#ifndef VSR_BIN_TPW_LARGE
#define VSR_BIN_TPW_LARGE 16
#endif

#ifndef VSR_BIN_CB_LARGE
#define VSR_BIN_CB_LARGE 1
#endif
// FILL: false = count + record, true = fill by searching again.
// CB: cones each lane fetches per step.  The search is bound by load latency:
// a grid larger than one resident wave hides it with warps (CB = 1: 40
// registers, 12 CTAs per SM), a smaller one with loads in flight per lane
// (CB = 4, 7 CTAs per SM).
// TPW: triangles per warp (lanes 0 .. TPW-1 run phase 1; phase 2 spreads
// their pairs over all 32 lanes).  8 for small scenes, so that they still
// give the GPU enough warps to hide the search's latency.
template <bool FILL, int CB, int TPW>
__global__ void __launch_bounds__(128, CB == 1 ? 12 : (CB == 2 ? 10 : 1)) bin_kernel(BinView v, int T,
                                                                                   uint32_t* __restrict__ ids,
                                                                     uint32_t cap, int* status)
{
    const unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int t = (int)(blockIdx.x * 4 + warp) * TPW + lane;
    const size_t TT = (size_t)T;
    // The index header, with every count that becomes an index clamped to
    // the arrays it indexes (identity for an index built by launch_tile_index),
    // so that no index content can make this kernel read or write out of
    // bounds.
    TileIndexHdr h;
    h.nlat = min(max(v.hdr->nlat, 1), IDX_NLAT_MAX);
    h.nlon = 2 * h.nlat;
    h.cell = v.hdr->cell;
    const int nlat = h.nlat, nlon = h.nlon;
    const float cell = h.cell;
    const float amax = __uint_as_float(v.hdr->alpha_small_max), hmax = __uint_as_float(v.hdr->h_max);
    // the map's field of view: a cone about +z of half-angle view_angle
    // holding every tile cone; a cap that misses it misses every tile (a
    // view angle of pi or more holds the whole sphere: no cap misses it)
    const float vang = __uint_as_float(v.hdr->view_angle);
    const bool fov = vang < PI_F;
    float vcos, vsin;
    sincosf(fminf(vang, PI_F), &vsin, &vcos);
    const uint32_t nbig = min(v.hdr->n_big, v.ntiles);
    const int bigpairs = (int)((nbig + BIN_BIG_CHUNK - 1) / BIN_BIG_CHUNK);

    // phase 1: this lane's triangle
    float sx = 0.0f, sy = 0.0f, sz = 1.0f, cb = 1.0f, sb = 0.0f;
    int r0 = 0, c0i = 0, ncol = 0, segs = 1, rowpairs = 0, npairs = 0;
    if (lane < TPW && t < T) {
        const float4 q0 = v.rec[rec_at(TT, t, RF_CAP)];
        const float4 q1 = v.rec[rec_at(TT, t, RF_CAP2)];
        if (q1.w != 0.0f) {
            sx = q0.x;
            sy = q0.y;
            sz = q0.z;
            // the cap enlarged once by the map's widest ramp (>= every tile's
            // own): cos / sin of its radius beta, so each tile test is a few FMAs
            cb = fmaxf(-1.0f, fminf(1.0f, q0.w - hmax * q1.x));
            sb = sqrtf(fmaxf(0.0f, 1.0f - cb * cb));
            // outside the field of view: no window, no pairs.  The cap of
            // radius beta reaches the view cone iff angle(S, +z) <= beta +
            // view angle, i.e. S.z >= cos(beta + view angle) while the sum
            // is below pi; with both angles in [0, pi) the sum is below pi
            // exactly when its sine is positive
            const float cbv = fmaf(cb, vcos, -sb * vsin), sbv = fmaf(sb, vcos, cb * vsin);
            const bool outside = fov && sbv > 0.0f && sz < cbv - 2e-6f;
            // search radius: enlarged cap + largest small tile
            const float gamma = outside ? PI_F : acosf(cb) + amax + 1e-4f;
            int r1 = nlat - 1;
            ncol = nlon;
            if (gamma < PI_F) {
                const float lat = asinf(fmaxf(-1.0f, fminf(1.0f, sy)));
                const float lon = atan2f(sx, sz);
                r0 = cell_row(lat - gamma, h);
                r1 = cell_row(lat + gamma, h);
                if (fabsf(lat) + gamma < 0.5f * PI_F - 1e-3f) {
                    // longitude half-width of a cap that holds no pole
                    const float dl = asinf(fminf(1.0f, sinf(gamma) / cosf(lat))) + 1e-4f;
                    c0i = (int)floorf((lon - dl + PI_F) / cell);
                    const int c1i = (int)floorf((lon + dl + PI_F) / cell);
                    ncol = max(1, min(nlon, c1i - c0i + 1));
                    c0i %= nlon;
                    if (c0i < 0) c0i += nlon;
                }
            }
            segs = c0i + ncol <= nlon ? 1 : 2;
            rowpairs = (r1 - r0 + 1) * segs;
            npairs = outside ? 0 : rowpairs + bigpairs;
        }
    }
    int incl = npairs;
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(FULL, incl, o);
        if (lane >= o) incl += y;
    }
    const int total = __shfl_sync(FULL, incl, 31);
    const int off = incl - npairs;

    // phase 2: one (triangle, range) pair per lane and round
    for (int base = 0; base < total; base += 32) {
        const int p = base + lane;
        int q = 0;  // the last lane whose pairs start at or before p
        for (int st = 16; st > 0; st >>= 1) {
            const int oc = __shfl_sync(FULL, off, q + st);
            if (oc <= p) q += st;
        }
        const int u = p - __shfl_sync(FULL, off, q);
        const float tx = __shfl_sync(FULL, sx, q), ty = __shfl_sync(FULL, sy, q), tz = __shfl_sync(FULL, sz, q);
        const float tcb = __shfl_sync(FULL, cb, q), tsb = __shfl_sync(FULL, sb, q);
        const int tr0 = __shfl_sync(FULL, r0, q), tc0 = __shfl_sync(FULL, c0i, q);
        const int tncol = __shfl_sync(FULL, ncol, q), tsegs = __shfl_sync(FULL, segs, q);
        const int trows = __shfl_sync(FULL, rowpairs, q);
        const uint32_t tt = (uint32_t)__shfl_sync(FULL, t, q);
        uint32_t a = 0, b = 0;
        const Cone* __restrict__ list = v.sorted;
        if (p < total) {
            if (u < trows) {
                const int row = tr0 + u / tsegs, seg = u - (u / tsegs) * tsegs;
                const uint32_t* __restrict__ rs = v.cell_start + (size_t)row * nlon;
                if (tsegs == 1) {
                    a = rs[tc0];
                    b = rs[tc0 + tncol];
                } else if (seg == 0) {  // the window wraps across longitude +-pi
                    a = rs[tc0];
                    b = rs[nlon];
                } else {
                    a = rs[0];
                    b = rs[tc0 + tncol - nlon];
                }
            } else {
                a = (uint32_t)(u - trows) * BIN_BIG_CHUNK;
                b = min(nbig, a + BIN_BIG_CHUNK);
                list = v.big;
            }
            b = min(b, v.ntiles);
            a = min(a, b);
        }
        // a hit: count and record it (count pass) or take a slot and fill it
        auto hit = [&](uint32_t tile, uint32_t tri) {
            if (!FILL) {
                atomicAdd(&v.counts[tile], 1u);
            } else {
                const uint32_t pos = v.offsets[tile] + atomicSub(&v.counts[tile], 1u) - 1u;
                if (pos < cap && pos < v.offsets[tile + 1])
                    ids[pos] = tri;
                else
                    raise_status(status, VSR_ERR_BIN_OVERFLOW);
            }
        };
        // the cap / cone test: angle(S, axis) <= alpha + beta (always when
        // alpha + beta >= pi)
        auto reaches = [&](const Cone& c, float x, float y, float z, float cbt, float sbt) {
            const float cg = fmaf(x, c.c0.x, fmaf(y, c.c0.y, z * c.c0.z));
            return cbt + c.c0.w <= 2e-6f || cg >= fmaf(c.c0.w, cbt, -c.c1.x * sbt) - 2e-6f;
        };
        // Two ways through the round's cones.  Each lane walks its own range
        // -- as many steps as the longest range, the other lanes idle once
        // theirs ends -- or, where the ranges are very unequal, the cones are
        // numbered across the warp (lane l's range is [excl_l, excl_l +
        // len_l)) and every lane takes the next cone each step, finding the
        // lane whose range holds it by a search over the lanes.  The second
        // costs more per step (the search and the range's parameters by
        // shuffle), so it is taken when the longest range is over
        // VSR_BIN_FLAT_RATIO times its step count.
        const int len = (int)(b - a);
        int incl = len, lmax = len;
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(FULL, incl, o);
            if (lane >= o) incl += y;
            lmax = max(lmax, __shfl_xor_sync(FULL, lmax, o));
        }
        const int ncones = __shfl_sync(FULL, incl, 31);
        if (lmax <= VSR_BIN_FLAT_RATIO * ((ncones + 31) / 32)) {
            for (uint32_t k0 = a; k0 < b; k0 += CB) {
                Cone cs[CB];
#pragma unroll
                for (int e = 0; e < CB; ++e)
                    if (k0 + e < b) cs[e] = list[k0 + e];
#pragma unroll
                for (int e = 0; e < CB; ++e) {
                    if (k0 + e >= b) break;
                    if (!reaches(cs[e], tx, ty, tz, tcb, tsb)) continue;
                    const uint32_t tile = __float_as_uint(cs[e].c1.z);
                    if (tile < v.ntiles) hit(tile, tt);
                }
            }
        } else {
            const int excl = incl - len;
            const int rel = (int)a - excl;  // list index = cone number + rel
            const int isbig = list == v.big;
            for (int k0 = 0; k0 < ncones; k0 += 32) {
                const int idx = k0 + lane;
                int o = 0;  // the last lane whose range starts at or before cone idx
                for (int st = 16; st > 0; st >>= 1) {
                    const int e = __shfl_sync(FULL, excl, o + st);
                    if (e <= idx) o += st;
                }
                const float ox = __shfl_sync(FULL, tx, o), oy = __shfl_sync(FULL, ty, o),
                            oz = __shfl_sync(FULL, tz, o);
                const float ocb = __shfl_sync(FULL, tcb, o), osb = __shfl_sync(FULL, tsb, o);
                const uint32_t ot = (uint32_t)__shfl_sync(FULL, (int)tt, o);
                const int orel = __shfl_sync(FULL, rel, o), obig = __shfl_sync(FULL, isbig, o);
                if (idx >= ncones) continue;
                const Cone c = (obig ? v.big : v.sorted)[idx + orel];
                if (!reaches(c, ox, oy, oz, ocb, osb)) continue;
                const uint32_t tile = __float_as_uint(c.c1.z);
                if (tile < v.ntiles) hit(tile, ot);
            }
        }
    }
}

// Exclusive scan of n counts into offsets[0..n] by one CTA of 1024 threads:
// chunks of 4096 (four consecutive elements per thread), carried across
// chunks.
__global__ void __launch_bounds__(1024) scan_kernel(const uint32_t* __restrict__ counts, int n,
                                                     uint32_t* __restrict__ offsets)
{
    __shared__ uint32_t warp_sums[32];
    __shared__ uint32_t carry_s;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (tid == 0) carry_s = 0;
    __syncthreads();
    for (int base = 0; base < n; base += 4096) {
        const int b = base + 4 * tid;
        uint32_t v[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) v[q] = b + q < n ? counts[b + q] : 0u;
        const uint32_t local = v[0] + v[1] + v[2] + v[3];
        uint32_t x = local;
        for (int o = 1; o < 32; o <<= 1) {
            uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += y;
        }
        if (lane == 31) warp_sums[warp] = x;
        __syncthreads();
        if (warp == 0) {
            uint32_t s = warp_sums[lane];
            for (int o = 1; o < 32; o <<= 1) {
                uint32_t y = __shfl_up_sync(0xffffffffu, s, o);
                if (lane >= o) s += y;
            }
            warp_sums[lane] = s;
        }
        __syncthreads();
        uint32_t run = carry_s + x - local + (warp > 0 ? warp_sums[warp - 1] : 0u);
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            if (b + q < n) offsets[b + q] = run;
            run += v[q];
        }
        __syncthreads();
        if (tid == 0) carry_s += warp_sums[31];
        __syncthreads();
    }
    if (tid == 0) offsets[n] = carry_s;
}

}  // namespace

vsr_status launch_scan(const uint32_t* counts, int n, uint32_t* offsets, cudaStream_t st)
{
    scan_kernel<<<1, 1024, 0, st>>>(counts, n, offsets);
    VSR_CUDA_TRY(cudaGetLastError());
    return VSR_OK;
}

vsr_status launch_tile_index(const Cone* tiles, int ntiles, TileIndex idx, cudaStream_t st)
{
    if (ntiles < 0 || ntiles > IDX_FUSED_TILES) return VSR_ERR_INVALID_ARG;
    // the shared-memory opt-in of the kernel, once per device
    static std::atomic<uint64_t> attr_set{0};
    int dev = 0;
    VSR_CUDA_TRY(cudaGetDevice(&dev));
    const uint64_t bit = 1ull << (dev & 63);
    if (!(attr_set.load() & bit)) {
        VSR_CUDA_TRY(cudaFuncSetAttribute(idx_fused_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                          (int)IDX_FUSED_SMEM));
        attr_set.fetch_or(bit);
    }
    idx_fused_kernel<<<1, IDX_FUSED_THREADS, IDX_FUSED_SMEM, st>>>(tiles, idx.geom, ntiles, idx.hdr, idx.cell_start,
                                                                    idx.sorted, idx.big);
    VSR_CUDA_TRY(cudaGetLastError());
    return VSR_OK;
}

int sm_count()
{
    static std::atomic<int> cache[64];
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return -1;
    const int slot = dev & 63;
    int n = cache[slot].load();
    if (n > 0) return n;
    if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n <= 0) return -1;
    cache[slot].store(n);
    return n;
}

// The binner's launch shape for T triangles on `sms` SMs: 0 = one cone per
// step and VSR_BIN_TPW_LARGE triangles per warp (grids beyond one resident wave at 7 CTAs
// per SM), 1 = four cones per step, 2 = four cones and 8 triangles per warp
// (scenes whose 8-per-warp grid still fits that wave).
static int bin_shape(int T, int sms)
{
    if ((T + 127) / 128 > 7 * sms) return 0;
    if ((T + 31) / 32 <= 7 * sms) return 2;
    return 1;
}

vsr_status launch_bin_count(const float4* rec, int T, TileIndex idx, uint32_t* counts, cudaStream_t st)
{
    if (T == 0) return VSR_OK;
    const BinView v{idx.hdr, idx.cell_start, idx.sorted, idx.big, rec, counts, nullptr, idx.ntiles};
    const int sms = sm_count();
    if (sms < 0) return VSR_ERR_CUDA;
    switch (bin_shape(T, sms)) {
    case 0:
        bin_kernel<false, VSR_BIN_CB_LARGE, VSR_BIN_TPW_LARGE>
            <<<(T + 4 * VSR_BIN_TPW_LARGE - 1) / (4 * VSR_BIN_TPW_LARGE), 128, 0, st>>>(v, T, nullptr, 0, nullptr);
        break;
    case 1: bin_kernel<false, 4, 32><<<(T + 127) / 128, 128, 0, st>>>(v, T, nullptr, 0, nullptr); break;
    default: bin_kernel<false, 4, 8><<<(T + 31) / 32, 128, 0, st>>>(v, T, nullptr, 0, nullptr); break;
    }
    VSR_CUDA_TRY(cudaGetLastError());
    return VSR_OK;
}

vsr_status launch_bin_fill(const float4* rec, int T, TileIndex idx, const uint32_t* offsets, uint32_t* counts,
                           uint32_t* ids, uint32_t cap, int* status, cudaStream_t st)
{
    if (T == 0) return VSR_OK;
    const BinView v{idx.hdr, idx.cell_start, idx.sorted, idx.big, rec, counts, offsets, idx.ntiles};
    const int sms = sm_count();
    if (sms < 0) return VSR_ERR_CUDA;
    switch (bin_shape(T, sms)) {
    case 0:
        bin_kernel<true, VSR_BIN_CB_LARGE, VSR_BIN_TPW_LARGE>
            <<<(T + 4 * VSR_BIN_TPW_LARGE - 1) / (4 * VSR_BIN_TPW_LARGE), 128, 0, st>>>(v, T, ids, cap, status);
        break;
    case 1: bin_kernel<true, 4, 32><<<(T + 127) / 128, 128, 0, st>>>(v, T, ids, cap, status); break;
    default: bin_kernel<true, 4, 8><<<(T + 31) / 32, 128, 0, st>>>(v, T, ids, cap, status); break;
    }
    VSR_CUDA_TRY(cudaGetLastError());
    return VSR_OK;
}
