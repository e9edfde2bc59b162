// raster_walk.cuh -- the raster that needs no stored bins (see walk.cuh for
// the candidates of a tile), for any pixel step.
#pragma once

#include <algorithm>

#include "tile.cuh"
#include "walk.cuh"

namespace {

// Binning and raster in one launch: every tile's CTA walks its candidates
// (walk.cuh) WALK_BLOCK at a time, lists the hits in shared memory and
// rasterizes them, so the bins are never stored and no pass over the tiles
// runs before; the walk's latency is hidden by the other CTAs' evaluation.
// 1920x1080, 220k triangles: 123.5 us, against 45 us for a tile-major binning
// in three launches, 3 us for the work items and 103 us for this evaluation
// over stored bins.  Bound by instruction issue (63 % of the cycles, 8 CTAs of
// 64 registers per SM): about half of the 94 M warp instructions are the
// evaluation, the rest staging, culls, the walk and the prologue.
//
// A tile with many candidates is processed by several CTAs that merge in an
// accumulator slot (merge_slot): the tile's own CTA takes a free slot and
// publishes the tile there, the CTAs past the tiles (helpers) look for such
// tiles, and each block of candidates goes to whoever adds 1 to the slot's
// claim word next, (tile << 32) | blocks claimed.  An owner without a slot
// works alone, a helper that finds nothing ends, and the part that finishes
// the last block writes the tile and frees the slot.  A claim names its tile,
// so one made on a slot that has changed hands is still a claim of the slot's
// present tile; a claim past the tile's last block is no block.  While a part
// holds unmerged blocks its slot cannot be freed.  Nobody waits for another,
// but that helpers which may start before the tiles have been published
// (`early`: fewer tiles than resident CTAs, or tiles that are skipped) look
// until every tile has got that far, 100 us at most: 480 x 480 pixels, 5000
// triangles 31 us a frame against 51 with 10 us of looks each.
struct WalkSlots {
    SplitAcc split;             // accumulators
    unsigned long long* claim;  // per slot: (tile << 32) | blocks claimed
    uint32_t* nblk;             // per slot: blocks of its tile; 0 free, ~0 being set up
    uint32_t* hits;             // per slot: hits of the parts merged so far
    uint32_t* hint;             // owners so far: where the next one looks first, times WALK_SLOT_STEP
    uint32_t* active;           // published tiles
    uint32_t* begun;            // tiles published or known not to be (zero between launches)
    uint32_t* ended;            // CTAs that have ended (zero between launches)
    uint32_t n;                 // slots that this launch uses: as many as it has tiles, WALK_SLOTS at most
};

// What a CTA knows of its tile, in shared memory: uniform, and needed only
// between the evaluations, whose loop has no registers to spare.
struct WalkTile {
    Cone cone;
    uint32_t nblk, next;  // blocks of the tile, this CTA's next one
    uint32_t block;       // candidates of a block
    uint32_t units, hits;  // blocks done and hits found by this CTA
    int tile, slot;        // slot: -1 unless the tile is shared
    uint32_t n;            // hits of the current block
};

// What a step's evaluation may want besides the staged triangle and the pixels.
template <class In>
struct WalkCtx {
    const RasterView& view;
    const In& in;
    const WalkSlots& slots;
    const WalkTile& wt;
    const uint32_t* ids;  // the current block's hits
    Stage& stage;  // a finish may use its memory, after a barrier: other warps may still evaluate
};

// The n staged triangles of a chunk at the warp's pixels: a lane-parallel cull
// of 32 triangles at a time against the warp's cone, then the survivors one by
// one.
template <class Step>
__device__ __forceinline__ void walk_eval(const WalkCtx<typename Step::In>& cx, const Stage& st, int n,
                                          const typename Step::Cones& wc, typename Step::Pix& q)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int gbase = 0; gbase < n; gbase += 32) {
        bool keep = false;
        const int jj = gbase + lane;
        if (jj < n && __float_as_uint(st.s6[jj].w) != STAGE_EMPTY) keep = Step::cull(st, jj, wc, warp);
        unsigned mask = __ballot_sync(0xffffffffu, keep);
        while (mask) {
            const int k = 31 - __clz(mask);  // any order: from the top, one instruction less than from the bottom
            mask ^= 1u << k;
            Step::eval(cx, st, gbase + k, q);
        }
        Step::group(cx, gbase / 32, q);
    }
}

// Step: how pixels are loaded, culled against, evaluated and written (the
// global step of raster.cu, the per-fragment step of pstep.cu, the fragment
// lists of grad.cu).
// block: candidates of a block where one CTA has the tile; share_from: tiles of
// more candidates are shared, in blocks of share_block.
// SHARE: the launch has helpers (no tile of one without them has enough
// candidates to be shared, and a small frame waits for every line of code that
// its kernel has to fetch).
template <class Step, bool ROWS, bool SHARE>
__global__ void __launch_bounds__(RT, Step::CTAS) raster_walk_kernel(RasterView view, typename Step::In in, WalkIndex wi,
                                                                     const float4* geom, int ntiles,
                                                                     uint32_t block, uint32_t share_from,
                                                                     uint32_t share_block, bool early, WalkSlots slots,
                                                                     uint32_t* __restrict__ tile_pairs,
                                                                     int* __restrict__ status)
{
    grid_wait();
    grid_go();
    __shared__ Stage st;
    __shared__ WalkShared ws;
    __shared__ typename Step::Cones wc;
    __shared__ WalkTile wt;
    __shared__ uint32_t s_ids[WALK_BLOCK];
    static_assert(RT == WALK_THREADS, "the walk's CTA");
    const bool helper = SHARE && blockIdx.x >= (uint32_t)ntiles;
    int looks = early ? 400 : 0;
    // a tile is past its publication
    auto begun = [&] {
        if (SHARE && early) {
            __threadfence();
            atomicAdd(slots.begun, 1u);
        }
    };
    const bool skip = !helper && Step::skip(in, (int)blockIdx.x);
    if (skip && threadIdx.x == 0) begun();
    const WalkCtx<typename Step::In> cx{view, in, slots, wt, s_ids, st};
    while (!skip) {
        typename Step::Pix q;
        bool warp_active;
        {
            int tile = (int)blockIdx.x, slot = -1;
            uint32_t first = 0u;
            if (helper) {
                // a published tile with blocks left: the lowest such slot from
                // a start of this CTA's own
                __syncthreads();
                if (threadIdx.x == 0) {
                    for (; looks > 0 && !*(volatile uint32_t*)slots.active &&
                           *(volatile uint32_t*)slots.begun < (uint32_t)ntiles;
                         --looks)
                        __nanosleep(250);
                    __threadfence();
                    wt.slot = *(volatile uint32_t*)slots.active ? (int)slots.n : -1;
                }
                __syncthreads();
                if (wt.slot < 0) break;
                // (read from shared memory: as an argument it would be held in a
                // register through the evaluation)
                const int ns = wt.slot, from = (int)((blockIdx.x * 37u) % (uint32_t)ns);
                __syncthreads();
                int mine = ns;
                for (int i = threadIdx.x; i < ns && mine == ns; i += RT) {
                    const int c = from + i < ns ? from + i : from + i - ns;
                    const uint32_t nb = *(volatile uint32_t*)&slots.nblk[c];
                    if (nb != 0u && nb != 0xffffffffu &&
                        (uint32_t)*(volatile unsigned long long*)&slots.claim[c] < nb)
                        mine = i;
                }
                if (mine < ns) atomicMin(&wt.slot, mine);
                __syncthreads();
                slot = wt.slot;
                if (slot == ns) break;
                slot = from + slot < ns ? from + slot : from + slot - ns;
                if (threadIdx.x == 0) {
                    const unsigned long long c = atomicAdd(&slots.claim[slot], 1ull);
                    wt.tile = (int)(c >> 32);
                    wt.next = (uint32_t)c;
                }
                __syncthreads();
                tile = wt.tile;
                first = wt.next;
                if (tile >= ntiles) break;
            }
            const float4 axis = view.tiles[tile].c0;
            typename Step::Raw g;
            Step::load(view, in, TilePos(tile, view.tiles_x), g);  // in flight while the first warp finds the ranges
            if (threadIdx.x == RT - 1) wt.cone = view.tiles[tile];
            if (threadIdx.x < 32) walk_ranges(wi, view.T, geom[tile], axis.y, ws);
            if (threadIdx.x == 0) {
                const bool crowded = SHARE && ws.total > share_from;
                const uint32_t parts = (ws.total + share_block - 1) / share_block;
                if (crowded && !helper) {
                    const uint32_t from = atomicAdd(slots.hint, 1u) * WALK_SLOT_STEP;
                    for (uint32_t i = 0; i < 8u && slot < 0; ++i) {
                        const uint32_t c = (from + i) % slots.n;
                        if (atomicCAS(&slots.nblk[c], 0u, 0xffffffffu) == 0u) {
                            atomicExch(&slots.claim[c], (unsigned long long)(uint32_t)tile << 32 | 1ull);
                            __threadfence();
                            atomicExch(&slots.nblk[c], parts);
                            atomicAdd(slots.active, 1u);
                            slot = (int)c;
                        }
                    }
                }
                wt.tile = tile;
                wt.slot = slot;
                const bool shared = SHARE && (helper || slot >= 0);
                wt.block = shared ? share_block : block;
                wt.nblk = shared ? parts : (ws.total + block - 1) / block;
                wt.next = first;
                wt.units = wt.hits = wt.n = 0u;
                if (!helper) begun();
            }
            warp_active = Step::start(g, axis, q, wc);
            __syncthreads();
            if (helper && first >= wt.nblk) continue;  // finished meanwhile
        }
        while (wt.next < wt.nblk) {
            {
                Walk w;
                w.init(wi, wt.cone, ws);
                const uint32_t e0 = wt.next * wt.block;
                walk_hits(w, wi, view.rec, view.T, ws, e0, min(ws.total, e0 + wt.block), s_ids, &wt.n);
            }
            __syncthreads();
            for (uint32_t base = 0; base < wt.n; base += CHUNK) {
                const int nc = (int)min((uint32_t)CHUNK, wt.n - base);
                Step::clamp(q);
                if (base) __syncthreads();
                if ((int)threadIdx.x < nc)
                    stage_checked(view.rec, view.T, s_ids[base + threadIdx.x], wt.cone.c0, st, threadIdx.x, status);
                __syncthreads();
                if (warp_active) walk_eval<Step>(cx, st, nc, wc, q);
            }
            // the only block of a tile that is not shared (almost every tile):
            // no one waits for the others' evaluation
            if (wt.nblk == 1u && (!SHARE || wt.slot < 0)) break;
            __syncthreads();
            if (threadIdx.x == 0) {
                wt.hits += wt.n;
                wt.n = 0u;
                ++wt.units;
                wt.next = SHARE && wt.slot >= 0 ? (uint32_t)atomicAdd(&slots.claim[wt.slot], 1ull) : wt.next + 1u;
            }
            __syncthreads();
        }
#pragma unroll
        for (int p = 0; p < PPT; ++p) q.acc[p] = Step::final_acc(q, p);
        const int tile = wt.tile, slot = wt.slot;
        const TilePos tp(tile, view.tiles_x);
        uint32_t hits = wt.hits + wt.n;
        bool last = true;
        if (SHARE && slot >= 0) {
            if (threadIdx.x == 0 && hits) atomicAdd(&slots.hits[slot], hits);
            last = merge_slot<Step::SATURATES>(slots.split, slot, tp, q, wt.units, wt.nblk);
            if (last) {
                __threadfence();
                __syncthreads();
                if (threadIdx.x == 0) {
                    hits = atomicExch(&slots.hits[slot], 0u);
                    __threadfence();
                    atomicSub(slots.active, 1u);
                    atomicExch(&slots.nblk[slot], 0u);  // free
                }
            }
        }
        if (last) {
            if (tile_pairs && threadIdx.x == 0) tile_pairs[tile] = hits;
            Step::template finish<ROWS>(cx, tp, q, status);
        }
        if (!helper) break;
    }
    if (SHARE && early && threadIdx.x == 0) {
        __threadfence();
        if (atomicAdd(slots.ended, 1u) == gridDim.x - 1) {
            atomicExch(slots.begun, 0u);
            atomicExch(slots.ended, 0u);
        }
    }
}

// grid and arguments of a walking raster over `work`'s slots
template <class Step>
inline vsr_status launch_walk(const RasterView& view, const typename Step::In& in, const WalkIndex& wi,
                              const float4* geom, const WalkWork& work, uint32_t* tile_pairs, int* status,
                              cudaStream_t st, bool host_out)
{
    const int ntiles = view.tiles_x * ((view.H + TILE - 1) / TILE);
    if (ntiles == 0) return VSR_OK;
    const int sms = sm_count();
    if (sms < 0) return VSR_ERR_CUDA;
    const size_t pix = (size_t)TILE_PIX * WALK_SLOTS;
    WalkSlots sl;
    sl.split.acc = (unsigned long long*)work.mem;
    sl.split.key = sl.split.acc + pix;
    sl.claim = sl.split.key + pix;
    sl.split.done = (uint32_t*)(sl.claim + WALK_SLOTS);
    sl.nblk = sl.split.done + WALK_SLOTS;
    sl.hits = sl.nblk + WALK_SLOTS;
    sl.hint = sl.hits + WALK_SLOTS;
    sl.n = (uint32_t)std::min(ntiles, WALK_SLOTS);
    sl.active = sl.hint + 1;
    sl.begun = sl.hint + 2;
    sl.ended = sl.hint + 3;
    // Helpers only where a tile can have enough candidates.  Pictures of fewer
    // tiles than CTAs are resident: small blocks, a tile shared from its third
    // on (200k triangles at 256x256: 142 us; in blocks of 512 159 us, of 1024
    // 193 us), but one block without a grid (900 triangles at 256x256: 19 us,
    // shared in blocks of 256 41 us).  Larger pictures: large blocks, but a tile
    // of more than one is shared, in small ones, so that an object in few tiles
    // is not left to few CTAs.  1920x1080, a raster shared so, shared from the
    // fourth large block on, and over bins stored before it: 200k triangles in
    // 0.06 rad 240, 302, 297 us; 100k in 0.02 rad 151, 251, 222; in an even
    // cloud under a 340 degree lens 300k 205, 361, 246, 1M 419, 452, 454; of
    // 200k small ones 121.5 both, 140 stored.  Where an even cloud already gives
    // its tiles that many (over 128 triangles a tile), from the third large block
    // on: 1M at 1024x1024 from inside 231 us from the second, 226 from the third
    // or the fourth.  A step may share later (FEW_FROM, SHARE_FROM).
    const int wave = sms * Step::CTAS;
    const bool few = ntiles < wave;
    static_assert(GRID_DIRECT <= WALK_BLOCK && Step::FEW_BLOCK <= WALK_BLOCK, "one block, and its hits");
    const int block = few && !wi.direct ? Step::FEW_BLOCK : WALK_BLOCK;
    const int share = few ? Step::FEW_FROM : std::max(Step::SHARE_FROM, view.T / 128 > ntiles ? 2 : 1);
    const int share_from = share * block;
    const int helpers = view.T > share_from ? wave : 0;
    auto kern = helpers ? raster_walk_kernel<Step, false, true> : raster_walk_kernel<Step, false, false>;
    if constexpr (Step::HOST_OUT) {
        if (host_out) kern = helpers ? raster_walk_kernel<Step, true, true> : raster_walk_kernel<Step, true, false>;
    }
    VSR_CUDA_TRY(launch_next(kern, ntiles + helpers, RT, st, view, in, wi, geom, ntiles, (uint32_t)block,
                             (uint32_t)share_from, (uint32_t)Step::FEW_BLOCK, helpers && (few || Step::SKIPS), sl,
                             tile_pairs, status));
    return VSR_OK;
}

}  // namespace
