// grid.cu -- the triangle grid of a set-up (TriGrid) and binning by the walk
// over it (walk.cuh).
//
// Filing is a counting sort spread over three launches: the set-up kernel
// finds every triangle's cell (its records are in registers) and counts it
// with an atomic that returns nothing, so the set-up, at two warps per
// scheduler, never waits for one (with the ranks returned there the set-up of
// 220k triangles took 38.2 us instead of 30); grid_rows_kernel turns a row's
// counts into entry numbers -- the rows take their places in any order, one
// atomic each, so no scan runs across them -- and grid_file_kernel takes each
// triangle's place in its cell and writes the entries.
#include <algorithm>

#include "walk.cuh"

namespace {

// One CTA per row of every level, and one for the list: the row's cells get
// consecutive entries in cell order.
constexpr int ROW_THREADS = 128;
constexpr int ROW_CELLS = (2 * grid_nlat(0) + ROW_THREADS - 1) / ROW_THREADS;  // cells per thread
__global__ void __launch_bounds__(ROW_THREADS) grid_rows_kernel(TriGrid g)
{
    grid_wait();
    grid_go();
    __shared__ uint32_t s_sum[ROW_THREADS / 32], s_base;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int l = 0, row = blockIdx.x;
    while (l < GRID_LEVELS && row >= grid_nlat_of(l)) row -= grid_nlat_of(l++);
    const bool list = l == GRID_LEVELS;
    const int nlat = grid_nlat_of(l);
    const int ncol = list ? 1 : grid_ncol(nlat, row);
    const int word = list ? GRID_LIST : grid_base_of(l) + row * (2 * nlat + 1);
    uint32_t v[ROW_CELLS], sum = 0;
#pragma unroll
    for (int q = 0; q < ROW_CELLS; ++q) {
        const int c = ROW_CELLS * threadIdx.x + q;
        v[q] = c < ncol ? g.counts[word + c] : 0u;
        sum += v[q];
    }
    uint32_t incl = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += y;
    }
    if (lane == 31) s_sum[warp] = incl;
    __syncthreads();
    uint32_t before = 0, total = 0;
#pragma unroll
    for (int w = 0; w < ROW_THREADS / 32; ++w) {
        if (w < warp) before += s_sum[w];
        total += s_sum[w];
    }
    if (threadIdx.x == 0) s_base = total ? atomicAdd(&g.hdr[GRID_H_CURSOR], total) : 0u;
    __syncthreads();
    uint32_t run = s_base + before + incl - sum;
#pragma unroll
    for (int q = 0; q < ROW_CELLS; ++q) {
        const int c = ROW_CELLS * threadIdx.x + q;
        if (c < ncol) {
            g.start[word + c] = run;
            run += v[q];
        }
    }
    if (threadIdx.x == 0) g.start[word + ncol] = s_base + total;
    if (list && threadIdx.x < GRID_LEVELS) {
        g.hdr[GRID_H_MAX + threadIdx.x] = g.hdr[GRID_H_BUILD + threadIdx.x];
        g.hdr[GRID_H_BUILD + threadIdx.x] = 0u;
    }
}

// Every triangle takes a place of its cell (the counts return to zero); the
// lanes of a warp that share a cell take theirs together, so a mesh whose
// triangles crowd a few cells does not queue on their counters.  Bound by the
// scattered writes: an entry is one 32-byte sector, written and later read
// whole (1M triangles: 20.5 us; as 16 + 8 bytes in two arrays 27.8).  Finding
// the lanes that share costs 0.7 us of it.
__global__ void __launch_bounds__(256) grid_file_kernel(const float4* rec, int T, TriGrid g)
{
    grid_wait();
    grid_go();
    const unsigned FULL = 0xffffffffu;
    const int t = blockIdx.x * 256 + threadIdx.x, lane = threadIdx.x & 31;
    if (t == 0) {
        g.hdr[GRID_H_N] = g.hdr[GRID_H_CURSOR];
        g.hdr[GRID_H_CURSOR] = 0u;
    }
    const uint32_t w = t < T ? g.where[t] : 0xffffffffu;
    const bool ok = w < (uint32_t)GRID_WORDS;
    F8 cap{};
    if (ok) cap = ld_f8(rec + rec_at((size_t)T, t, RF_CAP));
    const unsigned peers = __match_any_sync(FULL, w);
    const int leader = __ffs(peers) - 1;
    uint32_t left = 0;
    if (lane == leader && ok) left = g.start[w] + atomicSub(&g.counts[w], (uint32_t)__popc(peers));
    left = __shfl_sync(FULL, left, leader);
    const uint32_t e = left - 1u - (uint32_t)__popc(peers & ((1u << lane) - 1u));
    if (!ok || e >= (uint32_t)T) return;  // (counters left behind by a failed launch)
    st_f8(g.ent + 2 * (size_t)e, cap.a, make_float4(cap.b.x, __uint_as_float((uint32_t)t), 0.0f, 0.0f));
}

// One CTA per tile.  Up to WALK_BLOCK candidates: one pass, the hits listed in
// shared memory, the tile's range of the bins taken with one atomic.  More:
// a pass that counts and a pass that writes.  The last CTA to finish stores
// the total and clears the counters.
//
// The walk is a chain of loads, so a tile of many candidates (one at a rim
// whose cone spans a good part of the sphere) would outlast all the others:
// by itself a tile that tests 300k triangles took 2.1 ms, the rest of its view
// 30 us; shared, the binning of that view takes 105 us, and a burst of 32
// requests with two such views 3.7 ms instead of 4.3.  Tiles of more than `split` blocks are published in a BinShare,
// and the CTAs past the tiles (helpers) take blocks from them: first one claim
// per block that counts its hits, then, once every block is counted and the
// range taken, one per block that writes them.  A CTA waits for the counting
// only after it has claimed a block to write; every block to count was claimed
// before that, by a CTA that is running and does not wait.
constexpr int BIN_FEW = 12;  // CTAs of this kernel resident on an SM, about
struct BinShare {
    uint32_t tile, blocks;  // blocks: 0 until published
    uint32_t claim;         // blocks claimed, for counting and then for writing
    uint32_t done, n;       // blocks counted, hits found in them
    uint32_t cursor;        // next place in the bins
    uint32_t ready, pad;    // the range is taken
};
static_assert(sizeof(BinShare) == BIN_SHARE_WORDS * sizeof(uint32_t), "BIN_CTR_WORDS");

struct BinBlock {
    uint32_t n, claim, start;
    int entry, ok;
};

__global__ void __launch_bounds__(WALK_THREADS) bin_walk_kernel(const float4* rec, int T, WalkIndex wi,
                                                               const float4* geom,
                                                               const Cone* tiles, int ntiles,
                                                               uint32_t split, int looks, bool sizing,
                                                               uint32_t* __restrict__ ctr,
                                                               uint32_t* __restrict__ starts,
                                                               uint32_t* __restrict__ ends,
                                                               uint32_t* __restrict__ ids, uint32_t cap, int* status,
                                                               uint32_t* total_host)
{
    grid_wait();
    grid_go();
    __shared__ WalkShared ws;
    __shared__ uint32_t s_ids[WALK_BLOCK];
    __shared__ BinBlock bb;
    const bool helper = blockIdx.x >= (uint32_t)ntiles;
    BinShare* shares = (BinShare*)(ctr + BIN_CTR_SHARES);
    volatile uint32_t* published = ctr + 2;
    // takes the range of a tile with n hits
    auto take_range = [&](int tile, uint32_t n) {
        const uint32_t start = n ? atomicAdd(&ctr[0], n) : 0u;
        // (raised once, by the tile that lies across the bins' end: the word may
        // be host memory, and thousands can lie beyond)
        if (!sizing && start <= cap && (uint64_t)start + n > cap) raise_status(status, VSR_ERR_BIN_OVERFLOW);
        starts[tile] = start;
        ends[tile] = start + n;
        return start;
    };
    for (;;) {
        int tile = (int)blockIdx.x;
        if (helper) {
            // a published tile with blocks left, the first from a start of
            // this CTA's own
            __syncthreads();
            if (threadIdx.x == 0) {
                for (; !*published && looks > 0; --looks) __nanosleep(250);
                bb.claim = min(*published, (uint32_t)BIN_SHARES);
                bb.entry = BIN_SHARES;
            }
            __syncthreads();
            const int ne = (int)bb.claim, from = ne ? (int)((blockIdx.x * 37u) % (uint32_t)ne) : 0;
            int mine = BIN_SHARES;
            for (int i = threadIdx.x; i < ne && mine == BIN_SHARES; i += WALK_THREADS) {
                volatile BinShare* e = &shares[(from + i) % ne];
                if (e->claim < 2u * e->blocks) mine = i;
            }
            if (mine < BIN_SHARES) atomicMin(&bb.entry, mine);
            __syncthreads();
            const int found = bb.entry;
            if (found == BIN_SHARES) break;
            __syncthreads();
            if (threadIdx.x == 0) {
                bb.entry = (from + found) % ne;
                __threadfence();
                bb.claim = *(volatile uint32_t*)&shares[bb.entry].tile;
            }
            __syncthreads();
            tile = (int)bb.claim;
        }
        const Cone c = tiles[tile];
        if (threadIdx.x < 32) walk_ranges(wi, T, geom[tile], c.c0.y, ws);
        if (threadIdx.x == 0) {
            bb.n = 0u;
            const uint32_t nb = (ws.total + WALK_BLOCK - 1) / WALK_BLOCK;
            if (!helper) {
                bb.entry = -1;
                if (nb > split) {
                    const uint32_t i = atomicAdd(&ctr[2], 1u);
                    if (i < (uint32_t)BIN_SHARES) {
                        shares[i].tile = (uint32_t)tile;
                        __threadfence();
                        atomicExch(&shares[i].blocks, nb);
                        bb.entry = (int)i;
                    }
                }
            }
        }
        __syncthreads();
        const uint32_t E = ws.total;
        Walk w;
        w.init(wi, c, ws);
        if (bb.entry >= 0) {
            BinShare* e = &shares[bb.entry];
            const uint32_t nb = (E + WALK_BLOCK - 1) / WALK_BLOCK;
            for (;;) {
                __syncthreads();
                if (threadIdx.x == 0) {
                    bb.claim = atomicAdd(&e->claim, 1u);
                    bb.n = 0u;
                }
                __syncthreads();
                const uint32_t b = bb.claim;
                if (b >= 2u * nb) break;
                const uint32_t i0 = (b < nb ? b : b - nb) * WALK_BLOCK, i1 = min(E, i0 + WALK_BLOCK);
                walk_hits(w, wi, rec, T, ws, i0, i1, s_ids, &bb.n);
                __syncthreads();
                const uint32_t n = bb.n;
                if (b < nb) {
                    if (threadIdx.x == 0) {
                        atomicAdd(&e->n, n);
                        __threadfence();
                        if (atomicAdd(&e->done, 1u) == nb - 1u) {
                            __threadfence();
                            atomicExch(&e->cursor, take_range(tile, atomicAdd(&e->n, 0u)));
                            __threadfence();
                            atomicExch(&e->ready, 1u);
                        }
                    }
                    continue;
                }
                if (threadIdx.x == 0) {
                    // microseconds; a second of looks, then an error instead
                    uint32_t look = 0;
                    while (!*(volatile uint32_t*)&e->ready && look < 5000000u) {
                        __nanosleep(200);
                        ++look;
                    }
                    __threadfence();
                    bb.ok = *(volatile uint32_t*)&e->ready != 0u;
                    if (bb.ok)
                        bb.start = atomicAdd(&e->cursor, n);
                    else
                        raise_status(status, VSR_ERR_TIMEOUT);
                }
                __syncthreads();
                if (!bb.ok) break;
                const uint32_t start = bb.start;
                for (uint32_t j = threadIdx.x; j < n; j += WALK_THREADS)
                    if (start + j < cap) ids[start + j] = s_ids[j];
            }
        } else if (E <= WALK_BLOCK) {
            walk_hits(w, wi, rec, T, ws, 0u, E, s_ids, &bb.n);
            __syncthreads();
            const uint32_t n = bb.n;
            if (threadIdx.x == 0) bb.start = take_range(tile, n);
            __syncthreads();
            const uint32_t start = bb.start;
            for (uint32_t j = threadIdx.x; j < n; j += WALK_THREADS)
                if (start + j < cap) ids[start + j] = s_ids[j];
        } else {
            // block by block: count, take the range, write
            uint32_t total = 0, start = 0;
            for (int pass = 0; pass < 2; ++pass) {
                for (uint32_t i0 = 0; i0 < E; i0 += WALK_BLOCK) {
                    walk_hits(w, wi, rec, T, ws, i0, min(E, i0 + WALK_BLOCK), s_ids, &bb.n);
                    __syncthreads();
                    const uint32_t n = bb.n;
                    if (pass)
                        for (uint32_t j = threadIdx.x; j < n; j += WALK_THREADS)
                            if (start + j < cap) ids[start + j] = s_ids[j];
                    start += pass ? n : 0u;
                    total += pass ? 0u : n;
                    __syncthreads();
                    if (threadIdx.x == 0) bb.n = 0u;
                    __syncthreads();
                }
                if (!pass) {
                    if (threadIdx.x == 0) bb.start = take_range(tile, total);
                    __syncthreads();
                    start = bb.start;
                }
            }
        }
        if (!helper) break;
    }
    __syncthreads();  // this CTA's last look at the shares
    if (threadIdx.x == 0) {
        __threadfence();
        bb.ok = atomicAdd(&ctr[1], 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (!bb.ok) return;
    __threadfence();
    const uint32_t used = min(*published, (uint32_t)BIN_SHARES) * BIN_SHARE_WORDS;
    for (uint32_t i = threadIdx.x; i < used; i += WALK_THREADS) ctr[BIN_CTR_SHARES + i] = 0u;
    __syncthreads();
    if (threadIdx.x == 0) {
        const uint32_t total = atomicExch(&ctr[0], 0u);
        ctr[1] = 0u;
        ctr[2] = 0u;
        starts[ntiles] = total;
        if (total_host) {  // straight into the host's pinned word (read after an event)
            *(volatile uint32_t*)total_host = total;
            __threadfence_system();
        }
    }
}

}  // namespace

vsr_status grid_alloc(TriGrid* g, int64_t T)
{
    if (!g->counts) {
        // counters and header in one allocation, cleared by the first set-up
        if (cudaMalloc((void**)&g->counts, sizeof(uint32_t) * (2 * (size_t)GRID_WORDS + GRID_HDR)) != cudaSuccess) {
            cudaGetLastError();
            g->counts = nullptr;
            return VSR_ERR_OOM;
        }
        g->hdr = g->counts + GRID_WORDS;
        g->start = g->hdr + GRID_HDR;
        g->dirty = true;
    }
    if (T > g->T) {
        cudaFree(g->ent);
        g->where = nullptr;
        g->ent = nullptr;
        g->T = 0;
        if (cudaMalloc((void**)&g->ent, (2 * sizeof(float4) + sizeof(uint32_t)) * (size_t)T) !=
            cudaSuccess) {
            cudaGetLastError();
            return VSR_ERR_OOM;
        }
        g->where = (uint32_t*)(g->ent + 2 * T);
        g->T = T;
    }
    return VSR_OK;
}

void grid_free(TriGrid* g)
{
    cudaFree(g->counts);
    cudaFree(g->ent);
    *g = TriGrid{};
}

size_t grid_bytes(int64_t T)
{
    return sizeof(uint32_t) * (2 * (size_t)GRID_WORDS + GRID_HDR) +
           (sizeof(uint32_t) + 2 * sizeof(float4)) * (size_t)T;
}

vsr_status launch_grid_file(const float4* rec, int T, const TriGrid& g, cudaStream_t st)
{
    if (T <= 0) return VSR_OK;
    if ((int64_t)T > g.T || !g.counts) return VSR_ERR_INVALID_ARG;
    VSR_CUDA_TRY(launch_next(grid_rows_kernel, GRID_ROWS + 1, ROW_THREADS, st, g));
    VSR_CUDA_TRY(launch_next(grid_file_kernel, (T + 255) / 256, 256, st, rec, T, g));
    return VSR_OK;
}

vsr_status launch_bin_walk(const float4* rec, int T, const WalkIndex& wi, const float4* geom, const Cone* tiles,
                           int ntiles, uint32_t* ctr, uint32_t* starts, uint32_t* ends, uint32_t* ids, uint32_t cap,
                           bool sizing, int* status, uint32_t* total_host, cudaStream_t st)
{
    if (T < 0 || ntiles <= 0 || (!wi.direct && !wi.start)) return VSR_ERR_INVALID_ARG;
    const int sms = sm_count();
    if (sms < 0) return VSR_ERR_CUDA;
    // helpers, four CTAs per SM, only where a tile can have enough candidates;
    // with few tiles they start together with them and look for a while (the
    // others would finish the tiles' own blocks later than these start).  A
    // tile of 4 blocks by itself takes 58 us, about what the rest of a view
    // does; with few tiles there is nothing to hide 4 behind, so 2.
    const bool few = ntiles < BIN_FEW * sms;
    const uint32_t split = few ? 2u : 4u;
    const int helpers = (uint32_t)T > split * WALK_BLOCK ? 4 * sms : 0;
    VSR_CUDA_TRY(launch_next(bin_walk_kernel, ntiles + helpers, WALK_THREADS, st, rec, T, wi, geom, tiles, ntiles, split,
                             few ? 40 : 0, sizing, ctr, starts, ends, ids, cap, status, total_host));
    return VSR_OK;
}
