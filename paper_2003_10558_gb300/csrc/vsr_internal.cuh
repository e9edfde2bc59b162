// vsr_internal.cuh -- layouts and helpers shared by the kernels and the host
// library of the visual-sphere rasterizer.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <initializer_list>

#include "../../include/vsr.h"

// ---------------------------------------------------------------------------
// Tiling.  The map is cut into TILE x TILE pixel tiles (one raster CTA each).
constexpr int TILE = 16;
constexpr int TILE_PIX = TILE * TILE;

// ---------------------------------------------------------------------------
// Per-triangle set-up record: REC_F float4 fields in two arrays, the bodies
// (8 fields, one 128-byte line per triangle) first, then the caps (2 fields,
// one 32-byte sector per triangle).  The raster gathers the records of the
// triangles of a bin, in no order of memory: a record is five whole sectors
// (with every field in an array of its own it was ten half-used ones).  The
// binner reads the caps alone, coalesced.
enum {
    RF_N1 = 0,   // body: (n_AB.hi xyz, tie flags)      edge normals, FP32 high parts
    RF_N2 = 1,   // (n_BC.hi xyz, 0)
    RF_N3 = 2,   // (n_CA.hi xyz, 0)
    RF_PL = 3,   // (N-hat.hi xyz, (A'.N)/|N|)         plane for the ray-plane depth
    RF_N1L = 4,  // (n_AB.lo xyz, S-hat.lo.x)          low parts
    RF_N2L = 5,  // (n_BC.lo xyz, S-hat.lo.y)
    RF_N3L = 6,  // (n_CA.lo xyz, S-hat.lo.z)
    RF_PLL = 7,  // (N-hat.lo xyz, 0)
    REC_BODY = 8,
    RF_CAP = 8,  // cap: (S-hat.hi xyz, cos rho)        miter cap centre and radius
    RF_CAP2 = 9, // (sin rho, 2(1 - cos rho), 1/(2 sin rho), valid ? 1 : 0)
    REC_F = 10
};
// field f of triangle t in the records of TT triangles
__host__ __device__ __forceinline__ size_t rec_at(size_t TT, size_t t, int f)
{
    return f < REC_BODY ? REC_BODY * t + f : REC_BODY * TT + (REC_F - REC_BODY) * t + (f - REC_BODY);
}

// Two consecutive fields (32 bytes, 32-byte aligned: an even field) in one
// 256-bit access of sm_100+.  A plain load that stays where it stands: what it
// reads is written by a kernel that may end while this one's CTAs are already
// resident (grid_wait), so it is not read-only for this kernel's lifetime, as
// ld.global.nc wants it.  For the same reason a kernel that waits takes no
// `const T* __restrict__`, which lets the compiler choose that load.
struct __align__(16) F8 {
    float4 a, b;
};
__device__ __forceinline__ F8 ld_f8(const float4* p)
{
    F8 v;
    asm volatile("ld.global.v8.f32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=f"(v.a.x), "=f"(v.a.y), "=f"(v.a.z), "=f"(v.a.w), "=f"(v.b.x), "=f"(v.b.y), "=f"(v.b.z),
                   "=f"(v.b.w)
                 : "l"(p)
                 : "memory");
    return v;
}
__device__ __forceinline__ void st_f8(float4* p, const float4& a, const float4& b)
{
    asm volatile("st.global.v8.f32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(p), "f"(a.x), "f"(a.y), "f"(a.z),
                 "f"(a.w), "f"(b.x), "f"(b.y), "f"(b.z), "f"(b.w)
                 : "memory");
}

// tie flags in RF_N1.w (as integer bits): bit i set <=> the first nonzero
// component of edge normal i is positive (simulation-of-simplicity rule for
// g_i == 0 in the centre test).

// ---------------------------------------------------------------------------
// Tile cones (per tile, 2 float4):
//   c0 = (axis xyz, cos alpha)   all valid pixel directions of the tile lie
//                                within alpha of the axis
//   c1 = (sin alpha, h, n_valid, 0) with h = max over valid pixels of
//                                1/(2 delta) (the widest ramp half-width)
// An empty tile has n_valid = 0.
struct Cone {
    float4 c0, c1;
};

// ---------------------------------------------------------------------------
// Tile index of a map: a latitude-longitude grid over the view sphere
// (latitude = asin(y), longitude = atan2(x, z), so the grid's poles are the
// camera's +-y axis).  Every tile whose cone half-angle is at most alpha_cut
// is filed once, in the cell holding its axis; larger ("big") tiles are kept
// in a separate list that every triangle scans.  A triangle whose enlarged
// cap has angular radius beta can only reach small tiles whose axis lies
// within beta + alpha_small_max of the cap centre, i.e. in a small
// latitude/longitude window of cells.  Grid size and alpha_cut are chosen on
// the device from the distribution of tile half-angles.  The index serves
// the triangle-major search of the fixed-array path and is built on its
// first use after each generation of the map.
constexpr int IDX_NLAT_MAX = 128;
constexpr int IDX_CELLS_MAX = IDX_NLAT_MAX * 2 * IDX_NLAT_MAX;
constexpr int IDX_HIST = 64;

struct TileIndexHdr {
    int nlat, nlon;             // grid: nlon = 2 nlat, square cells of `cell` radians
    int ncell;                  // nlat * nlon
    float cell;
    float alpha_cut;            // small / big tile threshold (radians)
    unsigned alpha_small_max;   // float bits: largest half-angle of a small tile
    unsigned h_max;             // float bits: largest ramp half-width 1/(2 delta)
    unsigned n_big;
    unsigned n_valid;
    // float bits: the half-angle about the camera's +z axis of a cone that
    // holds every tile cone (the map's field of view), plus a margin; 0 for a
    // map without a valid pixel
    unsigned view_angle;
    unsigned hist[IDX_HIST];    // third-of-an-octave histogram of half-angles
};

// Device-side status word (vsr_status values; 0 = OK), one int per device
// owned by the host library and passed to the kernels that can fail.
__device__ __forceinline__ void raise_status(int* status, int code)
{
    if (status) atomicCAS(status, 0, code);
}

// Conservative test: may a cap (centre S, cos/sin of radius, enlarged by the
// ramp half-width h measured on the miter's normalised distance) reach a
// direction inside the cone (axis, cos/sin alpha)?
//   fragment region of the miter:  G.S - cos rho > -h sin rho
//   i.e. a cap of cos(beta) = cos rho - h sin rho.
__device__ __forceinline__ bool cap_hits_cone(float3 S, float cos_rho, float sin_rho, float3 axis, float cos_a,
                                              float sin_a, float h)
{
    const float eps = 2e-6f;
    float cb = cos_rho - h * sin_rho;
    if (cb + cos_a <= eps) return true;  // alpha + beta >= pi
    if (cb <= -1.0f) return true;
    float sb = sqrtf(fmaxf(0.0f, 1.0f - cb * cb));
    float cg = S.x * axis.x + S.y * axis.y + S.z * axis.z;
    return cg >= cos_a * cb - sin_a * sb - eps;
}

// (the failed call's error is taken from the runtime, or a later check of
// another launch would find it)
#define VSR_CUDA_TRY(expr)                                                                                              \
    do {                                                                                                                \
        cudaError_t _e = (expr);                                                                                        \
        if (_e != cudaSuccess) {                                                                                        \
            cudaGetLastError();                                                                                         \
            return VSR_ERR_CUDA;                                                                                        \
        }                                                                                                               \
    } while (0)

// Launches one after another on a stream hand over without draining the GPU
// in between (programmatic dependent launch): a kernel launched with
// launch_next may have its CTAs placed while its predecessor's last ones still
// run; grid_go in the predecessor allows it.  Nothing before grid_wait, which
// returns with the predecessor's end and memory, touches global memory: most
// kernels wait first, and the map kernels evaluate what depends on their
// arguments alone, in registers and shared memory, before they wait.  A
// frame's five launches: about 10 us less.
__device__ __forceinline__ void grid_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void grid_go() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
template <class... P, class... A>
inline cudaError_t launch_next(void (*kernel)(P...), dim3 grid, dim3 block, cudaStream_t st, A... args)
{
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.stream = st;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, P(args)...);
}

// Kernel launchers (defined in the .cu files, called by the host library).
// The map kernels write the map, the tile cones and their geometry.
vsr_status launch_map(int W, int H, int aov, float k, float l, float s, float omega_deg, float4* map, Cone* tiles,
                      float4* geom, cudaStream_t st);
vsr_status launch_map_cones(const float4* map, int W, int H, Cone* tiles, float4* geom, cudaStream_t st);
// a map of any vsr_map_kind (param after limits for the Universal kind);
// deriv (optional): 2 float4 per pixel, (d_i G, d_j G) for the pixel step
vsr_status launch_map_spec(const vsr_map_spec& spec, float4* map, Cone* tiles, float4* geom, float4* deriv,
                           cudaStream_t st);
struct TriGrid;
// grid: count the triangles' cells for launch_grid_file (NULL: no grid);
// on_host: tris is the device address of host memory
vsr_status launch_setup(const float* tris, int T, const float cam[12], float4* rec, const TriGrid* grid,
                        cudaStream_t st, bool on_host);

// Device memory of a tile index (sized for IDX_CELLS_MAX cells, ntiles tiles).
// The cones of the small tiles are stored sorted by home cell, so the cells
// of one grid row form one contiguous range: (axis xyz, cos alpha),
// (sin alpha, h, tile index bits, 0).  Big tiles are stored the same way.
struct TileIndex {
    TileIndexHdr* hdr;
    uint32_t* cell_start;  // IDX_CELLS_MAX + 1
    Cone* sorted;          // ntiles
    Cone* big;             // ntiles
    float4* geom;          // ntiles: (alpha, latitude, longitude of the axis, h), h = -1 if the tile is empty;
                           // written with the cones by the map kernels
    uint32_t ntiles;       // tiles of the map (the length of sorted, big and geom)
};
// The whole index from the tile cones and geometry (any generation).
vsr_status launch_tile_index(const Cone* tiles, int ntiles, TileIndex idx, cudaStream_t st);

// Grid arithmetic of the tile index (bin.cu).
constexpr float IDX_PI = 3.14159265358979f;

__device__ __forceinline__ int hist_bin(float a)
{
    // third-of-an-octave bins from 2^-17 rad
    int b = (int)floorf((log2f(fmaxf(a, 1e-30f)) + 17.0f) * 3.0f);
    return min(IDX_HIST - 1, max(0, b));
}

__device__ __forceinline__ int cell_row(float lat, const TileIndexHdr& h)
{
    return min(h.nlat - 1, max(0, (int)floorf((lat + 0.5f * IDX_PI) / h.cell)));
}

__device__ __forceinline__ int cell_col(float lon, const TileIndexHdr& h)
{
    int c = (int)floorf((lon + IDX_PI) / h.cell);
    c %= h.nlon;
    return c < 0 ? c + h.nlon : c;
}

__device__ __forceinline__ int home_cell_geom(const float4& g, const TileIndexHdr& h)
{
    return cell_row(g.y, h) * h.nlon + cell_col(g.z, h);
}

// A tile's reach from the camera's +z axis, as float bits (non-negative, so
// they order as the floats): the angle of its axis from +z plus its
// half-angle and a margin for the FP32 rounding.
__device__ __forceinline__ unsigned view_angle_bits(const Cone& c, float alpha)
{
    return __float_as_uint(acosf(fmaxf(-1.0f, fminf(1.0f, c.c0.z))) + alpha + 1e-5f);
}

// The index's copy of tile i's cone: (axis xyz, cos alpha), (sin alpha, h,
// tile index bits, 0).
__device__ __forceinline__ Cone index_entry(const Cone& c, int i)
{
    Cone e;
    e.c0 = c.c0;
    e.c1 = make_float4(c.c1.x, c.c1.y, __uint_as_float((uint32_t)i), 0.0f);
    return e;
}
// triangle-major binning of one frame (vsr_raster_noalloc): counts zeroed by
// the caller -> launch_bin_count -> launch_scan -> launch_bin_fill (a second
// search)
vsr_status launch_bin_count(const float4* rec, int T, TileIndex idx, uint32_t* counts, cudaStream_t st);
vsr_status launch_scan(const uint32_t* counts, int n, uint32_t* offsets, cudaStream_t st);
vsr_status launch_bin_fill(const float4* rec, int T, TileIndex idx, const uint32_t* offsets, uint32_t* counts,
                           uint32_t* ids, uint32_t cap, int* status, cudaStream_t st);

// ---------------------------------------------------------------------------
// Triangle grid: the triangles of a set-up by the place of their caps on the
// view sphere, built with the set-up (it does not depend on the map) and
// walked by every tile of a raster or binning (walk.cuh).
//
// GRID_LEVELS latitude-longitude grids (latitude = asin(y), longitude =
// atan2(x, z)), 192 rows in the finest; a triangle is filed by its cap's
// centre in the finest level whose cells are at least as tall as its cap
// radius (twice the height in the coarsest), and in a list beyond that.  Rows
// near the poles have fewer cells (grid_ncol), so cells are of about equal
// area.  The triangles of a row's cells are consecutive entries in cell order,
// so a window of a row is one range of entries (two where it wraps), and the
// levels' largest radii bound how far a tile has to look.  The entries are
// sorted by counting (cell counts in the set-up kernel, row starts, entries),
// so there is no capacity per cell.
// The levels by a model of the candidates per tile (window area x density) on
// the 1080p frame, a 4096 x 2176 frame, a view inside a cloud and smaller
// ones: 2.4 - 4.2 per triangle whose cap reaches the tile, against 2.4 - 4.3
// with levels of 192, 48, 12 rows and 3.0 - 7.5 with 128, 16; levels of 256
// and 512 rows save up to a fifth of the candidates but double the ranges.
constexpr int GRID_LEVELS = 4;
__host__ __device__ constexpr int grid_nlat(int l) { return l == 0 ? 192 : (l == 1 ? 96 : (l == 2 ? 48 : 12)); }
__host__ __device__ constexpr int grid_stride(int l) { return 2 * grid_nlat(l) + 1; }  // words per row: cells, end
__host__ __device__ constexpr int grid_base(int l)
{
    int b = 0;
    for (int q = 0; q < l; ++q) b += grid_nlat(q) * grid_stride(q);
    return b;
}
constexpr int GRID_LIST = grid_base(GRID_LEVELS);  // the list: its start, its end
constexpr int GRID_WORDS = GRID_LIST + 2;
constexpr int GRID_ROWS = grid_nlat(0) + grid_nlat(1) + grid_nlat(2) + grid_nlat(3);
// header words
constexpr int GRID_H_BUILD = 0;   // [0 .. 3] per level: float bits of the largest sin(cap radius), while filing
constexpr int GRID_H_CURSOR = 4;  // entries given to rows, while filing
constexpr int GRID_H_MAX = 8;     // [8 .. 11] the filed triangles' largest sin(cap radius) per level, 0: level empty
constexpr int GRID_H_N = 12;      // entries
constexpr int GRID_HDR = 16;
// Scenes of up to this many triangles have no grid: every tile tests them all,
// at most five steps of a CTA, against two filing launches and the search for
// its ranges.  us a frame, without and with a grid: 400 triangles 17.8 / 24.8
// at 256x256, 55.5 / 66.3 at 1920x1080; 600 triangles 18.6 / 29.4, 59.8 / 67.5,
// and 201 / 216 at 4096x2176, but 768 triangles 258 / 254 there with a wide
// lens, and 1024 triangles 242 / 228.
constexpr int GRID_DIRECT = 640;
struct TriGrid {
    uint32_t* counts = nullptr;  // GRID_WORDS: triangles counted per cell, then left to place; zero between set-ups
    uint32_t* start = nullptr;   // GRID_WORDS: first entry of each cell, each row closed by its end
    uint32_t* hdr = nullptr;     // GRID_HDR
    uint32_t* where = nullptr;   // T: cell word, or ~0 without a cap
    float4* ent = nullptr;       // 2 per entry: (S-hat xyz, cos rho), (sin rho, triangle bits, 0, 0)
    int64_t T = 0;               // capacity
    bool dirty = false;          // host side: a failed set-up may have left counters behind
};
vsr_status grid_alloc(TriGrid* g, int64_t T);
void grid_free(TriGrid* g);
size_t grid_bytes(int64_t T);
// row starts and entries from the cells and counts of the set-up kernel
vsr_status launch_grid_file(const float4* rec, int T, const TriGrid& g, cudaStream_t st);
// what the walk reads: a grid, or (direct) the caps of all T triangles
struct WalkIndex {
    const uint32_t* start;
    const uint32_t* hdr;
    const float4* ent;
    int direct;
    int pstep;  // caps of the per-fragment pixel step
};
inline bool grid_used(int64_t T) { return T > GRID_DIRECT; }
inline WalkIndex walk_index(const TriGrid& g, int64_t T, int pstep = 0)
{
    return WalkIndex{g.start, g.hdr, g.ent, grid_used(T) ? 0 : 1, pstep};
}
// binning by the walk: every tile's bin, in one launch.  starts / ends: ntiles
// + 1 / ntiles words, tile u's ids at [starts[u], ends[u]) in no order of
// tiles, starts[ntiles] the total; ctr: BIN_CTR_WORDS words, zero between
// binnings (pairs, CTAs done, tiles shared between CTAs, and those tiles' words).
// With more pairs than cap the bins are cut at cap and VSR_ERR_BIN_OVERFLOW is
// raised, unless the launch only sizes the bins; total_host (optional): the device address of a pinned host word that
// also receives the total.
constexpr int BIN_SHARES = 1024, BIN_SHARE_WORDS = 8, BIN_CTR_SHARES = 8;
constexpr int BIN_CTR_WORDS = BIN_CTR_SHARES + BIN_SHARES * BIN_SHARE_WORDS;
vsr_status launch_bin_walk(const float4* rec, int T, const WalkIndex& wi, const float4* geom, const Cone* tiles,
                           int ntiles, uint32_t* ctr, uint32_t* starts, uint32_t* ends, uint32_t* ids, uint32_t cap,
                           bool sizing, int* status, uint32_t* total_host, cudaStream_t st);
// One view as the raster kernel sees it: its map, tile cones, set-up
// records, bin offsets (indexed by the view's own tile number), bin ids and
// outputs.
struct RasterView {
    const float4* map;
    int W, H;
    const Cone* tiles;
    int tiles_x;
    const float4* rec;
    int T;
    const uint32_t* offsets;
    const uint32_t* ids;
    uint32_t cap;
    uint32_t* out_id;
    float* out_depth;
    float* out_cov;
    // stored bins of the walk: tile u's bin ends at ends[u] (NULL: bins in
    // tile order, tile u's ending at offsets[u + 1])
    const uint32_t* ends = nullptr;
};

// One view as the binner sees it (tile index of the view's map, the view's
// set-up records, its per-tile counters and offsets).
struct BinView {
    const TileIndexHdr* hdr;
    const uint32_t* cell_start;
    const Cone* sorted;
    const Cone* big;
    const float4* rec;
    uint32_t* counts;
    const uint32_t* offsets;
    uint32_t ntiles;    // tiles of the map: every index read from the tile index is clamped to it
};

// The cap that holds every fragment of the per-fragment pixel step
// (pstep.cu): its miter test G.S - cos rho > -(|S.d_i G| + |S.d_j G|)/2 is
// not scaled by sin rho like the global step's, and |S.d G| <= sin(theta)
// |d G| at angle theta from S, so with h >= the widest ramp half-width
// (|d_i G| + |d_j G|)/2 every fragment lies within the angle rho + 4h of S.
// pstep_ramp: (cos, sin) of 4h, (-1, 0) from pi on; pstep_cap: (cos, sin) of
// rho + 4h, cos -1 (the whole sphere) past the antipode.
__device__ __forceinline__ float2 pstep_ramp(float h)
{
    float2 e = make_float2(-1.0f, 0.0f);
    if (4.0f * h < IDX_PI) sincosf(4.0f * h, &e.y, &e.x);
    return e;
}
__device__ __forceinline__ float2 pstep_cap(float cos_rho, float sin_rho, float2 ramp)
{
    float c = fmaf(cos_rho, ramp.x, -sin_rho * ramp.y);
    const float s = fmaf(sin_rho, ramp.x, cos_rho * ramp.y);
    if (ramp.x <= -1.0f || (s < 0.0f && c < 0.0f)) c = -1.0f;
    return make_float2(c, s);
}

// Work items of the raster: a tile whose bin is longer than split_max
// triangles is processed by several CTAs whose results merge order-free
// (see SplitAcc in tile.cuh).
constexpr uint32_t SPLIT_SLOTS = 4096;    // split tiles per launch (others run unsplit)
constexpr uint32_t EXTRA_ITEMS = 1u << 16;  // extra items per launch
constexpr int SPLIT_MAX_DEFAULT = 512;    // triangles per item of a split tile
struct RasterWork {
    uint32_t* nsplit_of;      // n_tiles: items of each tile
    int32_t* split_slot;      // n_tiles: accumulator slot of a split tile, -1 if not split
    uint32_t* counters;       // 2: split tiles, extra items
    uint2* extra;             // extra_cap: (tile, k) of the further items
    uint32_t split_cap, extra_cap;
    unsigned long long* acc;  // split_cap x TILE_PIX, zero between frames
    unsigned long long* key;  // split_cap x TILE_PIX, all ones between frames
    uint32_t* done;           // split_cap, zero between frames
};
// SMs of the current device (looked up once per device), or -1.
int sm_count();
// Fills workspace that the library has just allocated or found dirty with its
// initial bytes: on st, before the launches that follow there; where st
// captures, at once, since eager work may use it before the graph's first
// launch, and replays find it as any launch leaves it.
struct Fill {
    void* p;
    int byte;
    size_t n;
};
vsr_status clear_workspace(std::initializer_list<Fill> fills, cudaStream_t st);

// A view's raster work for the pooled launch: the view, its item assignment
// (from launch_raster_assign) and its split accumulators.
struct PoolView {
    RasterView view;
    uint32_t n_tiles;
    const uint32_t* nsplit_of;
    const int32_t* split_slot;
    const uint2* extra;
    const uint32_t* n_extra;  // the work's counters + 1
    unsigned long long* acc;
    unsigned long long* key;
    uint32_t* done;
};
// items of a tile's split (a multiple of the staging chunk) and the room for
// extra items a view's work gets for bins of capacity cap
int raster_split_items(int split_max);
uint32_t raster_extra_cap(uint32_t cap, const RasterWork& w, int split_max);
// the work items of one view (split tiles, extra items), for the pooled
// launch; ends: as RasterView::ends
vsr_status launch_raster_assign(const uint32_t* offsets, uint32_t n_tiles, uint32_t cap, RasterWork w, int split_max,
                                cudaStream_t st, const uint32_t* ends = nullptr);
// one persistent raster launch over the items of several views: view v owns
// items item_start[v] .. item_start[v + 1] - 1 (its tiles, then its extra
// items); queue: a device counter (zeroed here)
vsr_status launch_raster_pool(const PoolView* views_dev, const uint32_t* item_start_dev, int nviews,
                              uint32_t* queue, int split_max, int* status, cudaStream_t st);
// items + raster over all tiles of a view; offsets: its bin offsets
// (n_tiles + 1 entries, or the bins' starts with view.ends); cap: the bins' capacity (bounds the extra items);
// host_out: the outputs are pinned host memory (written in whole tile rows)
vsr_status launch_raster_items(const RasterView& view, const uint32_t* offsets, uint32_t n_tiles, uint32_t cap,
                               RasterWork w, int split_max, int* status, cudaStream_t st, bool host_out = false);
// binning and raster in one launch over the grid (raster_walk_kernel): the
// slots in which the parts of a tile with many candidates merge
// (at least the tiles of one wave of CTAs, so that where every tile of a small
// picture is crowded none is left to one CTA: 1200 tiles of 9000 triangles each,
// 50k of 0.5 rad at 640x480, 2570 us a frame with 1024 slots, 1334 with 1280)
constexpr int WALK_SLOTS = 1280;
// Owners take slots this far apart (modulo their number), so that published
// tiles lie evenly among them: helpers look from starts of their own, and where
// the slots in use are side by side nearly all come to the first.  1920x1080,
// 100k triangles in 0.06 rad 284 -> 226 us, 640x480, 200k in 0.15 rad 244 -> 159.
constexpr uint32_t WALK_SLOT_STEP = 797;
struct WalkWork {
    char* mem = nullptr;
};
// (cleared with clear_workspace; a launch leaves the slots as it found them)
vsr_status walk_work_alloc(WalkWork* w, cudaStream_t st);
void walk_work_free(WalkWork* w);
constexpr size_t WALK_WORK_BYTES = (size_t)WALK_SLOTS * (16 * TILE_PIX + 20) + 16;
// view: no bins needed; tile_pairs (optional): the triangles found per tile;
// host_out: as launch_raster_items
vsr_status launch_raster_walk(const RasterView& view, const WalkIndex& wi, const float4* geom, const WalkWork& work,
                              uint32_t* tile_pairs, int* status, cudaStream_t st, bool host_out = false);
// the dense reference: every pixel against every triangle, no bins
vsr_status launch_raster_dense(const RasterView& view, int* status, cudaStream_t st);
// allocate / free a RasterWork for up to n_tiles tiles (accumulators cleared
// with clear_workspace: a clear on another stream would race with the launches)
vsr_status raster_work_alloc(RasterWork* w, uint32_t n_tiles, cudaStream_t st);
void raster_work_free(RasterWork* w);
int raster_threads_per_cta();
// the same with the camera in device memory (12 floats: O xyz, M 3x3 row-major)
vsr_status launch_setup_view(const float* tris, int T, const float* cam_dev, float4* rec, const TriGrid* grid,
                              cudaStream_t st);
vsr_status launch_raster(const float4* map, int W, int H, const Cone* tiles, const float4* rec, int T,
                         const uint32_t* offsets, const uint32_t* ids, uint32_t cap, uint32_t* id, float* depth,
                         float* cov, unsigned long long* n_alg, unsigned long long* n_exec, int32_t* n_inside,
                         int* status, cudaStream_t st, const uint32_t* ends = nullptr);

// ---------------------------------------------------------------------------
// Differentiable path (grad.cu, map.cu).
// Gradient of the set-up records, field-major [GF_COUNT][T] float4:
enum {
    GF_N1 = 0,   // d/d n_AB (xyz), 0
    GF_N2 = 1,   // d/d n_BC
    GF_N3 = 2,   // d/d n_CA
    GF_CAP = 3,  // d/d S-hat (xyz), d/d cos rho
    GF_PL = 4,   // d/d N-hat (xyz), d/d colour
    GF_D = 5,    // d/d (A'.N-hat), 0, 0, 0
    GF_COUNT = 6
};
constexpr int FRAG_LIST = 128;  // triangles of a tile whose fragment bits the count pass keeps
struct FragArgs {
    const float4* map;
    int W, H, tiles_x;
    const Cone* tiles;
    const float4* geom;
    const float4* rec;
    int T;
    WalkIndex wi;
    const float* colors;  // per triangle, NULL = 1
    uint32_t* cursor;     // fragments given out, tiles without a list (zero before the count, cleared by the fill)
    uint32_t* tile_n;     // per tile: its triangles, or ~0: no list (see grad.cu)
    uint32_t* tile_ids;   // per tile: FRAG_LIST of them
    uint2* span;          // per pixel: (first fragment, fragments)
    uint32_t* bits;       // FRAG_LIST / 32 pictures: a bit per triangle of the tile's list that is a fragment
    float4* frags;        // fragment records (r, t, m^f, shade)
    uint32_t fcap;
    bool early;           // the room is not known to be enough: what does not fit is left out, not an error
    float* image;
    float* cov;
    uint32_t* out_id;
    float* out_depth;
    int* status;
};
// tile_pairs: the triangles found per tile, as launch_raster_walk
vsr_status launch_frag_count(const FragArgs& a, const WalkWork& work, uint32_t* tile_pairs, cudaStream_t st);
vsr_status launch_frag_fill(const FragArgs& a, cudaStream_t st);  // tiles with a list; clears the cursor
vsr_status launch_frag_fill_walk(const FragArgs& a, const WalkWork& work, cudaStream_t st);  // the others
vsr_status launch_frag_backward(const FragArgs& a, const uint32_t* id, const float* dimage, const float* dcov,
                                const float* ddepth, float4* grad, float4* dmap, cudaStream_t st);
// (clears the record gradients it reads)
vsr_status launch_setup_backward(const float* tris, int T, const float cam[12], const float4* rec, float4* grad,
                                 float* dtris, float* dcolors, cudaStream_t st);
// size of launch_map_backward's workspace in floats, the first of which is a
// counter, zero between launches
size_t map_backward_partials(size_t ntiles);
vsr_status launch_map_backward(int W, int H, int aov, float k, float l, float s, float omega_deg,
                               const float4* dmap, float* partials, double* dlens, cudaStream_t st);

// rasterization with the per-fragment pixel step (pstep.cu), as
// launch_raster_walk with a pstep index; deriv: 2 float4 per pixel from
// launch_map_spec
vsr_status launch_raster_pstep(const RasterView& view, const float4* deriv, const WalkIndex& wi, const float4* geom,
                               const WalkWork& work, uint32_t* tile_pairs, int* status, cudaStream_t st);
