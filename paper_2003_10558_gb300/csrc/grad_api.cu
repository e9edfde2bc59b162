// grad_api.cu -- C ABI of the differentiable path: vsr_frags,
// vsr_raster_shaded and vsr_raster_backward (kernels in grad.cu, map.cu).
#include <math.h>
#include <new>

#include "handles.cuh"

struct vsr_frags_s {
    size_t npix = 0, ntiles = 0;  // per-pixel and per-tile buffers sized for these
    uint2* span = nullptr;        // npix
    uint32_t* bits = nullptr;     // npix x FRAG_LIST / 32
    uint32_t* tile_n = nullptr;   // ntiles
    uint32_t* tile_ids = nullptr; // ntiles x FRAG_LIST
    uint32_t* cursor = nullptr;
    bool dirty = true;            // the cursor is not known to be zero
    float4* frags = nullptr;
    uint32_t fcap = 0;
    bool unlisted = false;        // the last frame had tiles without a list
    uint32_t* h_total = nullptr;  // pinned: fragments, tiles without a list
    cudaEvent_t counted = nullptr;  // the total is in h_total
    float4* dmap = nullptr;       // npix
    float* lens_part = nullptr;
    float4* grad = nullptr;       // GF_COUNT x grad_T
    int64_t grad_T = 0;
    bool grad_clean = false;      // grad is all zero, after the work queued so far and between replays of captured work
    // the forward the lists belong to
    uint64_t map_gen = 0, scene_gen = 0;
    int W = 0, H = 0;
    bool valid = false;
};

namespace {

void frags_release_pixels(vsr_frags f)
{
    cudaFree(f->span);
    cudaFree(f->bits);
    cudaFree(f->tile_n);
    cudaFree(f->tile_ids);
    cudaFree(f->dmap);
    cudaFree(f->lens_part);
    f->span = nullptr;
    f->bits = nullptr;
    f->tile_n = f->tile_ids = nullptr;
    f->dmap = nullptr;
    f->lens_part = nullptr;
    f->npix = f->ntiles = 0;
}

vsr_status frags_ensure_pixels(vsr_frags f, int W, int H, size_t ntiles, cudaStream_t st)
{
    const size_t n = (size_t)W * H;
    vsr_status s;
    if (!f->cursor && (s = dalloc(&f->cursor, 2)) != VSR_OK) return s;
    if (n <= f->npix && ntiles <= f->ntiles) return VSR_OK;
    frags_release_pixels(f);
    if ((s = dalloc(&f->span, n)) != VSR_OK || (s = dalloc(&f->bits, n * (FRAG_LIST / 32))) != VSR_OK ||
        (s = dalloc(&f->tile_n, ntiles)) != VSR_OK || (s = dalloc(&f->tile_ids, ntiles * FRAG_LIST)) != VSR_OK ||
        (s = dalloc(&f->dmap, n)) != VSR_OK || (s = dalloc(&f->lens_part, map_backward_partials(ntiles))) != VSR_OK) {
        frags_release_pixels(f);
        return s;
    }
    if (cudaMemsetAsync(f->lens_part, 0, sizeof(float), st) != cudaSuccess) {
        frags_release_pixels(f);
        return VSR_ERR_CUDA;
    }
    f->npix = n;
    f->ntiles = ntiles;
    return VSR_OK;
}

FragArgs frag_args(vsr_map m, vsr_scene sc, const float* colors, vsr_frags f)
{
    FragArgs a{};
    a.map = m->map;
    a.W = m->p.W;
    a.H = m->p.H;
    a.tiles_x = m->tx;
    a.tiles = m->tiles;
    a.geom = m->idx.geom;
    a.rec = sc->rec;
    a.T = (int)sc->T;
    a.wi = walk_index(sc->grid, sc->T);
    a.colors = colors;
    a.cursor = f->cursor;
    a.tile_n = f->tile_n;
    a.tile_ids = f->tile_ids;
    a.span = f->span;
    a.bits = f->bits;
    a.frags = f->frags;
    a.fcap = f->fcap;
    a.status = scene_status(sc);
    return a;
}

}  // namespace

extern "C" {

vsr_status vsr_frags_create(vsr_frags* out)
{
    if (!out) return VSR_ERR_INVALID_ARG;
    *out = nullptr;
    vsr_frags f = new (std::nothrow) vsr_frags_s;
    if (!f) return VSR_ERR_OOM;
    if (cudaMallocHost((void**)&f->h_total, 2 * sizeof(uint32_t)) != cudaSuccess ||
        cudaEventCreateWithFlags(&f->counted, cudaEventDisableTiming) != cudaSuccess) {
        cudaGetLastError();
        if (f->h_total) cudaFreeHost(f->h_total);
        delete f;
        return VSR_ERR_OOM;
    }
    *out = f;
    return VSR_OK;
}

void vsr_frags_free(vsr_frags f)
{
    if (!f) return;
    frags_release_pixels(f);
    cudaFree(f->cursor);
    cudaFree(f->frags);
    cudaFree(f->grad);
    if (f->h_total) cudaFreeHost(f->h_total);
    if (f->counted) cudaEventDestroy(f->counted);
    delete f;
}

vsr_status vsr_raster_shaded(vsr_map m, vsr_scene sc, const float* colors_dev, vsr_frags f, float* image_dev,
                             float* cov_dev, uint32_t* id_dev, float* depth_dev, void* stream)
{
    if (!m || !sc || !f) return VSR_ERR_INVALID_ARG;
    cudaStream_t st = (cudaStream_t)stream;
    f->valid = false;
    vsr_status s;
    // the first frame of a shape also sizes the stored bins (see raster_frame)
    if ((s = scene_walk_begin(m, sc, st)) != VSR_OK) return s;
    const int W = m->p.W, H = m->p.H;
    if ((s = frags_ensure_pixels(f, W, H, (size_t)m->tx * m->ty, st)) != VSR_OK) return s;
    FragArgs a = frag_args(m, sc, colors_dev, f);
    a.out_id = id_dev;
    a.out_depth = depth_dev;
    if (f->dirty) VSR_CUDA_TRY(cudaMemsetAsync(f->cursor, 0, 2 * sizeof(uint32_t), st));
    f->dirty = true;  // until the fill, which clears it, is queued
    if ((s = launch_frag_count(a, sc->walk, sc->tile_pairs, st)) != VSR_OK) return s;
    VSR_CUDA_TRY(cudaMemcpyAsync(f->h_total, f->cursor, 2 * sizeof(uint32_t), cudaMemcpyDeviceToHost, st));
    VSR_CUDA_TRY(cudaEventRecord(f->counted, st));
    a.image = image_dev;
    a.cov = cov_dev;
    // Filled into the room there is before the host knows the total: it is
    // almost always enough (kept a quarter above the largest so far), and the
    // device does not stand still for the host's round trip (1024^2 pixels, 10k
    // triangles, a frame with its backward: 158.7 us before, 153.0 with it).
    // If it was not, once more with more.
    const bool early = f->fcap > 0, early_walk = early && f->unlisted;
    if (early) {
        a.early = true;
        if ((s = launch_frag_fill(a, st)) != VSR_OK) return s;
        if (early_walk && (s = launch_frag_fill_walk(a, sc->walk, st)) != VSR_OK) return s;
        a.early = false;
    }
    VSR_CUDA_TRY(cudaEventSynchronize(f->counted));
    const uint32_t total = f->h_total[0], unlisted = f->h_total[1];
    if (total > f->fcap) {
        cudaFree(f->frags);
        f->frags = nullptr;
        f->fcap = 0;
        uint64_t want = (uint64_t)total + total / 4 + 1024;
        if (want > 0xffffffffull) want = 0xffffffffull;
        if ((s = dalloc(&f->frags, (size_t)want)) != VSR_OK) return s;
        f->fcap = (uint32_t)want;
    }
    const bool again = !early || a.fcap != f->fcap;
    if (again) {
        a.frags = f->frags;
        a.fcap = f->fcap;
        if ((s = launch_frag_fill(a, st)) != VSR_OK) return s;
    }
    f->unlisted = unlisted > 0;
    if (f->unlisted && (again || !early_walk) && (s = launch_frag_fill_walk(a, sc->walk, st)) != VSR_OK) return s;
    f->dirty = false;
    f->map_gen = m->gen;
    f->scene_gen = sc->gen;
    f->W = W;
    f->H = H;
    f->valid = true;
    return scene_used(sc, st);
}

vsr_status vsr_raster_backward(vsr_map m, vsr_scene sc, const float* tris_dev, const float* colors_dev, vsr_frags f,
                               const uint32_t* id_dev, const float* dimage_dev, const float* dcov_dev,
                               const float* ddepth_dev, float* dtris_dev, float* dcolors_dev, double* dlens_dev,
                               void* stream)
{
    if (!m || !sc || !f || !f->valid) return VSR_ERR_INVALID_ARG;
    if (f->map_gen != m->gen || f->scene_gen != sc->gen || f->W != m->p.W || f->H != m->p.H)
        return VSR_ERR_INVALID_ARG;
    if (ddepth_dev && !id_dev) return VSR_ERR_INVALID_ARG;
    if (dtris_dev && sc->T > 0 && !tris_dev) return VSR_ERR_INVALID_ARG;
    if (dlens_dev && !m->lens_grad) return VSR_ERR_INVALID_ARG;
    cudaStream_t st = (cudaStream_t)stream;
    const int64_t T = sc->T;
    vsr_status s;
    if (T > f->grad_T) {
        cudaFree(f->grad);
        f->grad = nullptr;
        f->grad_T = 0;
        if ((s = dalloc(&f->grad, (size_t)GF_COUNT * (size_t)T)) != VSR_OK) return s;
        f->grad_T = T;
        f->grad_clean = false;
    }
    // Every backward leaves the record gradients cleared, the set-up adjoint
    // by itself.  A captured one does so at each replay and changes nothing
    // before, so the flag stays what it was: a clear that the buffer still
    // needs is captured with it, and the next eager call has its own.
    bool captures;
    if ((s = stream_captures(st, &captures)) != VSR_OK) return s;
    const bool clean = f->grad_clean;
    if (f->grad_T > 0 && !clean)
        VSR_CUDA_TRY(cudaMemsetAsync(f->grad, 0, sizeof(float4) * GF_COUNT * (size_t)f->grad_T, st));
    f->grad_clean = false;  // until all of it is queued
    FragArgs a = frag_args(m, sc, colors_dev, f);
    if ((s = launch_frag_backward(a, id_dev, dimage_dev, dcov_dev, ddepth_dev, f->grad, f->dmap, st)) != VSR_OK)
        return s;
    if (dtris_dev || dcolors_dev) {
        if ((s = launch_setup_backward(tris_dev, (int)T, sc->cam, sc->rec, f->grad, dtris_dev, dcolors_dev, st)) !=
            VSR_OK)
            return s;
    } else if (T > 0) {
        VSR_CUDA_TRY(cudaMemsetAsync(f->grad, 0, sizeof(float4) * GF_COUNT * (size_t)T, st));
    }
    f->grad_clean = !captures || clean;
    if (dlens_dev) {
        if ((s = launch_map_backward(m->p.W, m->p.H, m->p.aov, m->p.k, m->p.l, m->p.s, m->p.omega_deg, f->dmap,
                                     f->lens_part, dlens_dev, st)) != VSR_OK)
            return s;
    }
    return scene_used(sc, st);
}

}  // extern "C"
