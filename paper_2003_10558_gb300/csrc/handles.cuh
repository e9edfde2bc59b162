// handles.cuh -- the library's handle structures and host helpers, shared
// by the host files of the library (api.cu, serve.cu).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "vsr_internal.cuh"

// The device-side status word of the current device (allocated and zeroed
// on first use).
int* status_word();

template <class Tp>
inline vsr_status dalloc(Tp** p, size_t n)
{
    *p = nullptr;
    if (n == 0) n = 1;
    if (cudaMalloc((void**)p, n * sizeof(Tp)) != cudaSuccess) {
        cudaGetLastError();
        *p = nullptr;
        return VSR_ERR_OOM;
    }
    return VSR_OK;
}

struct vsr_map_s {
    vsr_map_params p;  // effective parameters
    vsr_map_spec spec = {};  // the projection (kind VSR_MAP_UNIVERSAL with no distortion for vsr_make_map*)
    bool lens_grad = true;   // the lens gradient of vsr_raster_backward applies (undistorted Universal)
    float4* deriv = nullptr; // 2 float4 per pixel with VSR_MAP_DERIVATIVES
    float4* map = nullptr;
    Cone* tiles = nullptr;
    // tile geometry (every generation), and the tile index of the
    // triangle-major search, built for the current generation on first use
    // (vsr_raster_noalloc)
    TileIndex idx = {};
    bool idx_built = false;
    int tx = 0, ty = 0;
    uint64_t gen = 0;
};

// Status words in host memory that kernels raise errors in (mapped into the
// device's address space): zero between frames, read and cleared by the host
// once a frame's launches have completed.
struct HostStatus {
    int* host = nullptr;
    int* dev = nullptr;
    vsr_status alloc(int n)
    {
        if (cudaHostAlloc((void**)&host, sizeof(int) * (size_t)n, cudaHostAllocMapped) != cudaSuccess ||
            cudaHostGetDevicePointer((void**)&dev, host, 0) != cudaSuccess) {
            cudaGetLastError();
            release();
            return VSR_ERR_OOM;
        }
        for (int i = 0; i < n; ++i) host[i] = 0;
        return VSR_OK;
    }
    vsr_status take(int i = 0)
    {
        const int v = *(volatile int*)&host[i];
        *(volatile int*)&host[i] = 0;
        return (vsr_status)v;
    }
    void release()
    {
        if (host) cudaFreeHost(host);
        host = dev = nullptr;
    }
};

struct vsr_scene_s {
    // the status word of vsr_render_host's frames: an overflow of stored bins
    // renders the frame again, any other error is the call's result (first in
    // the handle, where the tests reach it to raise one)
    HostStatus host_status;
    int64_t T = 0;
    float cam[12] = {};  // camera of the current set-up
    int64_t T_alloc = 0;
    float4* rec = nullptr;
    uint64_t gen = 0;
    // bin workspace
    int ws_tiles = 0;
    // bins: tile u's at ids[offsets[u] .. ends[u]) (offsets[ntiles]: the total)
    uint32_t* offsets = nullptr;  // ntiles + 1
    uint32_t* ends = nullptr;     // ntiles
    uint32_t* bin_ctr = nullptr;  // BIN_CTR_WORDS, zero between binnings
    uint32_t* ids = nullptr;
    uint32_t cap = 0;
    TriGrid grid = {};  // the set-up's triangles by cap cell (T > GRID_DIRECT)
    // rasters without stored bins (launch_raster_walk): the split slots, the
    // pairs found per tile (ntiles), the generations of the last one, and
    // whether it came after the last binning
    WalkWork walk = {};
    uint32_t* tile_pairs = nullptr;
    uint64_t walked_map = 0, walked_scene = 0;
    bool walked_last = false;
    bool size_due = false;              // frames have walked since the bins were sized
    uint64_t sized_shape = 0;           // (tiles, T) the bins were last sized for,
    bool sized_pstep = false;           // with the wider caps of the pixel step
    uint32_t* h_total = nullptr;        // pinned: pair total of a recent binning
    uint32_t* h_total_dev = nullptr;    // its device address (the binning stores the total there)
    cudaEvent_t total_event = nullptr;  // completion of that copy
    bool total_pending = false;
    uint64_t total_map = 0, total_scene = 0;  // generations of the binning whose total it is
    int last_ntiles = 0;
    uint64_t binned_map = 0, binned_scene = 0;  // generations the current bins belong to
    RasterWork work = {};
    uint32_t work_tiles = 0;
    // host-path buffers (vsr_render_host)
    float* tris_dev = nullptr;
    int64_t tris_alloc = 0;
    void* out_dev = nullptr;  // id | depth | cov staging, 12 B per pixel
    size_t out_alloc = 0;
    // device status word of this scene's kernels: NULL = the per-device word
    // of vsr_last_device_status; the server gives its workspaces their own
    int* status = nullptr;
    // bins sized without waiting for the device when the map's shape changes
    // (the capacity of earlier binnings is kept and only grows): an owner
    // that renders a request again after a bin overflow (the server) needs
    // no synchronisation per new shape; everyone else's bins are sized for
    // each new shape and after frames that stored none (bin_scene)
    bool async_sizing = false;
    // vsr_render_host runs the set-up on a stream of the scene's own, beside
    // work the caller queued before the call that does not touch the scene
    // (a map update).  From its first call on, use_event is recorded after
    // every queued use of the scene's buffers, so that stream waits for
    // exactly those.
    cudaStream_t side = nullptr;
    cudaEvent_t use_event = nullptr;
    cudaEvent_t setup_event = nullptr;
    // vsr_render_host_async: the frame's completion, whether one is queued
    // and not yet waited for, and the map generation it was binned against
    cudaEvent_t host_done = nullptr;
    bool host_pending = false;
    uint64_t host_map_gen = 0;
};

inline int* scene_status(const vsr_scene_s* s) { return s->status ? s->status : status_word(); }

// A launch that walks the scene's grid follows on st: its workspace and
// bookkeeping; the first frame of a shape goes through stored bins first, so
// that they are sized (see raster_frame in api.cu).
vsr_status scene_walk_begin(vsr_map m, vsr_scene sc, cudaStream_t st);

// Whether work queued on st now is captured, to run when its graph is launched.
inline vsr_status stream_captures(cudaStream_t st, bool* captures)
{
    cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(st, &cs) != cudaSuccess) {
        cudaGetLastError();
        return VSR_ERR_CUDA;
    }
    *captures = cs != cudaStreamCaptureStatusNone;
    return VSR_OK;
}

// Note a use of the scene's buffers queued on st (see use_event).
inline vsr_status scene_used(vsr_scene_s* s, cudaStream_t st)
{
    if (!s->use_event) return VSR_OK;
    // uses inside a stream capture run when their graph is launched: the
    // caller orders those launches
    bool captures;
    if (stream_captures(st, &captures) != VSR_OK) return VSR_ERR_CUDA;
    if (!captures && cudaEventRecord(s->use_event, st) != cudaSuccess) {
        cudaGetLastError();
        return VSR_ERR_CUDA;
    }
    return VSR_OK;
}
