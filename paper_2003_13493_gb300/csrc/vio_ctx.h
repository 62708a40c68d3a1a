// Internal: the context object behind include/vio.h and the host helpers the
// runtime's translation units share (resident buffers, error recording).
#pragma once
#include <cuda.h>
#include <cuda_runtime.h>
#include <nvtx3/nvToolsExt.h>

#include <algorithm>
#include <array>
#include <string>
#include <unordered_map>
#include <vector>

#include "../../include/vio.h"
#include "vio_kernels.cuh"

namespace vio {

inline size_t align_up(size_t v, size_t a) { return (v + a - 1) / a * a; }

constexpr int kTileCap[2] = {8, 64};  // frames of the two forms of tile_detect_kernel
// d_counter: the work counter (16 bytes), then d_sums and d_done
constexpr size_t kCounterBytes = 16 + (sizeof(uint64_t) + sizeof(int32_t)) * kTileCap[1];
constexpr int kMaxCtasPerSm = 4;  // the detect kernels' launch bounds

using EncodeTiledFn = CUresult (*)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                   const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                   CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

struct ShapeKey {
    std::vector<int32_t> v;
    bool operator==(const ShapeKey& o) const { return v == o.v; }
};
struct ShapeHash {
    size_t operator()(const ShapeKey& k) const {
        size_t h = 1469598103934665603ull;
        for (int32_t x : k.v) h = (h ^ (uint32_t)x) * 1099511628211ull;
        return h;
    }
};

struct MapKey {
    uintptr_t ptr;
    int32_t w, h, pitch, bw, bh;
    bool operator==(const MapKey& o) const {
        return ptr == o.ptr && w == o.w && h == o.h && pitch == o.pitch && bw == o.bw && bh == o.bh;
    }
};
struct MapHash {
    size_t operator()(const MapKey& k) const {
        return std::hash<uintptr_t>()(k.ptr) ^ ((size_t)k.w * 73856093u) ^ ((size_t)k.h * 19349663u) ^
               ((size_t)k.pitch * 83492791u) ^ ((size_t)k.bw << 40) ^ ((size_t)k.bh << 52);
    }
};


// A named range on the profiler's timeline for the duration of a scope (NVTX;
// free when no profiler is attached).
struct NvtxRange {
    explicit NvtxRange(const char* name) { nvtxRangePushA(name); }
    ~NvtxRange() { nvtxRangePop(); }
    NvtxRange(const NvtxRange&) = delete;
    NvtxRange& operator=(const NvtxRange&) = delete;
};

// One input slot of vio_detect_host_async: frames of one call in flight.
struct HostSlot {
    uint8_t* d_in = nullptr;
    size_t in_cap = 0;
    int32_t* d_counts = nullptr;
    size_t counts_cap = 0;
    cudaEvent_t done = nullptr;  // after the kernels that read the slot
    bool used = false;
};
constexpr int kHostSlots = 3;

constexpr int kMaxGroups = 8;  // groups of a host call (vio_detect_host)

// Resident state of the feature tracker (vio_track).
struct TrackState {
    uint8_t* d_pyr = nullptr;    // levels 1..L-1 of both frames of every pair
    size_t pyr_cap = 0;
    uint8_t* d_in = nullptr;     // level-0 copies of frames that are not 16-byte aligned
    size_t in_cap = 0;
    cudaEvent_t done_ev = nullptr;  // after the last call's kernels: the next call's stream waits on it
    bool have_done = false;
};

}  // namespace vio

// ---------------------------------------------------------------------------
// Context
// ---------------------------------------------------------------------------
struct vio_ctx {
    using EncodeTiledFn = vio::EncodeTiledFn;
    using ShapeKey = vio::ShapeKey;
    using ShapeHash = vio::ShapeHash;
    using MapKey = vio::MapKey;
    using MapHash = vio::MapHash;
    vio_config cfg{};
    int sm_count = 0;
    std::string err;
    EncodeTiledFn encode = nullptr;
    size_t call_cap = 0;

    // resident device buffers
    uint8_t* d_call = nullptr;          // the current call block
    int32_t* d_counter = nullptr;       // work-item counter of the fused kernel
    // in the same allocation, zero when idle (see TileCall)
    uint64_t* d_sums = nullptr;
    int32_t* d_done = nullptr;
    uint64_t* d_keys = nullptr;         // packed cell keys, zero when idle
    size_t keys_cap = 0;
    uint8_t* d_pyr = nullptr;           // pyramid levels 1..L-1 of every frame
    size_t pyr_cap = 0;
    uint8_t* d_in = nullptr;            // staged level-0 frames (host path / unaligned frames)
    size_t in_cap = 0;
    int4* d_cells = nullptr;            // host path: device-side output records + counts
    size_t cells_cap = 0;
    size_t bytes_in_use = 0;

    // host
    uint32_t* h_status = nullptr;       // pinned, device-mapped status word
    uint32_t* d_status = nullptr;
    uint8_t* h_stage = nullptr;         // pinned ring of call blocks
    int ring = 8, ring_pos = 0;
    std::vector<cudaEvent_t> ring_ev;
    uint8_t* h_out = nullptr;           // pinned host-path output staging
    size_t h_out_cap = 0;

    cudaEvent_t stage_ev[4] = {nullptr, nullptr, nullptr, nullptr};
    cudaStream_t capture_stream = nullptr;  // the context's own: graphs are captured on it
    cudaEvent_t last_ev = nullptr;
    cudaStream_t last_stream = nullptr;
    bool have_last = false;
    // the latest clear of a buffer, while no call has followed it (clear_buffer)
    cudaEvent_t clear_ev = nullptr;
    bool clear_pending = false;
    bool counters_clear = false;            // d_counter, d_sums and d_done have been cleared

    // one graph per (variant, levels, CTAs per SM): every batch shape replays
    // it; CTAs per SM 0 = as many as fit
    cudaGraphExec_t graphs[8][vio::kMaxLevels + 1][vio::kMaxCtasPerSm + 1] = {};
    int occ_fused[8] = {};                 // CTAs per SM that fit, per variant
    int grid_sweep = 0;
    bool tile_ready[2] = {};               // attributes of the two forms of tile_detect_kernel are set
    int default_variant = 0;               // first variant of the context's NMS radius
    struct TuneChoice {
        int variant, ctas, cell;
    };
    std::unordered_map<ShapeKey, TuneChoice, ShapeHash> tuned;  // batch shape -> choice
    std::vector<vio_tuning> tune_log;      // the alternatives the last tuning run timed
    std::vector<float> tune_log_ms;
    std::unordered_map<MapKey, CUtensorMap, MapHash> map_cache;
    int pinned_variant = -1;
    int pinned_ctas = 0;
    int last_variant = 0;
    int last_ctas = 0;                     // CTAs per SM of the last launch (resolved); 0: the tile kernel's
    int last_tile_h = 0;                   // tile height of the tile kernel's last launch; 0: the variant's
    int last_cell = 0;                     // cell size of the last detection
    // levels of the most recent detection call, for vio_copy_level
    std::vector<std::array<const uint8_t*, vio::kMaxLevels>> last_lev;
    std::vector<std::array<int, vio::kMaxLevels>> last_pitch;
    std::vector<vio_dims> last_dims;
    int last_levels = 0;
    // a call detected in groups of frames: where this group's pyramid begins in
    // d_pyr, and whether it follows an earlier group, so that the levels of the
    // whole call stay readable
    size_t group_pyr0 = 0;
    bool group_follows = false;
    cudaStream_t copy_stream = nullptr;    // uploads of a grouped call
    cudaEvent_t group_ev[1 + vio::kMaxGroups] = {};  // the call's start, then each group's upload
    vio::TrackState track;
    vio::HostSlot hslots[vio::kHostSlots];
    int hslot_pos = 0;

    void drop_graphs() {
        for (auto& row : graphs)
            for (auto& shape : row)
                for (auto& g : shape)
                    if (g) {
                        cudaGraphExecDestroy(g);
                        g = nullptr;
                    }
    }
};

namespace vio {

inline vio_status fail(vio_ctx* c, vio_status s, const std::string& msg) {
    if (c) c->err = msg;
    return s;
}

#define VIO_CK(call)                                                                          \
    do {                                                                                      \
        cudaError_t e_ = (call);                                                              \
        if (e_ != cudaSuccess) {                                                              \
            return fail(ctx, e_ == cudaErrorMemoryAllocation ? VIO_ERR_OOM : VIO_ERR_CUDA,    \
                        std::string(#call) + ": " + cudaGetErrorString(e_));                  \
        }                                                                                     \
    } while (0)

// Clears device memory for the call on `s`, on that stream: the default stream is
// not ordered with a caller's non-blocking one.  A later call on another stream
// waits for the clear (follow_context).  A stream that is being captured would
// only record it: there it is done at once.
inline cudaError_t clear_buffer(vio_ctx* ctx, void* p, size_t bytes, cudaStream_t s) {
    cudaStreamCaptureStatus capture = cudaStreamCaptureStatusNone;
    cudaError_t e = cudaStreamIsCapturing(s, &capture);
    if (e != cudaSuccess) return e;
    if (capture != cudaStreamCaptureStatusNone) {
        e = cudaMemsetAsync(p, 0, bytes, ctx->capture_stream);
        return e != cudaSuccess ? e : cudaStreamSynchronize(ctx->capture_stream);
    }
    if (ctx->clear_pending) e = cudaStreamWaitEvent(s, ctx->clear_ev, 0);
    if (e == cudaSuccess) e = cudaMemsetAsync(p, 0, bytes, s);
    if (e == cudaSuccess) e = cudaEventRecord(ctx->clear_ev, s);
    if (e != cudaSuccess) return e;
    ctx->clear_pending = true;
    return e;
}

// Orders `s` after the context's work on another stream and after its clears;
// to be followed by mark_last once the call's work is enqueued.  (A call that fails
// in between leaves its clears pending for the next one.)
inline cudaError_t follow_context(vio_ctx* ctx, cudaStream_t s) {
    cudaError_t e = cudaSuccess;
    if (ctx->have_last && ctx->last_stream != s) e = cudaStreamWaitEvent(s, ctx->last_ev, 0);
    if (e == cudaSuccess && ctx->clear_pending) e = cudaStreamWaitEvent(s, ctx->clear_ev, 0);
    if (e == cudaSuccess && !ctx->counters_clear) {  // the context's first call
        e = clear_buffer(ctx, ctx->d_counter, kCounterBytes, s);
        ctx->counters_clear = e == cudaSuccess;
    }
    return e;
}

inline cudaError_t mark_last(vio_ctx* ctx, cudaStream_t s) {
    const cudaError_t e = cudaEventRecord(ctx->last_ev, s);
    if (e != cudaSuccess) return e;
    ctx->last_stream = s;
    ctx->have_last = true;
    ctx->clear_pending = false;  // last_ev follows them
    return e;
}

// Grows a resident buffer to `need` bytes.  Growing waits for the device
// (the old buffer may still be in use), so buffers grow geometrically.
// With clear_for the new buffer is zero for calls that follow_context, the first
// of them on that stream.
inline vio_status grow(vio_ctx* ctx, void** p, size_t* cap, size_t need, const cudaStream_t* clear_for = nullptr) {
    if (need <= *cap && *p) return VIO_OK;
    size_t want = std::max(need, *cap + *cap / 2);
    const size_t budget = ctx->cfg.mem_budget_bytes;
    if (budget && ctx->bytes_in_use - *cap + want > budget) {
        want = need;
        if (ctx->bytes_in_use - *cap + want > budget)
            return fail(ctx, VIO_ERR_OOM, "context memory budget exceeded");
    }
    if (*p) {
        VIO_CK(cudaDeviceSynchronize());
        VIO_CK(cudaFree(*p));
        ctx->bytes_in_use -= *cap;
        *p = nullptr;
        *cap = 0;
    }
    VIO_CK(cudaMalloc(p, want));
    if (clear_for) VIO_CK(clear_buffer(ctx, *p, want, *clear_for));
    *cap = want;
    ctx->bytes_in_use += want;
    return VIO_OK;
}

}  // namespace vio

namespace vio {
// Remembers the levels of a detection for vio_copy_level (after those of the
// call's earlier groups).
inline void remember_levels(vio_ctx* ctx, const FrameDesc* f, const vio_dims* dims, int n, int levels) {
    if (!ctx->group_follows) {
        ctx->last_dims.clear();
        ctx->last_lev.clear();
        ctx->last_pitch.clear();
    }
    ctx->last_levels = levels;
    ctx->last_dims.insert(ctx->last_dims.end(), dims, dims + n);
    for (int i = 0; i < n; ++i) {
        std::array<const uint8_t*, kMaxLevels> lev{};
        std::array<int, kMaxLevels> pitch{};
        for (int k = 0; k < levels; ++k) {
            lev[k] = f[i].lev[k];
            pitch[k] = f[i].pitch[k];
        }
        ctx->last_lev.push_back(lev);
        ctx->last_pitch.push_back(pitch);
    }
}

// Frees the tracker's resident buffers (vio_destroy).
void track_release(vio_ctx* ctx);
}  // namespace vio

namespace vio {
// Detects frames that live in host memory, asynchronously on s: pinned frames
// are uploaded by the pyramid kernel through their device mapping, others by
// the copy engines into the context's staging.  outs[i] may be device memory
// or the device mapping of pinned host memory; d_counts is device memory or
// nullptr.  may_group: a large upload may be detected in groups of frames, the
// copies of one beside the kernels of another.  Arguments are checked by the
// caller.
vio_status detect_from_host(vio_ctx* ctx, const uint8_t* const* host_frames, const vio_dims* dims, int n, int thresh,
                            int arc, int cell, int levels, int4* const* outs, int32_t* d_counts, cudaStream_t s,
                            bool may_group = false);
// Detects with tile_detect_kernel (vio_tiles.cuh) when the call is one that it
// takes, and sets *done then.  Frames of any alignment, in device memory; with
// src, frames whose src[i] is not nullptr (row pitch src_pitch[i]) are first
// copied to lev0[i] by the pyramid kernel, as by vio_api.cu's Upload.
vio_status detect_tiles(vio_ctx* ctx, const uint8_t* const* lev0, const int* pitch0, const vio_dims* dims, int n,
                        int thresh, int arc, int cell, int levels, int4* const* outs, int32_t* counts, cudaStream_t s,
                        bool* done, const uint8_t* const* src = nullptr, const int* src_pitch = nullptr);
// Device address of pinned host memory, else nullptr.
const void* host_device_alias(const void* host);
}  // namespace vio
