// Host side of tile_detect_kernel: which calls it takes, their layout in the
// resident buffers, and the launches.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstddef>
#include <cstring>

#include "vio_ctx.h"
#include "vio_tiles.cuh"

using namespace vio;

namespace {

static_assert(kConsumers == 256, "block size of both kernels");

// The kernels of a form for an NMS radius, by score.
template <int CAP>
struct TileKernel {
    void (*fn[3])(TileCall<CAP>);
    int tile_h, smem;
};

template <int SR, int R, int CAP>
constexpr TileKernel<CAP> make_kernel() {
    constexpr int TH = SR - 2 * R;
    using G = TileGeom<TH, R>;
    return {{tile_detect_kernel<TH, 0, R, CAP>, tile_detect_kernel<TH, 1, R, CAP>, tile_detect_kernel<TH, 2, R, CAP>},
            TH,
            G::BOXA + G::SR * G::SW * 2 + G::WARPS * G::QCAP * 2};
}

// Form 0: 32 score rows per tile, 4 per warp; form 1: 64 rows, 8 per warp.
template <int FORM>
const TileKernel<kTileCap[FORM]>& kernel_of(int radius) {
    constexpr int SR = FORM == 0 ? 32 : 64, CAP = kTileCap[FORM];
    static const TileKernel<CAP> k[4] = {make_kernel<SR, 1, CAP>(), make_kernel<SR, 2, CAP>(),
                                         make_kernel<SR, 3, CAP>(), make_kernel<SR, 4, CAP>()};
    return k[radius - 1];
}

template <int CAP>
void (*pyramid_of(int levels))(TileCall<CAP>) {
    switch (levels) {
        case 1: return tile_pyramid_kernel<1, CAP>;
        case 2: return tile_pyramid_kernel<2, CAP>;
        case 3: return tile_pyramid_kernel<3, CAP>;
        case 4: return tile_pyramid_kernel<4, CAP>;
        default: return tile_pyramid_kernel<5, CAP>;
    }
}

// Which calls are taken, by their tiles (of the form in question); us per call,
// three sets of frames in turn, the persistent three kernels -> these launches:
//   form 0, one launch, tiles of 30 rows at 3 levels
//                          752x480, 152 tiles: 20.3 -> 12.3; 1280x720, 354: 22.5 -> 12.3; 1920x1080,
//                          756: 26.1 -> 15.6; form 1 there 14.9, 16.4 and 18.5.  (The line is the last-tile
//                          decode's below; with a decode launch form 0 would still be ahead above it:
//                          8 frames 752x480, 1,216 tiles: 16.9, form 1 18.5.)
//   form 1, tiles of level 1 and 2 built from level 0
//                          16 mixed frames, 3 levels, 2,788 tiles: 56.7 -> 41.0; 32, 5,576 tiles:
//                          84.4 -> 77.7; 48, 8,364 tiles: 115.6 -> 113.3; 64, 11,152 tiles: 145.7 -> 150.0
//   form 1, levels in two launches (more than 3 levels, or unaligned frames)
//                          aligned: 4 4K frames, 4 levels, 6,000 tiles: 57.9 -> 57.2; 5, 7,500 tiles:
//                          69.7 -> 68.2; 6, 9,000 tiles: 79.4 -> 79.9
//                          unaligned: 24 of 1021x765 and less, 4 levels, 3,902 tiles: 83.6 -> 72.6; 48,
//                          7,777 tiles: 140.9 -> 128.0; 6 of 3001x2001, 3 levels, 6,852 tiles: 94.3 -> 89.4
//                          (8, 9,136 tiles, would be 117.7 -> 113.7)
//                          (aligned, 3 levels: 16, 32 and 48 mixed frames 47.2, 80.7 and 112.9)
//   form 1 after a pyramid kernel that uploads the frames
//                          host call, pinned frames apart, 3 levels: 8 mixed 90.2 -> 82.8; 16: 142.7 ->
//                          130.8; 32: 242.6 -> 235.6
// (a tile costs more here, 13.0 us per 1,000 of the mixed frames' against 10.6 in the
// pyramid and persistent kernels, whose loads run ahead; a call costs 8 to 22 us less to start).
constexpr int kFormTiles[2] = {800, 8000};      // aligned frames, at most 3 levels
constexpr int kTwoStepTiles[2] = {6000, 8000};  // others: aligned, unaligned
// A frame is decoded by the CTA of its last tile in a call of at most this many
// tiles; above it a decode launch is faster than a fence and a count per tile
// (8 1920x1080 frames, 3,040 tiles of 62 rows: 46.2 -> 43.2 us; 64 of 320x240, 1,088
// tiles: 22.6 and 22.5; one 752x480 frame in form 0: 12.3 either way).
constexpr int kLastTileDecodes = 800;

int tiles_of(const vio_dims& d, int k, int th) {
    return (((d.w >> k) + kTileW - 1) / kTileW) * (((d.h >> k) + th - 1) / th);
}

template <int FORM>
vio_status detect_form(vio_ctx* ctx, const uint8_t* const* lev0, const int* pitch0, const vio_dims* dims, int n,
                       int thresh, int arc, int cell, int levels, int4* const* outs, int32_t* counts, cudaStream_t s,
                       int tiles, bool two, const uint8_t* const* src, const int* src_pitch) {
    constexpr int CAP = kTileCap[FORM];
    const TileKernel<CAP>& kern = kernel_of<FORM>(ctx->cfg.nms_radius);
    const auto fn = kern.fn[ctx->cfg.score];
    TileCall<CAP> c;
    std::memset(&c, 0, offsetof(TileCall<CAP>, tiles) + sizeof(c.tiles[0]));
    size_t koff = 0, poff = ctx->group_pyr0;
    for (int i = 0; i < n; ++i) {
        FrameDesc& f = c.f[i];
        std::memset(&f, 0, sizeof(f));
        f.w = dims[i].w;
        f.h = dims[i].h;
        f.gw = (f.w + cell - 1) / cell;
        f.gh = (f.h + cell - 1) / cell;
        f.out = outs[i];
        f.lev[0] = const_cast<uint8_t*>(lev0[i]);
        f.pitch[0] = pitch0[i];
        if (src && src[i]) {
            f.src0 = src[i];
            f.src0_pitch = src_pitch[i];
        }
        koff += align_up((size_t)f.gw * f.gh, 16);
        for (int k = 1; k < levels; ++k) {
            f.pitch[k] = (int)align_up(f.w >> k, 128);
            poff += align_up((size_t)f.pitch[k] * (f.h >> k), 256);
        }
        for (int k = 0; k < levels; ++k) c.frame_tiles[i] += tiles_of(dims[i], k, kern.tile_h);
    }
    vio_status st;
    const void* keys0 = ctx->d_keys;
    const void* pyr0 = ctx->d_pyr;
    if ((st = grow(ctx, (void**)&ctx->d_keys, &ctx->keys_cap, koff * 8, &s)) != VIO_OK) return st;
    if ((st = grow(ctx, (void**)&ctx->d_pyr, &ctx->pyr_cap, std::max<size_t>(poff, 256))) != VIO_OK) return st;
    if (keys0 != ctx->d_keys || pyr0 != ctx->d_pyr) ctx->map_cache.clear();
    koff = 0;
    poff = ctx->group_pyr0;
    for (int i = 0; i < n; ++i) {
        FrameDesc& f = c.f[i];
        f.keys = ctx->d_keys + koff;
        koff += align_up((size_t)f.gw * f.gh, 16);
        for (int k = 1; k < levels; ++k) {
            f.lev[k] = ctx->d_pyr + poff;
            poff += align_up((size_t)f.pitch[k] * (f.h >> k), 256);
        }
    }
    c.thresh = thresh;
    c.arc = arc;
    c.n_frames = n;
    c.levels = levels;
    c.counts = counts;
    const bool decode_launch = src || two || tiles > kLastTileDecodes;
    c.done = decode_launch ? nullptr : ctx->d_done;
    c.sums = ctx->d_sums;
    c.status = ctx->d_status;
    for (int k = 0; k < levels; ++k) {
        const uint64_t d = (uint64_t)(cell >> k);
        c.cell_magic[k] = (uint32_t)(((1ull << 32) + d - 1) / d);
    }
    VIO_CK(follow_context(ctx, s));
    if (!ctx->tile_ready[FORM]) {
        VIO_CK(cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, kern.smem));
        ctx->tile_ready[FORM] = true;
    }
    const auto launch_grid = [&](void (*k)(TileCall<CAP>), int grid, int smem, bool dependent) -> vio_status {
        cudaLaunchAttribute pdl[1];
        pdl[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        pdl[0].val.programmaticStreamSerializationAllowed = 1;
        cudaLaunchConfig_t lc = {};
        lc.gridDim = dim3(grid);
        lc.blockDim = dim3(256);
        lc.dynamicSmemBytes = smem;
        lc.stream = s;
        lc.attrs = pdl;
        lc.numAttrs = dependent ? 1 : 0;
        VIO_CK(cudaLaunchKernelEx(&lc, k, c));
        return VIO_OK;
    };
    const auto launch_levels = [&](int top, int n_levels, bool dependent) -> vio_status {
        c.top = top;
        c.n_levels = n_levels;
        int acc = 0;
        c.tiles[0] = 0;
        for (int j = 0; j < n_levels; ++j)
            for (int i = 0; i < n; ++i) c.tiles[j * n + i + 1] = acc += tiles_of(dims[i], top - j, kern.tile_h);
        return launch_grid(fn, acc, kern.smem, dependent);
    };
    if (src) {
        for (int i = 0; i < n; ++i) c.tiles[i + 1] = c.tiles[i] + pyr_plan(c.f[i], levels);
        if ((st = launch_grid(pyramid_of<CAP>(levels), std::min(c.tiles[n], 8 * ctx->sm_count), 0, false)) != VIO_OK)
            return st;
        c.resident = levels - 1;
        if ((st = launch_levels(levels - 1, levels, true)) != VIO_OK) return st;
    } else if (!two) {
        if ((st = launch_levels(levels - 1, levels, false)) != VIO_OK) return st;
    } else {
        c.emit = std::min(levels - 1, 2);
        if ((st = launch_levels(0, 1, false)) != VIO_OK) return st;
        if (levels > 1) {
            c.resident = c.emit;
            c.emit = 0;
            if ((st = launch_levels(levels - 1, levels - 1, true)) != VIO_OK) return st;
        }
    }
    if (decode_launch) {
        c.tiles[0] = 0;
        for (int i = 0; i < n; ++i) c.tiles[i + 1] = c.tiles[i] + (c.f[i].gw * c.f[i].gh + 255) / 256;
        if ((st = launch_grid(tile_decode_kernel<CAP>, c.tiles[n], 0, true)) != VIO_OK) return st;
    }
    VIO_CK(mark_last(ctx, s));
    remember_levels(ctx, c.f, dims, n, levels);
    ctx->last_variant = ctx->default_variant;
    ctx->last_ctas = 0;
    ctx->last_tile_h = kern.tile_h;
    ctx->last_cell = cell;
    return VIO_OK;
}

}  // namespace

namespace vio {

vio_status detect_tiles(vio_ctx* ctx, const uint8_t* const* lev0, const int* pitch0, const vio_dims* dims, int n,
                        int thresh, int arc, int cell, int levels, int4* const* outs, int32_t* counts, cudaStream_t s,
                        bool* done, const uint8_t* const* src, const int* src_pitch) {
    *done = false;
    // a pinned or tuned launch shape and stage times ask for the three kernels
    if (n > kTileCap[1] || ctx->cfg.profile || ctx->cfg.autotune || ctx->pinned_variant >= 0) return VIO_OK;
    // So does a stream that is being captured: their call block keeps a detection
    // out of a graph, whose later launches would use resident buffers that may have
    // been given back (vio_detect_noalloc is the call to capture).
    cudaStreamCaptureStatus capture = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(s, &capture) != cudaSuccess || capture != cudaStreamCaptureStatusNone) {
        cudaGetLastError();
        return VIO_OK;
    }
    int tiles[2] = {0, 0};
    const int th[2] = {kernel_of<0>(ctx->cfg.nms_radius).tile_h, kernel_of<1>(ctx->cfg.nms_radius).tile_h};
    bool aligned = true;
    for (int i = 0; i < n; ++i) {
        aligned &= (((uintptr_t)lev0[i] | (uintptr_t)pitch0[i]) & 15) == 0;
        for (int k = 0; k < levels; ++k)
            for (int f = 0; f < 2; ++f) tiles[f] += tiles_of(dims[i], k, th[f]);
    }
    if (src) {
        if (tiles[1] > kFormTiles[1]) return VIO_OK;
        *done = true;
        return detect_form<1>(ctx, lev0, pitch0, dims, n, thresh, arc, cell, levels, outs, counts, s, tiles[1], false,
                              src, src_pitch);
    }
    const bool one = levels <= 3 && aligned;
    if (one && n <= kTileCap[0] && tiles[0] <= kFormTiles[0]) {
        *done = true;
        return detect_form<0>(ctx, lev0, pitch0, dims, n, thresh, arc, cell, levels, outs, counts, s, tiles[0], false,
                              nullptr, nullptr);
    }
    if (tiles[1] <= (one ? kFormTiles[1] : kTwoStepTiles[aligned ? 0 : 1])) {
        *done = true;
        return detect_form<1>(ctx, lev0, pitch0, dims, n, thresh, arc, cell, levels, outs, counts, s, tiles[1], !one,
                              nullptr, nullptr);
    }
    return VIO_OK;
}

}  // namespace vio
