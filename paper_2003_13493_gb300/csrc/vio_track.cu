// Host side of the feature tracker behind vio_track (Section II-E): argument
// checks, the resident pyramid of both frames of every pair (built by the
// detector's pyramid code) and the launches.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <vector>

#include "../../include/vio.h"
#include "vio_ctx.h"
#include "vio_track.cuh"

using namespace vio;

namespace {

// Launches of up to PAIRS pairs.
template <int PAIRS>
void (*track_pyr_fn(int levels))(TrackCall<PAIRS>) {
    switch (levels) {
        case 1: return track_pyramid_kernel<1, PAIRS>;
        case 2: return track_pyramid_kernel<2, PAIRS>;
        case 3: return track_pyramid_kernel<3, PAIRS>;
        case 4: return track_pyramid_kernel<4, PAIRS>;
        default: return track_pyramid_kernel<5, PAIRS>;
    }
}

bool valid_params(const vio_track_params& p) {
    return p.levels >= 1 && p.levels <= kMaxLevels && (p.patch_fine == 8 || p.patch_fine == 16) &&
           (p.patch_coarse == 8 || p.patch_coarse == 16) && p.max_iters >= 1 && p.max_iters <= 100 &&
           std::isfinite(p.min_update) && p.min_update >= 0.f && p.model >= 0 && p.model <= 3;
}

}  // namespace

namespace vio {

void track_release(vio_ctx* ctx) {
    TrackState& t = ctx->track;
    if (t.d_pyr) cudaFree(t.d_pyr);
    if (t.d_in) cudaFree(t.d_in);
    if (t.done_ev) cudaEventDestroy(t.done_ev);
    ctx->bytes_in_use -= t.pyr_cap + t.in_cap;
    t = TrackState{};
}

}  // namespace vio

namespace {

// Frame f of a call (2i: pair i's previous frame, 2i + 1 its next) and its place
// in the resident buffers.
struct TrackFrame {
    const uint8_t* src;
    size_t in_off;                 // (size_t)-1: read in place
    size_t lev_off[kMaxLevels];
};

// Pairs [first, first + n) in one launch.
template <int PAIRS>
vio_status track_launch(vio_ctx* ctx, const vio_track_params& p, const TrackFrame* frames, const vio_dims* dims,
                        int first, int n, const void* const* pts, const int* n_pts, vio_track_result* const* out,
                        bool cells_in, cudaStream_t s) {
    TrackState& T = ctx->track;
    const int L = p.levels;
    TrackCall<PAIRS> c;
    c.levels = L;
    c.patch_fine = p.patch_fine;
    c.patch_coarse = p.patch_coarse;
    c.max_iters = p.max_iters;
    c.min_update = p.min_update;
    c.model = p.model;
    c.n_pairs = n;
    c.cells_in = cells_in ? 1 : 0;
    c.blocks[0] = 0;
    c.prefix[0] = 0;
    for (int i = 0; i < n; ++i) {
        const vio_dims& d = dims[first + i];
        c.pairs[i].pts = reinterpret_cast<const float*>(pts[first + i]);
        c.pairs[i].out = reinterpret_cast<float*>(out[first + i]);
        c.prefix[i + 1] = c.prefix[i] + n_pts[first + i];
        for (int e = 0; e < 2; ++e) {
            const TrackFrame& tf = frames[2 * (first + i) + e];
            FrameDesc& fd = c.f[2 * i + e];
            std::memset(&fd, 0, sizeof(fd));
            fd.w = d.w;
            fd.h = d.h;
            if (tf.in_off != (size_t)-1) {
                // copied by the pyramid kernel as it reads it
                fd.src0 = tf.src;
                fd.src0_pitch = d.pitch;
                fd.lev[0] = T.d_in + tf.in_off;
                fd.pitch[0] = (int)align_up(d.w, 16);
            } else {
                fd.lev[0] = const_cast<uint8_t*>(tf.src);
                fd.pitch[0] = d.pitch;
            }
            for (int k = 1; k < L; ++k) {
                fd.lev[k] = T.d_pyr + tf.lev_off[k];
                fd.pitch[k] = (int)align_up(d.w >> k, 128);
            }
            c.blocks[2 * i + e + 1] = c.blocks[2 * i + e] + pyr_plan(fd, L);
        }
    }
    c.n_features = c.prefix[n];
    c.n_pyr_blocks = c.blocks[2 * n];
    if (c.n_features == 0) return VIO_OK;
    if (c.n_pyr_blocks > 0) {
        // the kernel strides over its grid
        const int grid = std::min(c.n_pyr_blocks, ctx->sm_count * 8);
        track_pyr_fn<PAIRS>(L)<<<grid, 256, 0, s>>>(c);
        VIO_CK(cudaGetLastError());
    }
    // few features are spread over the SMs, a warp or two each: a CTA's warps
    // share an SM's pipes and its L1
    const int warps = std::min(kTrackWarps, std::max(1, (c.n_features + ctx->sm_count - 1) / ctx->sm_count));
    cudaLaunchAttribute pdl[1];
    pdl[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    pdl[0].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t lc = {};
    lc.gridDim = dim3((c.n_features + warps - 1) / warps);
    lc.blockDim = dim3(warps * 32);
    lc.stream = s;
    lc.attrs = pdl;
    lc.numAttrs = c.n_pyr_blocks > 0 ? 1 : 0;
    VIO_CK(cudaLaunchKernelEx(&lc, track_kernel<PAIRS>, c));
    return VIO_OK;
}

}  // namespace

extern "C" {

void vio_track_params_default(vio_track_params* p) {
    if (!p) return;
    std::memset(p, 0, sizeof(*p));
    p->levels = 3;
    p->patch_fine = 16;
    p->patch_coarse = 8;
    p->max_iters = 30;
    p->min_update = 0.01f;
    p->model = VIO_TRACK_GAIN | VIO_TRACK_OFFSET;
}

namespace {

vio_status track_impl(vio_ctx* ctx, const uint8_t* const* prev, const uint8_t* const* next, const vio_dims* dims,
                      int n_pairs, const void* const* pts, const int* n_pts, const vio_track_params* params,
                      vio_track_result* const* out, vio_stream stream, bool cells_in) {
    if (!ctx) return VIO_ERR_INVALID_ARG;
    vio_track_params p;
    if (params) p = *params; else vio_track_params_default(&p);
    if (!valid_params(p)) return fail(ctx, VIO_ERR_INVALID_ARG, "tracker parameters out of range");
    if (n_pairs < 0 || n_pairs > ctx->cfg.max_frames)
        return fail(ctx, VIO_ERR_INVALID_ARG, "n_pairs must be in 0..max_frames");
    if (n_pairs == 0) return VIO_OK;
    if (!prev || !next || !dims || !pts || !n_pts || !out)
        return fail(ctx, VIO_ERR_INVALID_ARG, "NULL argument");
    const int L = p.levels;
    long long total = 0;
    for (int i = 0; i < n_pairs; ++i) {
        const vio_dims& d = dims[i];
        if (d.w < 7 || d.h < 7 || (d.w >> (L - 1)) < 7 || (d.h >> (L - 1)) < 7 || d.pitch < d.w ||
            (long long)d.w * d.h >= (1ll << 28))
            return fail(ctx, VIO_ERR_INVALID_ARG, "frame size out of range for the pyramid");
        if (!prev[i] || !next[i]) return fail(ctx, VIO_ERR_INVALID_ARG, "NULL frame");
        if (n_pts[i] < 0) return fail(ctx, VIO_ERR_INVALID_ARG, "negative feature count");
        if (n_pts[i] > 0 && (!pts[i] || !out[i])) return fail(ctx, VIO_ERR_INVALID_ARG, "NULL feature array");
        total += n_pts[i];
    }
    if (total == 0) return VIO_OK;
    if (total > (1ll << 24)) return fail(ctx, VIO_ERR_INVALID_ARG, "more than 2^24 features in one call");
    VIO_CK(cudaSetDevice(ctx->cfg.device));
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    TrackState& T = ctx->track;

    // resident layout: staged level-0 copies and levels 1..L-1 of every frame
    std::vector<TrackFrame> frames(2 * n_pairs);
    size_t ioff = 0, poff = 0;
    for (int f = 0; f < 2 * n_pairs; ++f) {
        const vio_dims& d = dims[f >> 1];
        TrackFrame& tf = frames[f];
        tf.src = (f & 1) ? next[f >> 1] : prev[f >> 1];
        tf.in_off = (size_t)-1;
        if (((uintptr_t)tf.src & 15) || (d.pitch & 15)) {
            tf.in_off = ioff;
            ioff += align_up(align_up(d.w, 16) * (size_t)d.h, 256);
        }
        for (int k = 1; k < L; ++k) {
            tf.lev_off[k] = poff;
            poff += align_up(align_up(d.w >> k, 128) * (size_t)(d.h >> k), 256);
        }
    }
    vio_status st;
    if (!T.done_ev) VIO_CK(cudaEventCreateWithFlags(&T.done_ev, cudaEventDisableTiming));
    // the previous call's kernels read the device buffers this call rewrites
    if (T.have_done) VIO_CK(cudaStreamWaitEvent(s, T.done_ev, 0));
    if ((st = grow(ctx, (void**)&T.d_in, &T.in_cap, std::max<size_t>(ioff, 256))) != VIO_OK) return st;
    if ((st = grow(ctx, (void**)&T.d_pyr, &T.pyr_cap, std::max<size_t>(poff, 256))) != VIO_OK) return st;
    if (n_pairs <= 8) {
        if ((st = track_launch<8>(ctx, p, frames.data(), dims, 0, n_pairs, pts, n_pts, out, cells_in, s)) != VIO_OK)
            return st;
    } else {
        for (int first = 0; first < n_pairs; first += 64)
            if ((st = track_launch<64>(ctx, p, frames.data(), dims, first, std::min(64, n_pairs - first), pts, n_pts,
                                       out, cells_in, s)) != VIO_OK)
                return st;
    }
    VIO_CK(cudaEventRecord(T.done_ev, s));
    T.have_done = true;
    return VIO_OK;
}

}  // namespace

vio_status vio_track(vio_ctx* ctx, const uint8_t* const* prev, const uint8_t* const* next, const vio_dims* dims,
                     int n_pairs, const float* const* pts, const int* n_pts, const vio_track_params* params,
                     vio_track_result* const* out, vio_stream stream) {
    NvtxRange nvtx("vio_track");
    return track_impl(ctx, prev, next, dims, n_pairs, reinterpret_cast<const void* const*>(pts), n_pts, params, out,
                      stream, false);
}

vio_status vio_track_cells(vio_ctx* ctx, const uint8_t* const* prev, const uint8_t* const* next,
                           const vio_dims* dims, int n_pairs, const vio_feature* const* cells, const int* n_cells,
                           const vio_track_params* params, vio_track_result* const* out, vio_stream stream) {
    NvtxRange nvtx("vio_track_cells");
    return track_impl(ctx, prev, next, dims, n_pairs, reinterpret_cast<const void* const*>(cells), n_cells, params,
                      out, stream, true);
}

}  // extern "C"
