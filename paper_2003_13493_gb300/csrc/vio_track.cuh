// Device code of the feature tracker (Section II-E, Eqs. 2-6): one warp per
// feature, patch sums reduced with an xor butterfly of warp shuffles, fp32.
#pragma once
#include <stdint.h>

#include "vio_kernels.cuh"

namespace vio {

struct TrackPair {
    const float* pts;   // 2 floats per feature, or 4 int32 per detector record (cells_in)
    float* out;         // 8 words per feature (vio_track_result)
};

// What a launch needs, passed as the parameter of the pyramid and the track
// kernel (frame 2i is pair i's previous frame, 2i+1 its next frame): there is no
// call block to upload, and a feature's chain of loads starts at its position.
// PAIRS: pairs it holds.
template <int PAIRS>
struct TrackCall {
    int32_t levels, patch_fine, patch_coarse, max_iters;
    float min_update;
    int32_t model, n_pairs, n_features;
    int32_t cells_in;            // 1: the inputs are detector records (x, y, level, score)
    int32_t n_pyr_blocks;
    int32_t prefix[PAIRS + 1];   // prefix sums of the features per pair
    int32_t blocks[2 * PAIRS + 1];  // prefix sums of the pyramid blocks per frame
    TrackPair pairs[PAIRS];
    FrameDesc f[2 * PAIRS];
};
static_assert(sizeof(TrackCall<64>) <= 32000, "kernel parameter");

constexpr int kTrackWarps = 8;  // most features per CTA
constexpr int kTrackMaxGrid = 18 * 18;
// A window of an image in shared memory: 25 rows of 32 columns from a column
// that is a multiple of 8, three or four 8-byte loads per lane.
constexpr int kWinRows = 25, kWinCols = 32, kWinUnits = kWinRows * kWinCols / 8, kWinLoads = (kWinUnits + 31) / 32;

__device__ __forceinline__ bool inside(float x, float y, int w, int h) {
    return x >= 0.f && y >= 0.f && x <= (float)(w - 2) && y <= (float)(h - 2);
}

// Lane that holds value k of n after warp_sums' exchange steps.
__host__ __device__ constexpr int sum_lane(int k, int n) {
    int lane = 0;
    for (int m = 16; m > 0; m >>= 1) {
        const int half = (n + 1) / 2;
        if (k >= half) {
            lane |= m;
            k -= half;
        }
        n = half;
    }
    return lane;
}

// Sums of N values over the warp; every lane ends with the same bits, those of
// an xor butterfly (masks 16, 8, .. 1) per value: each step adds the same two
// partial sums, but a lane hands over the values that its partner goes on with
// and keeps the others, so N = 5 takes 8 + 5 shuffles instead of 25 and N = 9
// takes 12 + 9 instead of 45.
template <int N>
__device__ __forceinline__ void warp_sums(float (&v)[N], int lane) {
    constexpr uint32_t kAll = 0xFFFFFFFFu;
    float t[N];
#pragma unroll
    for (int i = 0; i < N; ++i) t[i] = v[i];
    int n = N;
#pragma unroll
    for (int m = 16; m > 0; m >>= 1) {
        const int half = (n + 1) / 2;
        const bool up = lane & m;
#pragma unroll
        for (int i = 0; i < (N + 1) / 2; ++i) {
            if (i + half < n) {
                const float keep = up ? t[i + half] : t[i], send = up ? t[i] : t[i + half];
                t[i] = keep + __shfl_xor_sync(kAll, send, m);
            } else if (i < half) {
                t[i] += __shfl_xor_sync(kAll, t[i], m);
            }
        }
        n = half;
    }
#pragma unroll
    for (int i = 0; i < N; ++i) v[i] = __shfl_sync(kAll, t[0], sum_lane(i, N));
}

// Cholesky factor of the symmetric 4x4 A (lower triangle used) in place on
// every lane, and the reciprocals of its diagonal; false when a pivot is not
// positive.  Lane r & 3 divides for row r, so a column takes one division and
// the reciprocals one, instead of ten in a chain; the values are those of the
// plain factorisation.
__device__ __forceinline__ bool cholesky4(float (&A)[4][4], float (&inv)[4], int lane) {
    constexpr uint32_t kAll = 0xFFFFFFFFu;
    const int r = lane & 3;
    float diag = 1.f;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        float d = A[j][j];
#pragma unroll
        for (int k = 0; k < j; ++k) d = fmaf(-A[j][k], A[j][k], d);
        if (!(d > 0.f)) return false;
        const float l = sqrtf(d);
        A[j][j] = l;
        if (r == j) diag = l;
        if (j == 3) break;
        float s = 1.f;
#pragma unroll
        for (int i = j + 1; i < 4; ++i) {
            float si = A[i][j];
#pragma unroll
            for (int k = 0; k < j; ++k) si = fmaf(-A[i][k], A[j][k], si);
            if (r == i) s = si;
        }
        const float q = s / l;
#pragma unroll
        for (int i = j + 1; i < 4; ++i) A[i][j] = __shfl_sync(kAll, q, i);
    }
    const float q = 1.f / diag;
#pragma unroll
    for (int i = 0; i < 4; ++i) inv[i] = __shfl_sync(kAll, q, i);
    return true;
}

// Solves L L^T x = b with the factor from cholesky4 and the reciprocals of
// its diagonal (computed once per level: the iterations then multiply).
__device__ __forceinline__ void chol_solve4(const float (&L)[4][4], const float (&inv)[4], const float (&b)[4],
                                            float (&x)[4]) {
    float y[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        float s = b[i];
#pragma unroll
        for (int k = 0; k < i; ++k) s -= L[i][k] * y[k];
        y[i] = s * inv[i];
    }
#pragma unroll
    for (int i = 3; i >= 0; --i) {
        float s = y[i];
#pragma unroll
        for (int k = i + 1; k < 4; ++k) s -= L[k][i] * x[k];
        x[i] = s * inv[i];
    }
}

struct TrackLevel {
    const uint8_t* prev;
    const uint8_t* next;
    int pitch_prev, pitch_next, w, h;
};

// A window's place in a w x h image, so that it holds the pixels c0 - 1 ..
// c0 + need, r0 - 1 .. r0 + need that the image has: central, its column a
// multiple of 8, but not beyond the image (an image smaller than the window
// fills a part of it).  (The levels are written by the kernel before this one,
// which may run when this one starts, so they are read by plain loads and not as
// read-only data.)
struct Window {
    int x, y, w, h;
    __device__ __forceinline__ static Window around(int c0, int r0, int need, int w, int h) {
        Window v;
        v.x = max(0, c0 - max(1, (kWinCols - 8 - need) / 2)) & ~7;
        if (v.x + kWinCols > w) {
            // the last whole place, if that reaches far enough, or the border
            v.x = max(0, w - kWinCols);
            const int a = v.x & ~7;
            if (min(c0 + need, w - 1) < a + kWinCols) v.x = a;
        }
        v.y = min(max(0, r0 - max(1, (kWinRows - need) / 2)), max(0, h - kWinRows));
        v.w = w;
        v.h = h;
        return v;
    }
    __device__ __forceinline__ bool holds(int c0, int r0, int need) const {
        return max(0, c0 - 1) >= x && min(c0 + need, w - 1) < x + kWinCols && max(0, r0 - 1) >= y &&
               min(r0 + need, h - 1) < y + kWinRows;
    }
    // 8-byte loads stay inside the rows and start where they must
    __device__ __forceinline__ bool whole() const {
        return (x & 7) == 0 && x + kWinCols <= w && y + kWinRows <= h;
    }
};

__device__ __forceinline__ void window_load(const Window& v, const uint8_t* img, int pitch, int lane,
                                            uint2 (&w)[kWinLoads]) {
#pragma unroll
    for (int i = 0; i < kWinLoads; ++i) {
        const int u = lane + 32 * i;
        w[i] = make_uint2(0, 0);
        if (u < kWinUnits)
            w[i] = *reinterpret_cast<const uint2*>(img + (size_t)(v.y + (u >> 2)) * pitch + v.x + 8 * (u & 3));
    }
}

__device__ __forceinline__ void window_store(const uint2 (&w)[kWinLoads], uint8_t* win, int lane) {
#pragma unroll
    for (int i = 0; i < kWinLoads; ++i) {
        const int u = lane + 32 * i;
        if (u < kWinUnits) *reinterpret_cast<uint2*>(win + 8 * u) = w[i];
    }
}

// One window, out of line so that the loops stay short: a track that has left
// its window, and windows at the right or lower border or of a small image,
// which come byte by byte (a lane per column).  A feature that never settles
// (translation only, intensities that change) leaves its window again and again:
// byte by byte everywhere, 100 such features took 53.8 us a call, with 8-byte loads
// where they fit 43.3 (byte loads from memory in every iteration: 48.0).
__device__ __noinline__ void window_fill(const Window& v, const uint8_t* img, int pitch, int lane, uint8_t* win) {
    if (v.whole()) {
        uint2 w[kWinLoads];
        window_load(v, img, pitch, lane, w);
        window_store(w, win, lane);
    } else {
        const int rows = min(kWinRows, v.h - v.y);
        if (v.x + lane < v.w) {
            const uint8_t* p = img + (size_t)v.y * pitch + v.x + lane;
            uint8_t b[kWinRows];
#pragma unroll
            for (int r = 0; r < kWinRows; ++r) b[r] = r < rows ? p[(size_t)r * pitch] : (uint8_t)0;
#pragma unroll
            for (int r = 0; r < kWinRows; ++r) win[r * kWinCols + lane] = b[r];
        }
    }
    __syncwarp();
}

// Per warp: the template grid and the windows of both images.
struct TrackShared {
    float grid[kTrackMaxGrid];
    __align__(8) uint8_t prev[kWinRows * kWinCols], next[kWinRows * kWinCols];
};

__device__ __forceinline__ float to_float(uint8_t v) { return __uint2float_rn((uint32_t)v); }

// One pyramid level of one feature with a P x P patch.  State (t, alpha,
// beta, iters, residual) is kept identical on all lanes.  Returns false when
// the track is lost.
//
// A feature is a chain of latencies: per level the template's pixels, the
// factorisation, and per iteration the samples, the sums and the solve.  The
// pixels of both images around the feature come to shared memory once per level
// with all loads in flight at once (again when the track leaves the window), the
// sums and the divisions share the lanes.  (With byte loads from memory in every iteration, 25 shuffles for the
// five sums and a chain of ten divisions a 16 x 16 level took 4,800 cycles for
// the template, 2,000 for the factor and 1,700 per iteration; 100 features
// 30.9 -> 14.0 us a call, 64 pairs x 256 features 131 -> 102 us.  Sampling from
// memory where a window does not fit kept a second copy of every loop: a lone
// warp then waits for its instructions, and the detect-then-track loop took 45.5
// instead of 36.9 us a frame.)
template <int P>
__device__ bool track_level(const TrackLevel& lv, float cx, float cy, TrackShared& sh, int lane, int model,
                            int max_iters, float min_update, float& tx, float& ty, float& alpha, float& beta,
                            int& iters, float& residual) {
    constexpr int G = P + 2;       // template grid with a one-sample border
    constexpr int NPX = P * P / 32;  // patch pixels per lane
    constexpr int GS = (G * G + 31) / 32;  // grid samples per lane
    const float o0 = cx - 0.5f * (P - 1), o1 = cy - 0.5f * (P - 1);
    // template grid: sample (i, j) at (o0 - 1 + i, o1 - 1 + j), all inside the
    // image when the first and the last are (the positions do not decrease)
    if (!inside(o0 - 1.f, o1 - 1.f, lv.w, lv.h) ||
        !inside(o0 - 1.f + (float)(G - 1), o1 - 1.f + (float)(G - 1), lv.w, lv.h))
        return false;
    const int pc = (int)floorf(o0 - 1.f), pr = (int)floorf(o1 - 1.f);
    const Window wp = Window::around(pc, pr, G + 1, lv.w, lv.h);
    // (a position far outside the image overflows nothing: it is clamped, and no sample is taken)
    const auto cell = [](float v) { return (int)floorf(fminf(fmaxf(v, -1e6f), 1e6f)); };
    Window wn = Window::around(cell(o0 + tx), cell(o1 + ty), P + 2, lv.w, lv.h);
    if (wp.whole() && wn.whole()) {
        uint2 a[kWinLoads], b[kWinLoads];
        window_load(wp, lv.prev, lv.pitch_prev, lane, a);
        window_load(wn, lv.next, lv.pitch_next, lane, b);
        window_store(a, sh.prev, lane);
        window_store(b, sh.next, lane);
    } else {
        window_fill(wp, lv.prev, lv.pitch_prev, lane, sh.prev);
        window_fill(wn, lv.next, lv.pitch_next, lane, sh.next);
    }
    __syncwarp();
#pragma unroll
    for (int k = 0; k < GS; ++k) {
        const int idx = lane + 32 * k;
        if (idx < G * G) {
            const int j = idx / G, i = idx - j * G;
            const float gx = o0 - 1.f + (float)i, gy = o1 - 1.f + (float)j;
            const float fx = floorf(gx), fy = floorf(gy);
            const float ax = gx - fx, ay = gy - fy;
            const uint8_t* p = sh.prev + ((int)fy - wp.y) * kWinCols + ((int)fx - wp.x);
            const float a = to_float(p[0]), b = to_float(p[1]), c = to_float(p[kWinCols]), d = to_float(p[kWinCols + 1]);
            const float top = fmaf(ax, b - a, a), bot = fmaf(ax, d - c, c);
            sh.grid[idx] = fmaf(ay, bot - top, top);
        }
    }
    __syncwarp();

    // Each lane owns a strip of NPX consecutive patch rows in one column:
    // column i = lane % P, rows j = (lane / P) * NPX + m.  The samples of a
    // strip share their column, so each iteration reads NPX + 1 pairs of
    // pixels and blends each pair once (the bilinear weights are the same for
    // every sample of the patch: all sit at integer offsets from one point).
    const int col = lane % P, row0 = (lane / P) * NPX;
    // U (Eq. 4) of this lane's pixels, with the appearance at the start of the level
    const float g = 1.f + alpha;
    float T[NPX], Ux[NPX], Uy[NPX];
    // the sums of H but the last, which is the patch's pixel count
    float h[9] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (int m = 0; m < NPX; ++m) {
        const float* c = sh.grid + (row0 + m + 1) * G + (col + 1);
        T[m] = c[0];
        Ux[m] = g * (0.5f * (c[1] - c[-1]));
        Uy[m] = g * (0.5f * (c[G] - c[-G]));
        h[0] = fmaf(Ux[m], Ux[m], h[0]);
        h[1] = fmaf(Ux[m], Uy[m], h[1]);
        h[2] = fmaf(Ux[m], T[m], h[2]);
        h[3] += Ux[m];
        h[4] = fmaf(Uy[m], Uy[m], h[4]);
        h[5] = fmaf(Uy[m], T[m], h[5]);
        h[6] += Uy[m];
        h[7] = fmaf(T[m], T[m], h[7]);
        h[8] += T[m];
    }
    warp_sums(h, lane);
    const bool use_gain = model & 1, use_off = model & 2;
    float L[4][4];
    L[0][0] = h[0];
    L[1][0] = h[1];
    L[1][1] = h[4];
    // parameters the model does not estimate get an identity row: their update is 0
    L[2][0] = use_gain ? h[2] : 0.f;
    L[2][1] = use_gain ? h[5] : 0.f;
    L[2][2] = use_gain ? h[7] : 1.f;
    L[3][0] = use_off ? h[3] : 0.f;
    L[3][1] = use_off ? h[6] : 0.f;
    L[3][2] = use_off && use_gain ? h[8] : 0.f;
    L[3][3] = use_off ? (float)(P * P) : 1.f;
    L[0][1] = L[0][2] = L[0][3] = L[1][2] = L[1][3] = L[2][3] = 0.f;
    float inv[4];
    if (!cholesky4(L, inv, lane)) return false;
    const float min2 = min_update * min_update;
    float rr_last = -1.f;  // squared residual sum of the latest iteration

    for (int it = 0; it < max_iters; ++it) {
        // the patch's samples lie in the image when its corner samples do
        // (a strip's first sample is at ys, its last at ys + NPX - 1)
        const float x_lo = o0 + 0.f + tx, x_hi = o0 + (float)(P - 1) + tx;
        const float y_lo = o1 + 0.f + ty, y_hi = o1 + (float)(P - NPX) + ty + (float)(NPX - 1);
        if (!inside(x_lo, y_lo, lv.w, lv.h) || !inside(x_hi, y_hi, lv.w, lv.h)) {
            if (rr_last >= 0.f) residual = sqrtf(rr_last * (1.f / (P * P)));
            return false;
        }
        const int c0 = (int)floorf(x_lo), r0 = (int)floorf(y_lo);
        if (!wn.holds(c0, r0, P + 2)) {  // the track has left the window
            wn = Window::around(c0, r0, P + 2, lv.w, lv.h);
            __syncwarp();
            window_fill(wn, lv.next, lv.pitch_next, lane, sh.next);
        }
        // this lane's samples: column xs, rows ys .. ys + NPX - 1 of the next image
        const float xs = o0 + (float)col + tx, ys = o1 + (float)row0 + ty;
        const float fx = floorf(xs), fy = floorf(ys);
        const float ax = xs - fx, ay = ys - fy;
        const uint8_t* q = sh.next + ((int)fy - wn.y) * kWinCols + ((int)fx - wn.x);
        float p0[NPX + 1], p1[NPX + 1];
#pragma unroll
        for (int m = 0; m <= NPX; ++m) {
            p0[m] = to_float(q[m * kWinCols]);
            p1[m] = to_float(q[m * kWinCols + 1]);
        }
        float top = fmaf(ax, p1[0] - p0[0], p0[0]);
        float b[5] = {0.f, 0.f, 0.f, 0.f, 0.f};  // U r, and the squared residual
#pragma unroll
        for (int m = 0; m < NPX; ++m) {
            const float bot = fmaf(ax, p1[m + 1] - p0[m + 1], p0[m + 1]);
            const float r = fmaf(ay, bot - top, top) - fmaf(1.f + alpha, T[m], beta);
            top = bot;
            b[0] = fmaf(Ux[m], r, b[0]);
            b[1] = fmaf(Uy[m], r, b[1]);
            b[2] = fmaf(T[m], r, b[2]);
            b[3] += r;
            b[4] = fmaf(r, r, b[4]);
        }
        warp_sums(b, lane);
        const float rhs[4] = {b[0], b[1], use_gain ? b[2] : 0.f, use_off ? b[3] : 0.f};
        rr_last = b[4];
        float dq[4];
        chol_solve4(L, inv, rhs, dq);
        tx -= dq[0];
        ty -= dq[1];
        alpha += dq[2];
        beta += dq[3];
        ++iters;
        if (dq[0] * dq[0] + dq[1] * dq[1] < min2) {
            residual = sqrtf(rr_last * (1.f / (P * P)));
            return true;
        }
    }
    if (rr_last >= 0.f) residual = sqrtf(rr_last * (1.f / (P * P)));
    return true;
}

// Pyramids of both frames of every pair.
template <int L, int PAIRS>
__global__ void __launch_bounds__(256) track_pyramid_kernel(const __grid_constant__ TrackCall<PAIRS> call) {
    griddep_launch_dependents();
    for (int b = blockIdx.x; b < call.n_pyr_blocks; b += gridDim.x) {
        const int f = upper_index(call.blocks, 2 * call.n_pairs, b);
        pyramid_block<L>(call.f[f], b - call.blocks[f]);
    }
}

// One warp per feature; blockDim.x / 32 features per CTA.  Two CTAs per SM: the
// 128 registers hold a strip's template without spills, which is worth more
// than a third CTA (64 pairs x 256 features 107.9 against 111.8 us with both
// pyramids; 100 features 14.4 against 16.6 us).
template <int PAIRS>
__global__ void __launch_bounds__(kTrackWarps * 32, 2) track_kernel(const __grid_constant__ TrackCall<PAIRS> call) {
    __shared__ TrackShared shared[kTrackWarps];
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    const int f = blockIdx.x * (blockDim.x >> 5) + wib;
    if (f >= call.n_features) return;
    const int pr = upper_index(call.prefix, call.n_pairs, f);
    const int j = f - call.prefix[pr];
    const TrackPair tp = call.pairs[pr];
    const FrameDesc& fp = call.f[2 * pr];
    const FrameDesc& fn = call.f[2 * pr + 1];
    // the features were written before the pyramid kernel began; its levels are
    // final once it has completed (it may still be running: programmatic
    // dependent launch)
    float x, y;
    if (call.cells_in) {
        // a detector record: an empty cell (level < 0) gives an empty result
        const int4 rec = reinterpret_cast<const int4*>(tp.pts)[j];
        if (rec.z < 0) {
            griddep_wait();
            if (lane == 0) {
                float4* o = reinterpret_cast<float4*>(tp.out + 8 * j);
                o[0] = make_float4(-1.f, -1.f, 0.f, 0.f);
                o[1] = make_float4(__int_as_float(0), __int_as_float(0), 0.f, 0.f);
            }
            return;
        }
        x = (float)rec.x;
        y = (float)rec.y;
    } else {
        x = tp.pts[2 * j];
        y = tp.pts[2 * j + 1];
    }
    griddep_wait();
    float tx = 0.f, ty = 0.f, alpha = 0.f, beta = 0.f, residual = 0.f;
    int iters = 0;
    bool ok = true;
    const int L = call.levels;
    int k = L - 1;
    for (; k >= 0; --k) {
        const TrackLevel lv{fp.lev[k], fn.lev[k], fp.pitch[k], fn.pitch[k], fp.w >> k, fp.h >> k};
        const float s = 1.f / (float)(1 << k);
        const float cx = (x + 0.5f) * s - 0.5f, cy = (y + 0.5f) * s - 0.5f;
        const int P = k == 0 ? call.patch_fine : call.patch_coarse;
        ok = P == 16 ? track_level<16>(lv, cx, cy, shared[wib], lane, call.model, call.max_iters, call.min_update, tx,
                                       ty, alpha, beta, iters, residual)
                     : track_level<8>(lv, cx, cy, shared[wib], lane, call.model, call.max_iters, call.min_update, tx,
                                      ty, alpha, beta, iters, residual);
        if (!ok) break;
        if (k > 0) {
            tx *= 2.f;
            ty *= 2.f;
        }
        __syncwarp();  // the next level rewrites the warp's shared memory
    }
    if (lane == 0) {
        // a lost track reports its estimate so far in level-0 pixels
        const float sc = ok ? 1.f : (float)(1 << k);
        float4* o = reinterpret_cast<float4*>(tp.out + 8 * j);
        o[0] = make_float4(x + tx * sc, y + ty * sc, alpha, beta);
        o[1] = make_float4(__int_as_float(ok ? 1 : 0), __int_as_float(iters), residual, 0.f);
    }
}

}  // namespace vio
