// Detection with one CTA per tile and no call block: the pyramid is built by
// the tiles themselves, and the last CTA of a frame decodes it.
#pragma once
#include <stdint.h>

#include "vio_kernels.cuh"

namespace vio {

// What a launch needs, passed as the kernel's parameter (no upload, no tensor
// maps, and the fields come from the constant bank).  CAP: frames it holds.
template <int CAP>
struct TileCall {
    int32_t thresh, arc, n_frames, levels;
    int32_t top, n_levels;  // levels of this launch: top, top - 1, .. (n_levels of them)
    int32_t resident;       // highest level in memory before this launch (0: the frames alone)
    int32_t emit;           // coarser levels the tiles of level 0 write (0, 1 or 2)
    int32_t* counts;        // device int32[n_frames] or nullptr
    int32_t* done;          // device int32[n_frames], zero between calls: finished tiles of the frame;
                            // nullptr: a decode launch follows
    uint64_t* sums;         // device uint64[n_frames], zero between calls (tile_decode_kernel)
    uint32_t* status;
    uint32_t cell_magic[kMaxLevels];
    int32_t frame_tiles[CAP];             // tiles of the frame
    int32_t tiles[kMaxLevels * CAP + 1];  // prefix sums: entry j * n + f is level top - j of frame f
    FrameDesc f[CAP];
};
static_assert(sizeof(TileCall<64>) <= 16384, "kernel parameter");

// A level in memory.
struct LevelView {
    const uint8_t* p;
    int pitch, w, h;
    bool whole;  // every 16-byte chunk that starts inside a row can be loaded as one word
};

// 16 columns of row y from column x (a multiple of 16).  Outside the level the
// result is some of its pixels: no testable pixel looks there.  Without a
// branch (WHOLE) the loads of several units are in flight together (a level-2
// tile took 4.5 us with branches, 2.4 us without).
template <bool WHOLE>
__device__ __forceinline__ uint4 level_chunk(const LevelView& v, int x, int y) {
    const int xc = min(max(x, 0), (v.w - 1) & ~15), yc = min(max(y, 0), v.h - 1);
    const uint8_t* p = v.p + (size_t)yc * v.pitch + xc;
    if (WHOLE) return *reinterpret_cast<const uint4*>(p);
    return chunk_within(p, v.p, v.p + (size_t)v.pitch * (v.h - 1) + v.w);
}

// 8 pixels of the next level from 16 columns of two rows.
__device__ __forceinline__ uint2 halve16(uint4 t, uint4 u) {
    return make_uint2(__byte_perm(halve(t.x, u.x), halve(t.y, u.y), 0x6420),
                      __byte_perm(halve(t.z, u.z), halve(t.w, u.w), 0x6420));
}

// Fills the image box of a tile from the level K levels finer, and (K > 0) the
// tile's own level in memory with the part of it that the box covers (tiles
// overlap by their halos and write the same bytes there).  A thread's unit is a
// chunk of 16 columns x 2^K rows of the finer level, 16, 8 or 4 pixels of a row
// of the box; three units' loads are in flight at once.
template <int K, int TH, int R, bool WHOLE>
__device__ __forceinline__ void build_box(const LevelView& src, const ItemInfo& in, uint8_t* lev, int pitch,
                                          uint8_t* img) {
    using G = TileGeom<TH, R>;
    constexpr int PX = 16 >> K, UNITS = G::BW / PX, N = 1 << K;
    const int bx = (in.x0 - 8) & ~15, by = in.y0 - R - 3;
#pragma unroll 3
    for (int i = threadIdx.x; i < UNITS * G::BH; i += kConsumers) {
        const int r = i / UNITS, c = i - r * UNITS, x = bx + PX * c, y = by + r;
        uint4 v[N];
#pragma unroll
        for (int j = 0; j < N; ++j) v[j] = level_chunk<WHOLE>(src, x * N, y * N + j);
        uint8_t* d = img + r * G::BW + PX * c;
        if constexpr (K == 0) {
            *reinterpret_cast<uint4*>(d) = v[0];
        } else {
            // (pixels past the width land in the row padding)
            const bool inside = x >= 0 && x < in.wk && y >= 0 && y < in.hk;
            uint8_t* g = lev + (size_t)y * pitch + x;
            const uint2 a = halve16(v[0], v[1]);
            if constexpr (K == 1) {
                *reinterpret_cast<uint2*>(d) = a;
                if (inside) *reinterpret_cast<uint2*>(g) = a;
            } else {
                const uint2 b = halve16(v[2], v[3]);
                const uint32_t q = __byte_perm(halve(a.x, b.x), halve(a.y, b.y), 0x6420);
                *reinterpret_cast<uint32_t*>(d) = q;
                if (inside) *reinterpret_cast<uint32_t*>(g) = q;
            }
        }
    }
}

// A level-0 tile writes the pixels of levels 1 and 2 whose 4 x 4 blocks start
// in its rows and columns, from its box: the box reaches R + 3 >= 4 rows below
// the tile, enough for the last block.  One thread per 8 columns x 4 rows.
template <int TH, int R>
__device__ __forceinline__ void emit_levels(const FrameDesc& fd, const ItemInfo& in, int emit, const uint8_t* img) {
    using G = TileGeom<TH, R>;
    constexpr int UNITS = kTileW / 8, ROWS = (TH + 3) / 4 + 1;
    const int bx = (in.x0 - 8) & ~15, by = in.y0 - R - 3;
    for (int i = threadIdx.x; i < UNITS * ROWS; i += kConsumers) {
        const int r = i / UNITS, x = in.x0 + 8 * (i - r * UNITS), y = ((in.y0 + 3) & ~3) + 4 * r;
        if (y >= in.y0 + TH || y >= fd.h || x >= fd.w) continue;
        const uint8_t* p = img + (y - by) * G::BW + (x - bx);
        uint2 v[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) v[j] = *reinterpret_cast<const uint2*>(p + j * G::BW);
        uint32_t q[2];
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            q[j] = __byte_perm(halve(v[2 * j].x, v[2 * j + 1].x), halve(v[2 * j].y, v[2 * j + 1].y), 0x6420);
            if ((y >> 1) + j < (fd.h >> 1) && (x >> 1) < (fd.w >> 1))
                *reinterpret_cast<uint32_t*>(fd.lev[1] + (size_t)((y >> 1) + j) * fd.pitch[1] + (x >> 1)) = q[j];
        }
        if (emit > 1 && (y >> 2) < (fd.h >> 2) && (x >> 2) < (fd.w >> 2))
            *reinterpret_cast<uint16_t*>(fd.lev[2] + (size_t)(y >> 2) * fd.pitch[2] + (x >> 2)) =
                (uint16_t)__byte_perm(halve(q[0], q[1]), 0u, 0x4420);
    }
}

// One CTA of 8 warps per tile, five CTAs per SM (48 registers, 43 KB; with four,
// 43.0 us a call instead of 41.0 for 16 mixed frames, 79.8 instead of 77.5 for 32).
//
// The persistent kernel between a pyramid and a decode kernel costs a call about
// 20 us whatever its size: the call block's upload, three launches, the ramp
// and the tail of each.  Here
//  - with up to 3 levels all tiles are one launch: a tile of level 1 or 2
//    builds its box from level 0 (with its halo, 1.35 times the level-0 bytes
//    per level, from L2), so no tile waits for another and all run at once;
//  - with more (or frames that 16-byte loads cannot read) they are two: the tiles
//    of level 0, which write levels 1 and 2 from their boxes, then the others,
//    which build levels 3 and 4 from level 2;
//  - the CTA that finishes a frame's last tile decodes the frame in the smallest
//    calls, a decode launch in the others (counting the finished tiles costs each
//    tile 0.9 us for its fence).
// Each launch but the first is a programmatic dependent of the one before, so
// its CTAs move in as that drains.
// The phases of a tile are separated by CTA barriers, and the other four CTAs of
// the SM fill them.  A tile alone takes 3.4 us (load 1.3, coarse test 0.6, full
// test, scores and NMS 0.6, fence and count 0.9); one 752x480 frame, 152 tiles of
// 30 rows, 10.3 us a call with the decode.  The rule for which calls come here
// stands in vio_tiles.cu.
template <int TH, int MODE, int R, int CAP>
__global__ void __launch_bounds__(kConsumers, 5) tile_detect_kernel(const __grid_constant__ TileCall<CAP> call) {
    using G = TileGeom<TH, R>;
    extern __shared__ __align__(128) uint8_t smem[];
    uint8_t* img = smem;
    uint16_t* sc = reinterpret_cast<uint16_t*>(smem + G::BOXA);
    __shared__ int hits_sh, last_sh;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    uint16_t* queue = reinterpret_cast<uint16_t*>(smem + G::BOXA + G::SR * G::SW * 2) + warp * G::QCAP;
    const uint32_t lt_mask = (1u << lane) - 1u;

    griddep_launch_dependents();
    // one warp finds the tile, the others clear the score tile
    __shared__ ItemInfo in;
    __shared__ int f_sh;
    if (warp == 0) {
        const int it = blockIdx.x, n = call.n_frames;
        const int j = upper_index(call.tiles, n * call.n_levels, it);
        const int f = j % n;
        const FrameDesc& fd = call.f[f];
        ItemInfo i;
        i.id = it;
        i.level = call.top - j / n;
        i.wk = fd.w >> i.level;
        i.hk = fd.h >> i.level;
        i.gw = fd.gw;
        i.gh = fd.gh;
        i.keys = fd.keys;
        i.magic = call.cell_magic[i.level];
        const int ti = it - call.tiles[j], ntx = (i.wk + kTileW - 1) / kTileW, ty = ti / ntx;
        i.x0 = (ti - ty * ntx) * G::TW;
        i.y0 = ty * TH;
        tile_constants<TH, R>(i);
        if (lane == 0) {
            in = i;
            f_sh = f;
            hits_sh = 0;
        }
    } else {
        for (int i = tid - 32; i < G::SR * G::SW / 8; i += kConsumers - 32)
            reinterpret_cast<uint4*>(sc)[i] = make_uint4(0, 0, 0, 0);
    }
    __syncthreads();
    const int f = f_sh;
    const FrameDesc& fd = call.f[f];
    // everything below reads what earlier launches wrote
    griddep_wait();
    {
        const int from = min(in.level, call.resident);
        LevelView v{fd.lev[from], fd.pitch[from], fd.w >> from, fd.h >> from, false};
        // (a resident level's rows are padded to 128 bytes)
        v.whole = from > 0 ||
                  ((((uint32_t)reinterpret_cast<uintptr_t>(v.p) | (uint32_t)v.pitch | (uint32_t)v.w) & 15) == 0);
        uint8_t* lev = fd.lev[in.level];
        const int pitch = fd.pitch[in.level], up = in.level - from;
        if (v.whole) {
            if (up == 0) build_box<0, TH, R, true>(v, in, lev, pitch, img);
            else if (up == 1) build_box<1, TH, R, true>(v, in, lev, pitch, img);
            else build_box<2, TH, R, true>(v, in, lev, pitch, img);
        } else {
            if (up == 0) build_box<0, TH, R, false>(v, in, lev, pitch, img);
            else if (up == 1) build_box<1, TH, R, false>(v, in, lev, pitch, img);
            else build_box<2, TH, R, false>(v, in, lev, pitch, img);
        }
    }
    __syncthreads();
    if (call.emit > 0) emit_levels<TH, R>(fd, in, call.emit, img);

    const int thresh = call.thresh, n_arc = call.arc;
    const bool high_t = thresh >= 128;
    const uint32_t k7 = (uint32_t)((high_t ? 255 : 127) - thresh) * 0x01010101u;
    const uint32_t vm = kept_columns(in, lane);
    const int total = high_t ? coarse_and_compact<true, TH, R>(img, queue, in.xoff / 4, k7, n_arc, warp, lane,
                                                               in.row_lo, in.row_hi, vm, call.status)
                             : coarse_and_compact<false, TH, R>(img, queue, in.xoff / 4, k7, n_arc, warp, lane,
                                                                in.row_lo, in.row_hi, vm, call.status);
    __syncwarp();
    const uint8_t* img_base = img + 3 * G::BW + in.xoff;
    const int ncorner = full_test<MODE, TH, R>(img_base, queue, total, warp, lane, lt_mask, thresh, n_arc, call.status);
    __syncwarp();
    score_corners<MODE, TH, R>(img_base, queue, ncorner, lane, thresh, n_arc, sc);
    __syncthreads();
    nms_corners<TH, R>(queue, ncorner, sc, lane, lt_mask, in, call.status);

    if (!call.done) return;
    // the CTA that finishes a frame's last tile decodes the frame: its keys are
    // complete (each thread's reductions are ordered before the CTA's count)
    __threadfence();
    __syncthreads();
    if (tid == 0) last_sh = atomicAdd(&call.done[f], 1) == call.frame_tiles[f] - 1;
    __syncthreads();
    if (!last_sh) return;
    __threadfence();
    const int cells = fd.gw * fd.gh;
    int hits = 0;
    constexpr int KEYS = 4;  // keys in flight per thread
    for (int c0 = tid; c0 < cells; c0 += KEYS * kConsumers) {
        uint64_t key[KEYS];
#pragma unroll
        for (int q = 0; q < KEYS; ++q) {
            const int c = c0 + q * kConsumers;
            key[q] = c < cells ? __ldcg(reinterpret_cast<const unsigned long long*>(fd.keys) + c) : 0ull;
        }
#pragma unroll
        for (int q = 0; q < KEYS; ++q) {
            const int c = c0 + q * kConsumers;
            if (c >= cells) break;
            int4 rec = make_int4(-1, -1, -1, 0);
            if (key[q] != 0) {
                rec = decode_key(key[q], c, fd.w, fd.h, fd.gw, call.levels, call.cell_magic[0], call.status);
                fd.keys[c] = 0;
                ++hits;
            }
            fd.out[c] = rec;
        }
    }
    if (hits) atomicAdd(&hits_sh, hits);
    __syncthreads();
    if (tid == 0) {
        call.done[f] = 0;
        if (call.counts) call.counts[f] = hits_sh;
    }
}

// Pyramids of frames that it also uploads (FrameDesc::src0: the device mapping
// of host memory); blocks: prefix sums per frame, in tiles[].
template <int L, int CAP>
__global__ void __launch_bounds__(256) tile_pyramid_kernel(const __grid_constant__ TileCall<CAP> call) {
    griddep_launch_dependents();
    const int n = call.n_frames, blocks = call.tiles[n];
    for (int b = blockIdx.x; b < blocks; b += gridDim.x) {
        const int f = upper_index(call.tiles, n, b);
        pyramid_block<L>(call.f[f], b - call.tiles[f]);
    }
}

// Decode in a launch of its own: one thread per cell, blocks of 256 cells of
// one frame (blocks: prefix sums per frame, in tiles[]).  A frame's count is
// added up over its blocks in sums[], which the frame's last block hands over
// and clears: the low half counts blocks, the high half cells.
template <int CAP>
__global__ void __launch_bounds__(256) tile_decode_kernel(const __grid_constant__ TileCall<CAP> call) {
    const int b = blockIdx.x, f = upper_index(call.tiles, call.n_frames, b);
    const FrameDesc& fd = call.f[f];
    const int c = (b - call.tiles[f]) * 256 + (int)threadIdx.x;
    griddep_wait();
    bool hit = false;
    if (c < fd.gw * fd.gh) {
        const uint64_t key = fd.keys[c];
        int4 rec = make_int4(-1, -1, -1, 0);
        if (key != 0) {
            rec = decode_key(key, c, fd.w, fd.h, fd.gw, call.levels, call.cell_magic[0], call.status);
            fd.keys[c] = 0;
            hit = true;
        }
        fd.out[c] = rec;
    }
    if (!call.counts) return;
    const int hits = __syncthreads_count(hit);
    if (threadIdx.x == 0) {
        unsigned long long* sum = reinterpret_cast<unsigned long long*>(call.sums) + f;
        const unsigned long long was = atomicAdd(sum, 1ull | ((unsigned long long)hits << 32));
        if ((int)(was & 0xFFFFFFFFu) == call.tiles[f + 1] - call.tiles[f] - 1) {
            call.counts[f] = (int)(was >> 32) + hits;
            *sum = 0;
        }
    }
}

}  // namespace vio
