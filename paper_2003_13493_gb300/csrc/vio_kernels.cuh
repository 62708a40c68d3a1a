// Device code: pyramid half-sampling, the fused FAST + NMS + cell-max kernel
// (3x3 to 9x9 NMS windows, scores SAD-B / SAD-A / MT), and the cell decode.
// All arithmetic is integer.
#pragma once
#include <cuda.h>
#include <stdint.h>

#include "ptx.cuh"

namespace vio {

constexpr int kMaxLevels = 5;
constexpr int kPrefixCache = 1025;  // prefix-table entries a kernel copies to shared memory (1024 frames)
constexpr uint32_t kStatusTimeout = 1u;  // a bounded wait gave up
constexpr uint32_t kStatusBadKey = 2u;   // a decoded cell key lies outside its cell
constexpr uint32_t kStatusBounds = 4u;   // checked build: an index left its buffer

// Index checks of the checked build (compiled with -DVIO_CHECKED): a failed
// check records kStatusBounds and the access is skipped.  In the normal
// build every check is `true` and compiles away.
__device__ __forceinline__ bool vio_guard(bool in_bounds, uint32_t* status) {
#ifdef VIO_CHECKED
    if (!in_bounds && status) atomicOr(status, kStatusBounds);
    return in_bounds;
#else
    (void)in_bounds;
    (void)status;
    return true;
#endif
}
constexpr uint64_t kWaitLimitNs = 1000000000ull;  // 1 s per bounded wait

// Per-frame descriptor, rewritten by the host for every call.
struct FrameDesc {
    int32_t w, h;          // level-0 size
    int32_t gw, gh;        // cell grid
    int32_t pyr_cx;        // 16-column chunks per row of level 0 (at least 2)
    int32_t src0_pitch;    // row pitch of src0
    uint64_t* keys;        // gw * gh packed cell keys (0 = empty)
    int4* out;             // gw * gh output records (device or device-mapped host memory)
    const uint8_t* src0;   // non-null: level 0 is read from here (device-mapped host memory,
                           // or a frame that TMA cannot address, of any alignment) by the
                           // pyramid kernel, which also writes it to lev[0]
    uint8_t* lev[kMaxLevels];   // level 0 is the caller's frame (read only)
    int32_t pitch[kMaxLevels];
    uint32_t pyr_magic;    // ceil(2^32 / pyr_cx)
    int32_t pad1[2];
};

// Everything one call needs is uploaded as one contiguous block; this header
// sits at its start and holds the byte offsets of the other sections:
//   FrameDesc fds[n]
//   CUtensorMap maps0[n]                    level 0 (the caller's frames)
//   CUtensorMap mapsk[n][kMaxLevels - 1]    levels 1.. (resident pyramid)
//   int32 tiles[n * levels + 1]             prefix sums of tiles, coarsest
//                                           level first: entry (L-1-k)*n + f
//   int32 blocks[n + 1]                     prefix sums of pyramid blocks
//   int32 cells[n + 1]                      prefix sums of cells per frame
struct CallHeader {
    int32_t thresh, arc, n_frames, levels;
    int32_t cell, n_items, n_pyr_blocks, tile_h;
    int32_t* counts;       // device int32[n_frames] or nullptr
    uint32_t off_fds, off_maps0, off_mapsk, off_tiles, off_blocks, off_cells;
    // cell_magic[k] = ceil(2^32 / (cell >> k)): for level coordinates
    // x < 2^16, umulhi(x, magic) == x / (cell >> k) == (x << k) / cell exactly
    uint32_t cell_magic[kMaxLevels];
    int32_t n_cells;       // cells of all frames
    uint32_t* status;      // device-visible status word for the decode's checks, or nullptr
};

struct CallView {
    const CallHeader* h;
    const FrameDesc* fds;
    const CUtensorMap* maps0;
    const CUtensorMap* mapsk;
    const int32_t* tiles;
    const int32_t* blocks;
    const int32_t* cells;
    __device__ __forceinline__ explicit CallView(const uint8_t* call)
        : h(reinterpret_cast<const CallHeader*>(call)),
          fds(reinterpret_cast<const FrameDesc*>(call + h->off_fds)),
          maps0(reinterpret_cast<const CUtensorMap*>(call + h->off_maps0)),
          mapsk(reinterpret_cast<const CUtensorMap*>(call + h->off_mapsk)),
          tiles(reinterpret_cast<const int32_t*>(call + h->off_tiles)),
          blocks(reinterpret_cast<const int32_t*>(call + h->off_blocks)),
          cells(reinterpret_cast<const int32_t*>(call + h->off_cells)) {}
};

// Largest i in [0, n) with a[i] <= v, for a non-decreasing a with a[0] <= v.
__device__ __forceinline__ int upper_index(const int32_t* a, int n, int v) {
    int lo = 0, hi = n - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (a[mid] <= v) lo = mid; else hi = mid - 1;
    }
    return lo;
}

// ---------------------------------------------------------------------------
// Pyramid: one thread owns a chunk of 16 columns x B rows of level 0 (B =
// 2^(L-1)) and writes every pixel of levels 1..L-1 that it produces.  Level
// k+1 is the 2x2 mean of level k rounded half up, (a+b+c+d+2)>>2, taken from
// the rounded level-k values.  Level 0 is read with 16-byte loads; a pixel's
// four values are summed by two byte dot products (on the multiply-add pipe),
// two pixels per word are shifted and packed by one permute, and a thread
// stores 8, 4, 2 and 1 bytes of a row of levels 1 to 4.  Stores past a level's
// width land in the row padding (pitch: the width rounded up to 128).
//
// The chunks of a frame are numbered row by row and dealt to the threads of
// its blocks (blocks[] is the per-frame prefix sum of blocks of 256 chunks), so
// every lane has work whatever the width: blocks of 512 columns left a
// quarter to a third of the lanes of 640 and 752 pixel rows idle.
//
// A frame with src0 set is read from there instead and written to lev[0]
// (rows of a multiple of 16 bytes) as well, whatever its alignment: this kernel
// is then the upload or the staging copy too, and saves a copy per frame.  With
// one level (L = 1) that is all it does.
//
// Bound by memory latency and issue on batches of a few tens of megabytes, by
// HBM on large ones (32 4K frames: 353 MB in 63 us, 0.83 of the copy rate).  64
// mixed frames, 3 levels: 17.6 us alone (20.2 with blocks of 512 columns), 22 us in
// the call.  24 frames of odd width, 4 levels, by the persistent kernels: 83.6 us a
// call (180.6 with a copy per frame).
// ---------------------------------------------------------------------------
__host__ __device__ constexpr int pyr_rows(int levels) { return levels == 1 ? 4 : 1 << (levels - 1); }

// Fills a frame's pyramid fields (w, h set); returns its blocks.
inline int pyr_plan(FrameDesc& f, int levels) {
    f.pyr_cx = (f.w + 15) / 16 < 2 ? 2 : (f.w + 15) / 16;
    f.pyr_magic = (uint32_t)(((1ull << 32) + f.pyr_cx - 1) / f.pyr_cx);
    if (levels == 1 && !f.src0) return 0;
    const int64_t chunks = (int64_t)f.pyr_cx * ((f.h + pyr_rows(levels) - 1) / pyr_rows(levels));
    return (int)((chunks + 255) / 256);
}

// The word at p (4-byte aligned), bytes outside [begin, end) zero and not read.
__device__ __forceinline__ uint32_t word_within(const uint8_t* p, const uint8_t* begin, const uint8_t* end) {
    if (p >= begin && p + 4 <= end) return *reinterpret_cast<const uint32_t*>(p);
    uint32_t v = 0;
    for (int i = 0; i < 4; ++i)
        if (p + i >= begin && p + i < end) v |= (uint32_t)p[i] << (8 * i);
    return v;
}

// The 16 bytes at p, of any alignment, of a frame that occupies [begin, end).
__device__ __forceinline__ uint4 chunk_within(const uint8_t* p, const uint8_t* begin, const uint8_t* end) {
    const uint32_t a = (uint32_t)reinterpret_cast<uintptr_t>(p) & 3u, sh = 8u * a;
    const uint8_t* q = p - a;
    uint32_t w[5];
    if (q >= begin && q + 20 <= end) {
#pragma unroll
        for (int i = 0; i < 5; ++i) w[i] = reinterpret_cast<const uint32_t*>(q)[i];
    } else {  // at the ends of the frame
#pragma unroll
        for (int i = 0; i < 4; ++i) w[i] = word_within(q + 4 * i, begin, end);
        w[4] = a ? word_within(q + 16, begin, end) : 0u;
    }
    return make_uint4(__funnelshift_r(w[0], w[1], sh), __funnelshift_r(w[1], w[2], sh),
                      __funnelshift_r(w[2], w[3], sh), __funnelshift_r(w[3], w[4], sh));
}

// Two pixels of the next level from four columns of two rows: bytes 0 and 2
// (bytes 1 and 3 are left over).
__device__ __forceinline__ uint32_t halve(uint32_t t, uint32_t u) {
    const uint32_t lo = __dp4a(t, 0x00000101u, __dp4a(u, 0x00000101u, 2u));
    const uint32_t hi = __dp4a(t, 0x01010000u, __dp4a(u, 0x01010000u, 2u));
    return (lo + hi * 65536u) >> 2;
}

// A thread's chunk of one row of level K, from its level-0 rows r[], storing
// every row it makes on the way: 8 pixels in two words for K = 1, then 4, 2, 1.
template <int K, int N>
struct PyrRow {
    uint32_t w[K == 1 ? 2 : 1];
    __device__ __forceinline__ PyrRow(const FrameDesc& fd, const uint4 (&r)[N], int tx, int ty, int j) {
        constexpr int PX = 16 >> K, ROWS = N >> K;
        if constexpr (K == 1) {
            const uint4 t = r[2 * j], u = r[2 * j + 1];
            w[0] = __byte_perm(halve(t.x, u.x), halve(t.y, u.y), 0x6420);
            w[1] = __byte_perm(halve(t.z, u.z), halve(t.w, u.w), 0x6420);
        } else {
            const PyrRow<K - 1, N> a(fd, r, tx, ty, 2 * j), b(fd, r, tx, ty, 2 * j + 1);
            if constexpr (K == 2) w[0] = __byte_perm(halve(a.w[0], b.w[0]), halve(a.w[1], b.w[1]), 0x6420);
            if constexpr (K == 3) w[0] = __byte_perm(halve(a.w[0], b.w[0]), 0u, 0x4420);
            if constexpr (K == 4) w[0] = __dp4a(a.w[0], 0x0101u, __dp4a(b.w[0], 0x0101u, 2u)) >> 2;
        }
        const int x = tx * PX, y = ty * ROWS + j;
        if (x < (fd.w >> K) && y < (fd.h >> K)) {
            uint8_t* d = fd.lev[K] + (size_t)y * fd.pitch[K] + x;
            if constexpr (K == 1) *reinterpret_cast<uint2*>(d) = make_uint2(w[0], w[1]);
            if constexpr (K == 2) *reinterpret_cast<uint32_t*>(d) = w[0];
            if constexpr (K == 3) *reinterpret_cast<uint16_t*>(d) = (uint16_t)w[0];
            if constexpr (K == 4) *d = (uint8_t)w[0];
        }
    }
};

// Thread `thread`'s chunk in block `block` of a frame.
struct PyrChunk {
    int tx, ty;  // column and row of chunks
};
__host__ __device__ __forceinline__ PyrChunk pyr_chunk(const FrameDesc& fd, int block, int thread) {
    const int cx = fd.pyr_cx;
    // chunk number = ty * cx + tx.  The product with ceil(2^32 / cx) gives the
    // row of the block's first chunk or one more (a frame has at most 2^24
    // chunks), the division of a thread's chunk alike.
    const auto divide = [&](int v) {
        const int q = (int)(((uint64_t)(uint32_t)v * fd.pyr_magic) >> 32);
        return q * cx > v ? q - 1 : q;
    };
    const int first = block * 256, row = divide(first);
    const int off = first - row * cx + thread, down = divide(off);
    return {off - down * cx, row + down};
}

// Block `block` of a frame: 256 chunks, one per thread.
template <int L>
__device__ __forceinline__ void pyramid_block(const FrameDesc& fd, int block) {
    constexpr int B = pyr_rows(L);
    const PyrChunk c = pyr_chunk(fd, block, (int)threadIdx.x);
    const int tx = c.tx, ty = c.ty;
    const int W = fd.w, H = fd.h, x0 = tx * 16, y0 = ty * B;
    if (x0 >= W || y0 >= H) return;
    const bool upload = fd.src0 != nullptr;
    const uint8_t* src = upload ? fd.src0 : fd.lev[0];
    const int sp = upload ? fd.src0_pitch : fd.pitch[0];
    const uint8_t* p = src + (size_t)y0 * sp + x0;
    uint4 r[B];
    if (x0 + 16 <= W && ((reinterpret_cast<uintptr_t>(src) | (uint32_t)sp) & 15) == 0) {
#pragma unroll
        for (int j = 0; j < B; ++j)
            r[j] = y0 + j < H ? *reinterpret_cast<const uint4*>(p + (size_t)j * sp) : make_uint4(0, 0, 0, 0);
    } else {
        // the last partial chunk of a row, and frames of any alignment
        const uint8_t* end = src + (size_t)sp * (H - 1) + W;
#pragma unroll
        for (int j = 0; j < B; ++j)
            r[j] = y0 + j < H ? chunk_within(p + (size_t)j * sp, src, end) : make_uint4(0, 0, 0, 0);
    }
    if (upload) {
#pragma unroll
        for (int j = 0; j < B; ++j)
            if (y0 + j < H) *reinterpret_cast<uint4*>(fd.lev[0] + (size_t)(y0 + j) * fd.pitch[0] + x0) = r[j];
    }
    if constexpr (L > 1) {
        constexpr int TOP = L - 1;
        PyrRow<TOP, B> top(fd, r, tx, ty, 0);
        (void)top;
    }
}

template <int L>
__global__ void __launch_bounds__(256) pyramid_kernel(const uint8_t* __restrict__ call) {
    griddep_launch_dependents();
    const CallView cv(call);
    const int nf = cv.h->n_frames, nb = cv.h->n_pyr_blocks;
    // the block prefix sums, searched once per block by every thread: in
    // shared memory when they fit (a search of the global table is a chain of
    // dependent loads)
    __shared__ int32_t blocks_sh[kPrefixCache];
    const int32_t* blocks = nf < kPrefixCache ? blocks_sh : cv.blocks;
    if (nf < kPrefixCache)
        for (int i = threadIdx.x; i <= nf; i += blockDim.x) blocks_sh[i] = cv.blocks[i];
    __syncthreads();
    for (int b = blockIdx.x; b < nb; b += gridDim.x) {
        const int f = upper_index(blocks, nf, b);
        pyramid_block<L>(cv.fds[f], b - blocks[f]);
    }
}

// ---------------------------------------------------------------------------
// FAST segment test and scores on a shared-memory tile.
// ---------------------------------------------------------------------------

// Radius-3 Bresenham circle, clockwise from the top (Section II-D).
__host__ __device__ constexpr int circ_dx(int i) {
    return i == 0 ? 0 : i == 1 ? 1 : i == 2 ? 2 : i <= 5 ? 3 : i == 6 ? 2 : i == 7 ? 1 : i == 8 ? 0
         : i == 9 ? -1 : i == 10 ? -2 : i <= 13 ? -3 : i == 14 ? -2 : -1;
}
__host__ __device__ constexpr int circ_dy(int i) {
    return i <= 1 ? -3 : i == 2 ? -2 : i == 3 ? -1 : i == 4 ? 0 : i == 5 ? 1 : i == 6 ? 2 : i <= 9 ? 3
         : i == 10 ? 2 : i == 11 ? 1 : i == 12 ? 0 : i == 13 ? -1 : i == 14 ? -2 : -3;
}

// Start positions s (bits 0..15) of cyclic runs of >= n ones in the 16-bit
// mask m: the mask is doubled to 32 bits (a rotation without wrap-around),
// runs of 8 come from three AND-shift doublings and the run of n from two
// overlapping runs of 8 that are n-8 apart.
__device__ __forceinline__ uint32_t arc_starts(uint32_t m, int n) {
    uint32_t r = m * 0x10001u;
    r &= r >> 1;
    r &= r >> 2;
    r &= r >> 4;
    r &= r >> (n - 8);
    return r & 0xFFFFu;
}

// 16-bit rotate left of the low 16 bits.
__device__ __forceinline__ uint32_t rotl16(uint32_t m, int s) {
    return ((m << s) | (m >> (16 - s))) & 0xFFFFu;
}

// [sign(a byte 1), sign(a byte 3), sign(b byte 1), sign(b byte 3)]: each result
// byte is 0xFF when the bit 15 / bit 31 it is taken from is set, else 0x00
// (the PTX byte permute with the sign-replicate bit set in every selector).
__device__ __forceinline__ uint32_t prmt_sign_flags(uint32_t a, uint32_t b) {
    uint32_t d;
    asm("prmt.b32 %0, %1, %2, 0xFDB9;" : "=r"(d) : "r"(a), "r"(b));
    return d;
}

// Four bytes packed into one word, byte 0 first.
__device__ __forceinline__ uint32_t pack4(uint32_t a, uint32_t b, uint32_t c, uint32_t d) {
    return __byte_perm(__byte_perm(a, b, 0x0040), __byte_perm(c, d, 0x0040), 0x5410);
}

// 16-bit-lane minimum and maximum on the DPX unit.
__device__ __forceinline__ uint32_t min16x2(uint32_t a, uint32_t b) { return __vimin3_u16x2(a, b, b); }

// Window minima of the circle's signed differences (the sweep's full test,
// the MT score).  D[i] holds point i's biased
// differences, v - c + 256 in the low 16-bit lane (brighter) and c - v + 256
// in the high lane (darker), both in 1..511 so no lane borrows; W8[i] is the
// lane-wise minimum over points i .. i+7 (cyclic), from minima of three.
__device__ __forceinline__ void window_minima8_of(const uint32_t (&v)[16], uint32_t c, uint32_t (&W8)[16]) {
    const uint32_t K = (256u - c) | ((256u + c) << 16);
    uint32_t D[16];
#pragma unroll
    for (int i = 0; i < 16; ++i) D[i] = K + v[i] * 0xFFFF0001u;
    uint32_t W3[16];
#pragma unroll
    for (int i = 0; i < 16; ++i) W3[i] = __vimin3_u16x2(D[i], D[(i + 1) & 15], D[(i + 2) & 15]);
#pragma unroll
    for (int i = 0; i < 16; ++i) W8[i] = __vimin3_u16x2(W3[i], W3[(i + 3) & 15], W3[(i + 5) & 15]);
}

// p: the candidate in a tile of row pitch PITCH bytes.
template <int PITCH>
__device__ __forceinline__ void window_minima8(const uint8_t* __restrict__ p, uint32_t (&W8)[16]) {
    uint32_t v[16];
#pragma unroll
    for (int i = 0; i < 16; ++i) v[i] = p[circ_dy(i) * PITCH + circ_dx(i)];
    window_minima8_of(v, p[0], W8);
}

// Largest minimum over the 16 windows of 8 + R points (both polarities),
// still biased by 256: the candidate is a corner at threshold t for arc
// length 8 + R exactly when the result is >= t + 257.  A window of 8 + R
// points is two overlapping windows of 8, R apart.
template <int R>
__device__ __forceinline__ uint32_t best_window_min(const uint32_t (&W8)[16]) {
    uint32_t m[16];
#pragma unroll
    for (int i = 0; i < 16; ++i) m[i] = min16x2(W8[i], W8[(i + R) & 15]);
    uint32_t b = __vimax3_u16x2(m[0], m[1], m[2]);
    b = __vimax3_u16x2(b, m[3], m[4]);
    b = __vimax3_u16x2(b, m[5], m[6]);
    b = __vimax3_u16x2(b, m[7], m[8]);
    b = __vimax3_u16x2(b, m[9], m[10]);
    b = __vimax3_u16x2(b, m[11], m[12]);
    b = __vimax3_u16x2(b, m[13], m[14]);
    b = __vimax3_u16x2(b, m[15], m[15]);
    return max(b & 0xFFFFu, b >> 16);
}

__device__ __forceinline__ uint32_t best_window_min_for_arc(const uint32_t (&W8)[16], int n) {
    switch (n) {  // uniform over the launch
        case 9: return best_window_min<1>(W8);
        case 10: return best_window_min<2>(W8);
        case 11: return best_window_min<3>(W8);
        case 12: return best_window_min<4>(W8);
        case 13: return best_window_min<5>(W8);
        case 14: return best_window_min<6>(W8);
        case 15: return best_window_min<7>(W8);
        default: return best_window_min<8>(W8);
    }
}

// Full segment test and score of the pixel at shared-memory pointer p in a
// tile of row pitch P (compile time).  Returns 0 when it is not a corner.
//
// Eq. 1 labels come from one IMAD per circle point: with
//   W = ((0x7FFF - c - t) | (0x7FFF + c - t) << 16) + v * (1 - 2^16)
// the low 16-bit lane is v + 0x7FFF - (c + t), whose bit 15 is set exactly
// when v > c + t (brighter), and the high lane is 0x7FFF + (c - t) - v,
// whose bit 31 is set exactly when v < c - t (darker).  Neither lane leaves
// its 16 bits, so the two compares are exact for all v, c in 0..255 and
// t in 0..255.  The flags become masks in two steps: a byte permute with
// sign replication turns the flag bits (bits 15 and 31 are the sign bits of
// bytes 1 and 3) of points i and i + 8 into four 0x00 / 0xFF bytes
// [bright_i, dark_i, bright_i+8, dark_i+8]; keeping bit i of each byte and
// OR-ing the eight words gives bright 0..7, dark 0..7, bright 8..15 and
// dark 8..15 in bytes 0..3; a last permute orders them as the 16-bit bright
// mask in bits 0..15 and the dark mask in bits 16..31, bit i = point i.
template <int MODE, int P, bool SCORE = true>
__device__ __forceinline__ uint32_t eval_corner(const uint8_t* __restrict__ p, int t, int n) {
    const uint32_t c = p[0];
    uint32_t v[16];
#pragma unroll
    for (int i = 0; i < 16; ++i) v[i] = p[circ_dy(i) * P + circ_dx(i)];
    const uint32_t K = ((0x7FFFu - c - (uint32_t)t) & 0xFFFFu) | ((0x7FFFu + c - (uint32_t)t) << 16);
    uint32_t w[16];
#pragma unroll
    for (int i = 0; i < 16; ++i) w[i] = K + v[i] * 0xFFFF0001u;
    uint32_t bytes = 0;
#pragma unroll
    for (int i = 0; i < 8; ++i) bytes |= prmt_sign_flags(w[i], w[i + 8]) & (0x01010101u << i);
    const uint32_t acc = __byte_perm(bytes, 0u, 0x3120);
    const uint32_t bm = acc & 0xFFFFu, dm = acc >> 16;
    // at most one polarity can hold n >= 9 points
    const bool bright = __popc(bm) >= n;
    const uint32_t starts = arc_starts(bright ? bm : dm, n);
    if (starts == 0) return 0;
    if (!SCORE) return 1;
    if (MODE == 0) {  // SAD-B: sum of |I_x - I_c| over the circle
        const uint32_t c4 = c * 0x01010101u;
        uint32_t s = __vsadu4(pack4(v[0], v[1], v[2], v[3]), c4);
        s += __vsadu4(pack4(v[4], v[5], v[6], v[7]), c4);
        s += __vsadu4(pack4(v[8], v[9], v[10], v[11]), c4);
        s += __vsadu4(pack4(v[12], v[13], v[14], v[15]), c4);
        return s;
    } else if (MODE == 1) {  // SAD-A: the run is the union of all passing windows
        uint32_t d = starts;
        d |= rotl16(d, 1);
        d |= rotl16(d, 2);
        d |= rotl16(d, 4);  // windows of 8 starting at each start
        const uint32_t run = d | rotl16(d, n - 8);
        // SAD over the run: each nibble of the run mask spreads to a byte
        // mask of its four circle points (bit i -> bit 8i by one multiply;
        // the shifted copies occupy disjoint bits, so nothing carries)
        const uint32_t c4 = c * 0x01010101u;
        uint32_t s = 0;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const uint32_t m = (((run >> (4 * q)) & 0xFu) * 0x00204081u & 0x01010101u) * 0xFFu;
            s += __vsadu4(pack4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]) & m, c4 & m);
        }
        return s;
    } else {  // MT: the largest t at which the pixel is still a corner
        // = the largest minimum over all windows of n points of the signed
        // differences, minus 1 (both polarities at once: the one that is not
        // the corner's has no window above 0, as no pixel holds arcs of 9 of
        // both polarities); biased by 256
        uint32_t W8[16];
        window_minima8_of(v, c, W8);
        return best_window_min_for_arc(W8, n) - 257u;
    }
}

// MT score of a pixel already known to be a corner for arc length n: the
// largest minimum over the windows of n signed differences, minus 1 (biased
// by 256 as in eval_corner).
template <int P>
__device__ __forceinline__ uint32_t mt_of_corner(const uint8_t* __restrict__ p, int n) {
    uint32_t W8[16];
    window_minima8<P>(p, W8);
    return best_window_min_for_arc(W8, n) - 257u;
}

// SAD-B of the pixel at p (row pitch P): sum of |I_x - I_c| over the circle.
template <int P>
__device__ __forceinline__ uint32_t sad_b(const uint8_t* __restrict__ p) {
    const uint32_t c4 = p[0] * 0x01010101u;
    uint32_t v[16];
#pragma unroll
    for (int i = 0; i < 16; ++i) v[i] = p[circ_dy(i) * P + circ_dx(i)];
    uint32_t s = __vsadu4(pack4(v[0], v[1], v[2], v[3]), c4);
    s += __vsadu4(pack4(v[4], v[5], v[6], v[7]), c4);
    s += __vsadu4(pack4(v[8], v[9], v[10], v[11]), c4);
    s += __vsadu4(pack4(v[12], v[13], v[14], v[15]), c4);
    return s;
}

// Byte-wise |a - b| > t for the 4 pixels of a word: bit 7 of each byte, the
// other bits clear.  Never misses a pixel, and for t < 128 may flag one with
// |a - b| == t: with k7 = 127 - t the sum d + k7 reaches bit 7 when d > t, or
// d >= 128 holds bit 7 itself; a byte that overflows (d > 128 + t) carries 1
// into its neighbour, which changes that neighbour's flag only at d == t.
// The coarse test keeps a superset anyway and the full test decides, so the
// mask that would stop the carry is left out (one instruction in four).  With
// t >= 128 a byte that overflowed would lose its flag: there (d & 0x7F) is
// added to k7 = 255 - t, the carry into bit 7 means (d & 0x7F) > t - 128, and
// it counts only together with bit 7 of d (exact).
template <bool HIGH_T>
__device__ __forceinline__ uint32_t gt_flags(uint32_t a, uint32_t b, uint32_t k7) {
    const uint32_t d = __vabsdiffu4(a, b);
    return HIGH_T ? (((d & 0x7F7F7F7Fu) + k7) & d & 0x80808080u) : (((d + k7) | d) & 0x80808080u);
}

// Appends a row's flags to a word of eight rows: the rows move down one bit
// in their bytes, the oldest falls out, the new row enters at bit 7.
__device__ __forceinline__ uint32_t push_row(uint32_t acc, uint32_t flags) {
    return ((acc >> 1) & 0x7F7F7F7Fu) | flags;
}

// Pixels with RUN cyclically consecutive flags among the eight even circle
// points f (N NE E SE S SW W NW), 32 pixels per word.
template <int RUN>
__device__ __forceinline__ uint32_t run_of_even(const uint32_t (&f)[8]) {
    static_assert(RUN == 5 || RUN == 6, "two runs of three that overlap or meet");
    uint32_t r3[8], keep = 0;
#pragma unroll
    for (int i = 0; i < 8; ++i) r3[i] = f[i] & f[(i + 1) & 7] & f[(i + 2) & 7];
#pragma unroll
    for (int i = 0; i < 8; ++i) keep |= r3[i] & r3[(i + RUN - 3) & 7];
    return keep;
}

// ---------------------------------------------------------------------------
// Fused detect: persistent CTAs pull (frame, level, tile) items from a
// counter.  A tile is 120 x TH level pixels; its "score region" adds a ring
// (4 px left and right, R rows up and down for an NMS radius R) so that it is
// exactly 128 pixels wide: lane l owns the 4-pixel word of columns 4l..4l+3
// of every row, and each of the 8 consumer warps owns a band of consecutive
// rows.
// Per item:
//   1. The producer (one warp) claims the item, decodes it, computes its
//      constants and TMA loads the region plus the 3-pixel circle halo (box
//      144 x TH+2R+6) into one of two image buffers; the other buffer is
//      loading the next item meanwhile (produce_tiles).
//   2. Coarse test on every score-region pixel of the warp's band, 4 pixels
//      per lane (runs of the eight even circle points), pixels outside the
//      testable area masked off; one warp
//      scan places each lane's kept pixels in the warp's queue, written by a
//      two-ended bit walk as raw codes (coarse_and_compact).
//   3. Each warp runs the full segment test on its queue and compacts the
//      corners in place, then scores the corners and writes the scores into
//      the score tile.
//   4. Once its two neighbouring warps have written their scores (the NMS
//      reads up to R rows of theirs; per-warp mbarriers, see neighbours_wait),
//      (2R+1)x(2R+1) NMS on the corner list (for R > 1 the nearest ring
//      first, the outer rings on its survivors); each survivor folds its
//      packed key into the global cell key with a 64-bit max reduction.
// ---------------------------------------------------------------------------
constexpr int kTileW = 120;  // output pixels per tile row, every variant

template <int TH, int R = 1>
struct TileGeom {
    static constexpr int TW = kTileW;      // output pixels per tile row
    static constexpr int SW = 128;         // score-region width (x0-4 .. x0+124)
    static constexpr int SR = TH + 2 * R;  // score-region rows (y0-R .. y0+TH+R): NMS radius R
    static constexpr int BW = 144;         // TMA box width (16-byte multiple)
    static constexpr int BH = SR + 6;      // box rows y0-R-3 .. y0+TH+R+3
    static constexpr int BOX = BW * BH;
    static constexpr int BOXA = (BOX + 127) / 128 * 128;
    static constexpr int WARPS = 8;
    static constexpr int PPW = SR / 2 / WARPS;  // row pairs per warp
    static constexpr int QCAP = PPW * 2 * SW;   // per-warp queue capacity (every pixel)
    static constexpr int NBUF = 2;              // image buffers in the TMA ring
    static constexpr int IMG_OFF = 0;
    static constexpr int SC_OFF = NBUF * BOXA;
    static constexpr int Q_OFF = SC_OFF + SR * SW * 2;
    static constexpr int SMEM = Q_OFF + WARPS * QCAP * 2 + 128;  // +128: base alignment slack
    static_assert(SR % (2 * WARPS) == 0, "row pairs must split evenly over the warps");
    static_assert(BH <= 256, "TMA box limit");
    static_assert(R >= 1 && R <= 4, "the 4-pixel column ring holds NMS radii up to 4");
};

constexpr int kConsumers = 256;             // 8 warps that detect
constexpr int kThreads = kConsumers + 32;   // + 1 producer warp (items, TMA)

// What the consumers need of an item, written by the producer next to the
// image buffer it fills.
struct ItemInfo {
    int32_t id;            // item index; >= n_items ends the consumers' loop
    int32_t level, x0, y0;
    int32_t wk, hk, gw, gh;
    uint32_t magic;                    // cell magic of the level
    int32_t xoff;                      // box column of score column 0
    int32_t row_lo, row_hi, xlo, xhi;  // testable score rows, kept score columns
    uint64_t* keys;
};

// The constants of a tile whose x0, y0, wk and hk are set: score column 0 is
// level x = x0 - 4 and box column 0 is (x0 - 8) & ~15; score row r is level
// y = y0 - R + r; testable pixels are 3 <= x < Wk - 3, 3 <= y < Hk - 3; the NMS
// reads score columns 4 - R .. 123 + R only.
template <int TH, int R>
__device__ __forceinline__ void tile_constants(ItemInfo& in) {
    in.xoff = in.x0 - 4 - ((in.x0 - 8) & ~15);
    in.row_lo = max(0, 3 - in.y0 + R);
    in.row_hi = min(TileGeom<TH, R>::SR, in.hk - 3 - in.y0 + R);
    in.xlo = max(4 - R, 7 - in.x0);
    in.xhi = min(124 + R, in.wk + 1 - in.x0);
}

// Bit 7 of byte j set when xlo <= 4 lane + j < xhi: byte j of cols4 + (128 - x)
// reaches bit 7 exactly when 4 lane + j >= x (all values below 256: no carries
// between bytes).
__device__ __forceinline__ uint32_t kept_columns(const ItemInfo& in, int lane) {
    const uint32_t cols4 = (uint32_t)(4 * lane) * 0x01010101u + 0x03020100u;
    return (cols4 + (uint32_t)(0x80 - in.xlo) * 0x01010101u) & ~(cols4 + (uint32_t)(0x80 - in.xhi) * 0x01010101u) &
           0x80808080u;
}

// upper_index by a whole warp (all lanes call it with the same arguments):
// 32 entries per step, so 1024 entries take two dependent loads instead of ten.
__device__ __forceinline__ int upper_index_warp(const int32_t* a, int n, int v, int lane) {
    int lo = 0, len = n;
    while (len > 1) {  // the answer lies in [lo, lo + len)
        const int step = (len + 31) / 32, o = lane * step;
        const uint32_t le = __ballot_sync(0xFFFFFFFFu, o < len && a[lo + o] <= v);
        const int k = 31 - __clz(le);  // a[lo] <= v: bit 0 is set
        lo += k * step;
        len = min(step, len - k * step);
    }
    return lo;
}

// Score-region index of a raw walk code (w << 10 | lane << 5 | bit b) of the
// warp whose rows start at r0: row r0 + 8w + (b & 7), column 4 lane + (b >> 3);
// (code >> 3) & 0x7F is that column, (code >> 7) & ~7 is 8w.
__device__ __forceinline__ int walk_code_index(uint32_t code, int r0) {
    return (int)(((uint32_t)r0 + (code & 7u) + ((code >> 7) & ~7u)) << 7) + (int)((code >> 3) & 0x7Fu);
}

// bits 7, 15, 23, 31 -> bits 28..31: the product's other terms stay below bit 28
__device__ __forceinline__ uint32_t nibble(uint32_t keep) { return (keep * 0x00204081u) >> 28; }

// Coarse test (the CCRF of Algorithm 1) over this warp's score rows,
// appending the kept pixels (as raw walk codes) to the warp's queue; returns
// the queue length.
//
// Warp w owns the 2*PPW score rows starting at r0 = 2*PPW*w; lane l owns the
// 4-pixel word of score columns 4l .. 4l+3 in every one of them, so a row is
// one conflict-free 128-byte read per warp.  The rule: an arc of n >= 9
// contiguous points holds floor(n/2) cyclically consecutive of the eight even
// circle points (compass points and the (+-2, +-2) diagonals), all darker or
// all brighter and so all with |I_x - I_c| > t.  A pixel is kept when 4 (n =
// 9), 5 (n = 10, 11) or 6 (n >= 12) consecutive even points differ from the
// centre by more than t; without EIGHT, when two adjacent compass points do.
// No corner is dropped.  On the mixed batch's recipe at t = 10, n = 10 the run
// of 5 keeps 4.9 % of the level-0 pixels where the two compass points keep
// 19.5 %; at t = 20, n = 12 the run of 6 keeps 0.2 / 3.4 / 10 % of levels
// 0 / 1 / 2 where three compass points keep 0.9 / 8.7 / 22 %.
//
// Each comparison is made once and serves two pixels: rows y and y+3 of a
// column give the S flag of row y and the N flag of row y+3; columns x and
// x+3 of a row give the E flag of x and the W flag of x+3; (x, y)-(x+2, y+2)
// is SE of the first and NW of the second, and (x, y)-(x+2, y-2) is NE of the
// first and SW of the second.  A row thus costs two word loads, two byte
// permutes and four compares.  The flags of a lane gather in words of eight
// rows (bit 8j + i = row i, column 4l + j), so the second pixel's flags are
// the same words a few rows later (one running word per comparison,
// read at two points) and, where the columns differ, byte-permuted with the
// word of the lane to the left: three shuffles and the rule itself once per
// eight rows instead of once per row.  The kernel is bound by the ALU pipe
// (logic, shifts, permutes: one instruction every two cycles) and by issue,
// and this test is half of its ALU work: with the rule and the shuffles per
// row the mixed batch took 107.1 M warp instructions and 133.7 us, so 94.0 M
// and 117.5 us (96.7 M and 120 us with the producer's whole-warp decoding).
// Lane 0 has no lane to its left: its W flags of columns 0..2 and NW / SW
// flags of columns 0, 1 count as set, which keeps more, never fewer.
//
// One warp scan of the popcounts places each lane's run in the queue, and each
// lane writes its pixels by walking its set bits, from both ends
// at once, as raw codes.  (Spreading the
// bits over the warp first, by a skewed bit transpose, balances the walk but
// scatters the queue, and the full test's circle reads then conflict in
// shared memory: slower.)
// vm: bit 7 of byte j set when column 4l + j is inside the columns NMS reads.
template <bool HIGH_T, int TH, int R, bool EIGHT = true>
__device__ __forceinline__ int coarse_and_compact(const uint8_t* img, uint16_t* queue, int xw, uint32_t k7,
                                                  int n_arc, int warp, int lane, int row_lo, int row_hi, uint32_t vm,
                                                  uint32_t* status = nullptr) {
    using G = TileGeom<TH, R>;
    constexpr int RW = G::BW / 4;      // words per box row
    constexpr int RPW = 2 * G::PPW;    // score rows per warp
    constexpr int NW = (RPW + 7) / 8;  // mask words per lane
    static_assert(RPW == 4 || RPW % 8 == 0, "a word holds eight rows, or the only four");
    constexpr uint32_t kFull = 0xFFFFFFFFu;
    const int r0 = RPW * warp;
    // a band with no testable row (below or above the level) keeps nothing
    if (row_hi <= r0 || row_lo >= r0 + RPW) return 0;
    // this lane's word in box row r0 (score row r is box row r + 3)
    const uint32_t* col = reinterpret_cast<const uint32_t*>(img) + r0 * RW + xw + lane;
    // One pass down the rows: step jj reads box row r0 + jj and makes the
    // comparisons that it completes.  wv holds the vertical ones of box rows
    // (i, i+3), w1 and w2 the diagonal ones of box rows (i+1, i+3), we the
    // horizontal ones of box row i + 3, for i up to jj - 3.
    uint32_t C[RPW + 6], R2[RPW + 6];
    uint32_t wv = 0u, w1 = 0u, w2 = 0u, we = 0u;
    uint32_t fn[NW], fs[NW], fe[NW], fne[NW], fse[NW], fsw[NW], fnw[NW];
#pragma unroll
    for (int jj = 0; jj < RPW + 6; ++jj) {
        C[jj] = col[jj * RW];
        uint32_t rw = 0u;
        if ((EIGHT && jj >= 1 && jj < RPW + 5) || (jj >= 3 && jj < RPW + 3)) rw = col[jj * RW + 1];
        if (EIGHT) R2[jj] = __byte_perm(C[jj], rw, 0x5432);
        if (jj < 3) continue;
        const int i = jj - 3;
        // the flags of score rows 8w .. 8w+7 are complete (and at the top of
        // the word) once the row that holds row 8w + 7, or the last, is in
        const auto done = [](int row) { return row >= 0 && row < RPW && ((row & 7) == 7 || row == RPW - 1); };
        wv = push_row(wv, gt_flags<HIGH_T>(C[i], C[jj], k7));
        if (done(i)) fn[i / 8] = wv;
        if (done(i - 3)) fs[(i - 3) / 8] = wv;
        if (i < RPW) {
            we = push_row(we, gt_flags<HIGH_T>(C[jj], __byte_perm(C[jj], rw, 0x6543), k7));
            if (done(i)) fe[i / 8] = we;
        }
        if (EIGHT && i < RPW + 2) {
            w1 = push_row(w1, gt_flags<HIGH_T>(C[jj - 2], R2[jj], k7));
            w2 = push_row(w2, gt_flags<HIGH_T>(C[jj], R2[jj - 2], k7));
            if (done(i)) {
                fnw[i / 8] = w1;
                fne[i / 8] = w2;
            }
            if (done(i - 2)) {
                fse[(i - 2) / 8] = w1;
                fsw[(i - 2) / 8] = w2;
            }
        }
    }
    uint32_t m[NW];
#pragma unroll
    for (int w = 0; w < NW; ++w) {
        // columns x - 3 and x - 2 of the flags that belong to the pixel on their right
        const auto from_left = [&](uint32_t f) {
            const uint32_t l = __shfl_up_sync(kFull, f, 1);
            return lane == 0 ? kFull : l;
        };
        const uint32_t fw = __byte_perm(from_left(fe[w]), fe[w], 0x4321);
        if (EIGHT) {
            const uint32_t nw = __byte_perm(from_left(fnw[w]), fnw[w], 0x5432);
            const uint32_t sw = __byte_perm(from_left(fsw[w]), fsw[w], 0x5432);
            const uint32_t f[8] = {fn[w], fne[w], fe[w], fse[w], fs[w], sw, fw, nw};
            if (n_arc == 9) {  // uniform
                // the 8 runs of four, grouped by their middle three around a diagonal
                const uint32_t xne = f[0] & f[1] & f[2], xse = f[2] & f[3] & f[4], xsw = f[4] & f[5] & f[6],
                               xnw = f[6] & f[7] & f[0];
                m[w] = ((xne | xsw) & (f[3] | f[7])) | ((xse | xnw) & (f[1] | f[5]));
            } else if (n_arc < 12) {
                m[w] = run_of_even<5>(f);
            } else {
                m[w] = run_of_even<6>(f);
            }
        } else {  // two adjacent: (N|S) & (E|W)
            m[w] = (fn[w] | fs[w]) & (fe[w] | fw);
        }
    }
    // a word of four rows holds them in the upper half of each byte
    if constexpr (RPW < 8) m[0] >>= 8 - RPW;
    // rows outside the testable area and columns outside the NMS region
    const uint32_t cols = ((vm >> 7) & 0x01010101u) * 0xFFu;
#pragma unroll
    for (int w = 0; w < NW; ++w) {
        constexpr int kRows = RPW < 8 ? RPW : 8;
        const int lo = min(max(row_lo - r0 - 8 * w, 0), 8), hi = min(max(row_hi - r0 - 8 * w, 0), kRows);
        const uint32_t rows = ((0xFFu << lo) & ~(0xFFu << hi) & 0xFFu) * 0x01010101u;
        m[w] &= rows & cols;
    }
    int cnt = 0;
#pragma unroll
    for (int w = 0; w < NW; ++w) cnt += __popc(m[w]);
    int incl = cnt;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(kFull, incl, o);
        if (lane >= o) incl += y;
    }
    int pos = incl - cnt;
    // bit b of word w stands for row r0 + 8w + (b & 7), column 4l + (b >> 3)
#pragma unroll
    for (int w = 0; w < NW; ++w) {
        uint32_t mw = m[w];
        // the highest and the lowest set bit per step: half the steps, and
        // two chains that do not depend on each other.  The queue takes the
        // raw code w << 10 | lane << 5 | bit, which the full test turns into
        // the pixel (walk_code_index): the walk is as slow as its busiest
        // lane, the full test is balanced.
        const int cbase = (w << 10) | (lane << 5);
        while (mw) {
            const int bh = 31 - __clz(mw);
            const uint32_t lowbit = mw & (0u - mw);
            const int bl = 31 - __clz(lowbit);
            const uint32_t hb = 1u << bh;
            mw &= (mw - 1u) & ~hb;
            if (vio_guard(pos < G::QCAP, status)) queue[pos] = (uint16_t)(cbase | bh);
            const bool two = lowbit != hb;
            if (two && vio_guard(pos + 1 < G::QCAP, status)) queue[pos + 1] = (uint16_t)(cbase | bl);
            pos += two ? 2 : 1;
        }
    }
    return __shfl_sync(kFull, incl, 31);
}

// Consumer warps synchronise with their neighbours only.  Warp w owns score
// rows [2*PPW*w, 2*PPW*(w+1)) and its NMS reads R <= 2*PPW rows beyond them,
// so only warps w-1 and w+1 read its rows.  Per tile t each warp arrives on
// sc_bar[w] once its scores are written and on nms_bar[w] once its NMS is
// done (one arrival per phase, phase t for tile t).  Before its NMS a warp
// waits for phase t of its neighbours' sc_bar; before writing the scores of
// tile t (its own rows only) it waits for phase t-1 of its neighbours'
// nms_bar and zeroes its rows.  A warp can thus run at most one phase ahead
// of a neighbour, which keeps the parity waits exact.  Returns false on a
// timed-out wait (status set).
__device__ __forceinline__ bool neighbours_wait(uint64_t* bars, int warp, int n_warps, uint32_t parity, int lane,
                                                uint32_t* status) {
    const bool ok = (warp == 0 || mbar_wait_bounded(&bars[warp - 1], parity, kWaitLimitNs)) &&
                    (warp == n_warps - 1 || mbar_wait_bounded(&bars[warp + 1], parity, kWaitLimitNs));
    if (!ok && lane == 0) atomicOr(status, kStatusTimeout);
    return ok;
}

// Start of a tile's score writes (see neighbours_wait).  T: the tile's
// element type (rows of G::SW elements).
template <int TH, int R, typename T>
__device__ __forceinline__ bool own_rows_reset(uint64_t* nms_bars, int t, T* tile, int warp, int lane,
                                               uint32_t* status) {
    using G = TileGeom<TH, R>;
    static_assert(2 * G::PPW * G::WARPS == G::SR, "warps own all score rows");
    static_assert(R <= 2 * G::PPW, "the NMS reads the rows of adjacent warps only");
    constexpr int N16 = 2 * G::PPW * G::SW * (int)sizeof(T) / 16;  // 16-byte words per warp
    static_assert(N16 % 32 == 0, "whole 16-byte stores per lane");
    if (t == 0) return true;  // zeroed at kernel start
    if (!neighbours_wait(nms_bars, warp, G::WARPS, (t - 1) & 1, lane, status)) return false;
    uint4* own = reinterpret_cast<uint4*>(tile + 2 * G::PPW * warp * G::SW);
#pragma unroll
    for (int j = 0; j < N16 / 32; ++j) own[lane + 32 * j] = make_uint4(0u, 0u, 0u, 0u);
    __syncwarp();
    return true;
}

// Producer of the detect kernels (one warp): takes work items (the CTA's own
// index first, then from the counter, claimed one ahead of their use), decodes
// each into the tile it covers, and issues the TMA load of the tile and its
// halo into the next buffer of the ring once the consumer warps have released
// it.  An item index >= n_items tells the consumers to stop.
//
// Decoding is a chain of dependent loads (the tile table, the frame), about
// 2,400 cycles by one thread and after the release, which the consumers then
// waited for on top of the load itself: 2,100 of 7,950 cycles per tile on 4K
// frames with few corners.  It is done by the warp and before the wait for the
// release (8 4K frames, FAST-12: 107.5 -> 101.8 us a call, 96 now; 64 mixed
// frames 148.3 -> 145.5 us, 138 now).
//
// The pyramid's levels are written by the kernel before this one, which may
// still be running (programmatic dependent launch); a level-0 tile reads the
// caller's frame and need not wait for it, unless that kernel also uploads the
// frame.
template <int TH, int R>
__device__ __forceinline__ void produce_tiles(const CallView& cv, const int32_t* tiles, int32_t* counter,
                                              uint32_t* status, ItemInfo* info, uint64_t* full_bar,
                                              uint64_t* empty_bar, uint8_t* smem, int lane) {
    using G = TileGeom<TH, R>;
    constexpr int NB = G::NBUF;
    const int n_items = cv.h->n_items, n = cv.h->n_frames, L = cv.h->levels;
    int claimed = 0;  // lane 0's
    bool pyramid_done = false;
    for (int t = 0;; ++t) {
        const int b = t % NB;
        const int it = t == 0 ? (int)blockIdx.x : (int)gridDim.x + __shfl_sync(0xFFFFFFFFu, claimed, 0);
        if (lane == 0 && it < n_items) claimed = atomicAdd(counter, 1);
        ItemInfo in = {};
        in.id = it;
        const CUtensorMap* map = nullptr;
        if (it < n_items) {
            // entry j = (L-1-k) * n + f of the tile table (coarsest level first)
            const int j = upper_index_warp(tiles, n * L, it, lane);
            const int f = j % n;
            in.level = L - 1 - j / n;
            const FrameDesc& fd = cv.fds[f];
            const uint8_t* uploaded = fd.src0;
            in.gw = fd.gw;
            in.gh = fd.gh;
            in.keys = fd.keys;
            in.wk = fd.w >> in.level;
            in.hk = fd.h >> in.level;
            in.magic = cv.h->cell_magic[in.level];
            const int ti = it - tiles[j], ntx = (in.wk + kTileW - 1) / kTileW;
            const int ty = ti / ntx;
            in.x0 = (ti - ty * ntx) * G::TW;
            in.y0 = ty * TH;
            // computed once here instead of by every consumer warp
            tile_constants<TH, R>(in);
            map = in.level == 0 ? &cv.maps0[f] : &cv.mapsk[f * (kMaxLevels - 1) + in.level - 1];
            if (lane == 0) fence_tensormap_acquire(map);
            if (!pyramid_done && (in.level > 0 || uploaded)) {
                griddep_wait();
                pyramid_done = true;
            }
        }
        if (t >= NB && !mbar_wait_bounded(&empty_bar[b], ((t / NB) - 1) & 1, kWaitLimitNs)) {
            if (lane == 0) atomicOr(status, kStatusTimeout);
            return;
        }
        if (lane == 0) {
            info[b] = in;
            if (it >= n_items) {
                mbar_arrive(&full_bar[b]);
            } else {
                mbar_arrive_expect_tx(&full_bar[b], G::BOX);
                tma_load_2d(smem + G::IMG_OFF + b * G::BOXA, map, &full_bar[b], (in.x0 - 8) & ~15, in.y0 - R - 3);
            }
        }
        if (it >= n_items) return;
    }
}

// NMS ring K around the score at q (row pitch SW): true when s is >= the
// 8K scores at Chebyshev distance K.
template <int K, int SW>
__device__ __forceinline__ bool ring_max(const uint16_t* q, uint32_t s) {
    bool ok = true;
#pragma unroll
    for (int dx = -K; dx <= K; ++dx) ok &= (s >= q[-K * SW + dx]) & (s >= q[K * SW + dx]);
#pragma unroll
    for (int dy = -K + 1; dy <= K - 1; ++dy) ok &= (s >= q[dy * SW - K]) & (s >= q[dy * SW + K]);
    return ok;
}

// One NMS pass of a wide window: keeps the corners of queue[0, n) that pass
// ring K, compacted in place; returns how many.
template <int K, int SW>
__device__ __forceinline__ int nms_ring_pass(uint16_t* queue, int n, const uint16_t* sc, int lane, uint32_t lt_mask) {
    int np = 0;
    for (int e0 = 0; e0 < n; e0 += 32) {
        const int e = e0 + lane;
        int idx = 0;
        bool ok = false;
        if (e < n) {
            idx = queue[e];
            ok = ring_max<K, SW>(sc + idx, sc[idx]);
        }
        const uint32_t bm = __ballot_sync(0xFFFFFFFFu, ok);
        if (ok) queue[np + __popc(bm & lt_mask)] = (uint16_t)idx;
        np += __popc(bm);
    }
    return np;
}

// Full segment test of a warp's queue (raw walk codes); the corners, as score
// indices, are compacted in place.  Returns how many.
template <int MODE, int TH, int R>
__device__ __forceinline__ int full_test(const uint8_t* img_base, uint16_t* queue, int total, int warp, int lane,
                                         uint32_t lt_mask, int thresh, int n_arc, uint32_t* status) {
    using G = TileGeom<TH, R>;
    int ncorner = 0;
    for (int e0 = 0; e0 < total; e0 += 32) {
        const int e = e0 + lane;
        uint32_t s = 0;
        int idx = 0;
        if (e < total && vio_guard(e < G::QCAP, status)) {
            idx = walk_code_index(queue[e], 2 * G::PPW * warp);
            // box offset of score-region pixel (idx >> 7, idx & 127); the
            // score is taken below, on the compacted corners only
            if (vio_guard(idx < G::SR * G::SW, status))
                s = eval_corner<MODE, G::BW, false>(img_base + idx + 16 * (idx >> 7), thresh, n_arc);
        }
        const uint32_t cm = __ballot_sync(0xFFFFFFFFu, s != 0);
        if (s) queue[ncorner + __popc(cm & lt_mask)] = (uint16_t)idx;
        ncorner += __popc(cm);
    }
    return ncorner;
}

// Scores of the corners queue[0, ncorner) into the score tile.
template <int MODE, int TH, int R>
__device__ __forceinline__ void score_corners(const uint8_t* img_base, const uint16_t* queue, int ncorner, int lane,
                                              int thresh, int n_arc, uint16_t* sc) {
    using G = TileGeom<TH, R>;
    for (int e = lane; e < ncorner; e += 32) {
        const int idx = queue[e];
        const uint8_t* p = img_base + idx + 16 * (idx >> 7);
        // MT of a known corner needs no segment test: the largest window
        // minimum alone (see eval_corner)
        sc[idx] = (uint16_t)(MODE == 0   ? sad_b<G::BW>(p)
                             : MODE == 2 ? mt_of_corner<G::BW>(p, n_arc)
                                         : eval_corner<MODE, G::BW, true>(p, thresh, n_arc));
    }
}

// NMS on the corners queue[0, ncorner), cell maximum by a 64-bit max reduction
// per survivor.  A window wider than 3x3 is tested ring by ring: the 8
// nearest neighbours of every corner first, which suppress most
// corners, then each further ring on the corners that passed the
// rings inside it (compacted to the front of the queue).
template <int TH, int R>
__device__ __forceinline__ void nms_corners(uint16_t* queue, int ncorner, const uint16_t* sc, int lane,
                                            uint32_t lt_mask, const ItemInfo& in, uint32_t* status) {
    using G = TileGeom<TH, R>;
    const int k = in.level, Wk = in.wk, x0 = in.x0, y0 = in.y0;
    const uint32_t magic = in.magic;
    int nnms = ncorner;
    if constexpr (R > 1) {
        int npass = 0;
        for (int e0 = 0; e0 < ncorner; e0 += 32) {
            const int e = e0 + lane;
            int idx = 0;
            bool ok = false;
            if (e < ncorner) {
                idx = queue[e];
                const int sr = idx >> 7, scx = idx & 127;
                if (scx >= 4 && scx < 4 + G::TW && sr >= R && sr < R + TH) {
                    const uint16_t* q = sc + idx;
                    const uint32_t s = q[0];
                    ok = true;
#pragma unroll
                    for (int dy = -1; dy <= 1; ++dy)
#pragma unroll
                        for (int dx = -1; dx <= 1; ++dx)
                            if (dy != 0 || dx != 0) ok &= s >= q[dy * G::SW + dx];
                }
            }
            const uint32_t bm = __ballot_sync(0xFFFFFFFFu, ok);
            if (ok) queue[npass + __popc(bm & lt_mask)] = (uint16_t)idx;
            npass += __popc(bm);
        }
        nnms = npass;
        if constexpr (R > 2) nnms = nms_ring_pass<2, G::SW>(queue, nnms, sc, lane, lt_mask);
        if constexpr (R > 3) nnms = nms_ring_pass<3, G::SW>(queue, nnms, sc, lane, lt_mask);
    }
    for (int e0 = 0; e0 < nnms; e0 += 32) {
        const int e = e0 + lane;
        uint32_t cell_id = 0xFFFFFFFFu;
        uint32_t hi = 0, lo = 0;
        if (e < nnms) {
            const int idx = queue[e];
            const int sr = idx >> 7, scx = idx & 127;
            // (with R > 1 the first pass kept corners inside the tile only)
            const bool inside = R > 1 || (scx >= 4 && scx < 4 + G::TW && sr >= R && sr < R + TH);
            if (inside) {
                // (2R+1) x (2R+1) neighbourhood: keep when >= every neighbour
                // (for R > 1 the outermost ring; the passes above did the rest)
                const uint16_t* q = sc + idx;
                const uint32_t s = q[0];
                bool keep = true;
                if constexpr (R == 1) {
                    // (this loop form, not ring_max<1>: the MT kernel is
                    // 5 % slower with the latter)
#pragma unroll
                    for (int dy = -1; dy <= 1; ++dy)
#pragma unroll
                        for (int dx = -1; dx <= 1; ++dx)
                            if (dy != 0 || dx != 0) keep &= s >= q[dy * G::SW + dx];
                } else {
                    keep = ring_max<R, G::SW>(q, s);
                }
                if (keep) {
                    const uint32_t x = (uint32_t)(x0 - 4 + scx), y = (uint32_t)(y0 - R + sr);
                    const uint32_t cx = __umulhi(x, magic), cy = __umulhi(y, magic);
                    if (vio_guard(cx < (uint32_t)in.gw && cy < (uint32_t)in.gh, status)) {
                        cell_id = cy * (uint32_t)in.gw + cx;
                        hi = s;
                        lo = 0xFFFFFFFFu - (((uint32_t)k << 28) | (y * (uint32_t)Wk + x));
                    }
                }
            }
        }
        // each survivor folds its key into the cell's (a warp-wide max
        // for survivors sharing a cell first was 2.6 % slower: its votes,
        // shuffle and reductions form one long dependent chain)
        if (hi != 0) red_max_u64(reinterpret_cast<unsigned long long*>(&in.keys[cell_id]),
                                 ((unsigned long long)hi << 32) | lo);
    }
}

template <int TH, int MODE, int R = 1>
__global__ void __launch_bounds__(kThreads, 4) fast_nms_cell_kernel(const uint8_t* __restrict__ call,
                                                                 int32_t* __restrict__ counter,
                                                                 uint32_t* __restrict__ status) {
    using G = TileGeom<TH, R>;
    constexpr int NB = G::NBUF;
    extern __shared__ __align__(128) uint8_t smem_raw[];
    __shared__ uint64_t full_bar[NB], empty_bar[NB], sc_bar[G::WARPS], nms_bar[G::WARPS];
    __shared__ ItemInfo info[NB];
    // the tile table, copied once so that the producer's search stays on chip
    constexpr int kTileCache = 512;
    __shared__ int32_t tiles_sh[kTileCache];
    // TMA destinations must be 128-byte aligned
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 127) & ~uintptr_t(127));
    uint16_t* sc = reinterpret_cast<uint16_t*>(smem + G::SC_OFF);

    const CallView cv(call);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int n_items = cv.h->n_items;

    if (tid == 0) {
        for (int b = 0; b < NB; ++b) {
            mbar_init(&full_bar[b], 1);
            mbar_init(&empty_bar[b], kConsumers / 32);  // one arrival per consumer warp
        }
        for (int w = 0; w < G::WARPS; ++w) {
            mbar_init(&sc_bar[w], 1);
            mbar_init(&nms_bar[w], 1);
        }
        fence_barrier_init();
    }
    // the score tile starts zero; only corners are written, and each warp
    // zeroes its rows before the next tile's writes
    for (int i = tid; i < G::SR * G::SW / 8; i += kThreads) reinterpret_cast<uint4*>(sc)[i] = make_uint4(0, 0, 0, 0);
    // the decode kernel adds up the per-frame counts from zero
    if (blockIdx.x == 0 && cv.h->counts)
        for (int f = tid; f < cv.h->n_frames; f += kThreads) cv.h->counts[f] = 0;
    const int n_tiles = cv.h->n_frames * cv.h->levels + 1;
    const bool cached = n_tiles <= kTileCache;
    if (cached)
        for (int i = tid; i < n_tiles; i += kThreads) tiles_sh[i] = cv.tiles[i];
    __syncthreads();

    griddep_launch_dependents();
    if (warp == kConsumers / 32) {
        produce_tiles<TH, R>(cv, cached ? tiles_sh : cv.tiles, counter, status, info, full_bar, empty_bar, smem, lane);
        return;
    }

    // ---- consumer warps ----
    uint16_t* queue = reinterpret_cast<uint16_t*>(smem + G::Q_OFF) + warp * G::QCAP;
    const uint32_t lt_mask = (1u << lane) - 1u;
    const int thresh = cv.h->thresh, n_arc = cv.h->arc;
    const bool high_t = thresh >= 128;
    const uint32_t k7 = (uint32_t)((high_t ? 255 : 127) - thresh) * 0x01010101u;

    for (int t = 0;; ++t) {
        const int b = t % NB;
        if (!mbar_wait_bounded(&full_bar[b], (t / NB) & 1, kWaitLimitNs)) {
            if (lane == 0) atomicOr(status, kStatusTimeout);
            return;
        }
        const ItemInfo in = info[b];
        if (in.id >= n_items) break;
        const uint8_t* img = smem + G::IMG_OFF + b * G::BOXA;
        const int xoff = in.xoff;

        // 2. coarse test + compaction
        const uint32_t vm = kept_columns(in, lane);
        const int total =
            high_t ? coarse_and_compact<true, TH, R>(img, queue, xoff / 4, k7, n_arc, warp, lane, in.row_lo, in.row_hi,
                                                     vm, status)
                   : coarse_and_compact<false, TH, R>(img, queue, xoff / 4, k7, n_arc, warp, lane, in.row_lo,
                                                      in.row_hi, vm, status);
        __syncwarp();

        // 3. full test on this warp's queue
        const uint8_t* img_base = img + 3 * G::BW + xoff;
        const int ncorner = full_test<MODE, TH, R>(img_base, queue, total, warp, lane, lt_mask, thresh, n_arc, status);
        if (!own_rows_reset<TH, R>(nms_bar, t, sc, warp, lane, status)) return;
        score_corners<MODE, TH, R>(img_base, queue, ncorner, lane, thresh, n_arc, sc);
        // this warp is done with the image buffer, and its scores are written
        __syncwarp();
        if (lane == 0) {
            mbar_arrive(&empty_bar[b]);
            mbar_arrive(&sc_bar[warp]);
        }
        // the neighbours' scores of this tile are written
        if (!neighbours_wait(sc_bar, warp, G::WARPS, t & 1, lane, status)) return;

        // 4. NMS and cell maximum
        nms_corners<TH, R>(queue, ncorner, sc, lane, lt_mask, in, status);
        // this warp's NMS reads of the score tile are done
        __syncwarp();
        if (lane == 0) mbar_arrive(&nms_bar[warp]);
    }
}

// The record of a non-empty cell key of cell c of a w x h frame (gw cells per
// row); reports a key that does not lie in its cell.
__device__ __forceinline__ int4 decode_key(uint64_t key, int c, int w, int h, int gw, int levels, uint32_t magic,
                                           uint32_t* status) {
    const uint32_t lin = 0xFFFFFFFFu - (uint32_t)key;
    const int k = (int)(lin >> 28);
    const uint32_t idx = lin & 0x0FFFFFFFu;
    const uint32_t wk = (uint32_t)(w >> k);
    const int y = (int)(idx / wk), x = (int)(idx - (uint32_t)y * wk);
    const int4 rec = make_int4(x << k, y << k, k, (int)(key >> 32));
    // consistency of the packed key with the cell it was folded into
    if (status && (k >= levels || rec.x >= w || rec.y >= h ||
                   __umulhi((uint32_t)rec.y, magic) * (uint32_t)gw + __umulhi((uint32_t)rec.x, magic) != (uint32_t)c))
        atomicOr(status, kStatusBadKey);
    return rec;
}

// ---------------------------------------------------------------------------
// Decode: one thread per cell of all frames turns its key into a record,
// clears the key for the next call and counts non-empty cells per frame
// (warp-aggregated; the fused kernel zeroed the counts).
// ---------------------------------------------------------------------------
static __global__ void __launch_bounds__(256) decode_kernel(const uint8_t* __restrict__ call, int32_t* __restrict__ counter) {
    const CallView cv(call);
    const int nf = cv.h->n_frames, total = cv.h->n_cells;
    int32_t* counts = cv.h->counts;
    uint32_t* status = cv.h->status;
    const uint32_t magic = cv.h->cell_magic[0];
    const int levels = cv.h->levels;
    const int lane = threadIdx.x & 31;
    // the cell prefix sums in shared memory when they fit (see pyramid_kernel)
    __shared__ int32_t cells_sh[kPrefixCache];
    const int32_t* cells = nf < kPrefixCache ? cells_sh : cv.cells;
    if (nf < kPrefixCache)
        for (int j = threadIdx.x; j <= nf; j += blockDim.x) cells_sh[j] = cv.cells[j];
    __syncthreads();
    // the cell keys are final once the detect kernel before this one has
    // completed; it may still be running (programmatic dependent launch), so
    // the cell's frame, which the call block holds since before, is found first
    bool keys_final = false;
    for (int base = blockIdx.x * blockDim.x; base < total; base += gridDim.x * blockDim.x) {
        const int i = base + threadIdx.x;
        int f = -1, c = 0, w = 1, h = 0, gw = 0;
        uint64_t* kp = nullptr;
        int4* out = nullptr;
        if (i < total) {
            f = upper_index(cells, nf, i);
            const FrameDesc& fd = cv.fds[f];
            c = i - cells[f];
            w = fd.w;
            h = fd.h;
            gw = fd.gw;
            kp = fd.keys + c;
            out = fd.out + c;
        }
        if (!keys_final) griddep_wait();
        keys_final = true;
        bool hit = false;
        if (i < total) {
            const uint64_t key = *kp;
            int4 rec = make_int4(-1, -1, -1, 0);
            if (key != 0) {
                rec = decode_key(key, c, w, h, gw, levels, magic, status);
                *kp = 0;
                hit = true;
            }
            *out = rec;
        }
        if (counts) {
            // lanes of one frame add their hits with one atomic
            uint32_t pend = __ballot_sync(0xFFFFFFFFu, f >= 0);
            while (pend) {
                const int leader = __ffs(pend) - 1;
                const int fl = __shfl_sync(0xFFFFFFFFu, f, leader);
                const uint32_t grp = __ballot_sync(0xFFFFFFFFu, f == fl);
                const uint32_t hits = __popc(__ballot_sync(0xFFFFFFFFu, f == fl && hit));
                if (lane == leader && hits) atomicAdd(&counts[fl], (int)hits);
                pend &= ~grp;
            }
        }
    }
    if (!keys_final) griddep_wait();
    if (blockIdx.x == 0 && threadIdx.x == 0) *counter = 0;
}

}  // namespace vio
