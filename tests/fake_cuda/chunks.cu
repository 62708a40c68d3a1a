// The pyramid kernel's chunk of a thread, for tests: blocks [first, first + n) of
// a w x h frame, 256 (column, row) pairs each; returns the frame's blocks.
#include "../../paper_2003_13493_gb300/csrc/vio_kernels.cuh"

extern "C" int fake_pyramid_chunks(int w, int h, int levels, int first, int n, int* out) {
    vio::FrameDesc f = {};
    f.w = w;
    f.h = h;
    uint8_t staged = 0;
    f.src0 = &staged;  // so that one level has blocks too
    const int blocks = vio::pyr_plan(f, levels);
    for (int b = first; b < first + n && b < blocks; ++b)
        for (int t = 0; t < 256; ++t) {
            const vio::PyrChunk c = vio::pyr_chunk(f, b, t);
            *out++ = c.tx;
            *out++ = c.ty;
        }
    return blocks;
}
