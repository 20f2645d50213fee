// Next step before the path: grayscale opening by a disk (Table I, "Morph.
// Open", by a 19x19 disk).  The disk of radius r is the set of integer
// offsets (dx, dy) with dx^2 + dy^2 <= r^2; pixels outside the image take no
// part.  Opening = dilation of the erosion, each by that disk: two streaming
// passes, through a plane of the pipe.
//
// One pass: a warp streams the input rows down a strip of 128 columns and a
// segment of rows, lane l holding columns 4l .. 4l + 3 as two pairs of 16-bit
// lanes, (4l, 4l + 2) and (4l + 1, 4l + 3), with the pixel in the high byte (the
// low bytes are left as they come: they cannot change the high byte of a
// minimum or a maximum).  A word of four pixels is then the second pair as it
// is, and any pair at another column is one byte permute of two words.
//  * A row enters a per-warp buffer of 4-pixel words with a halo of r columns;
//    a lane reads the words around it once and takes the chords of half-widths
//    0 .. r from them, which are nested: C_w = min(C_{w-1}, pair at -w, pair at
//    +w), one 3-input SIMD instruction each.
//  * Instead of keeping rows, a lane keeps one accumulator per output row that
//    the entering rows reach.  Rows enter two at a time, so an accumulator takes
//    both rows' chords in one 3-input instruction, and two output rows are
//    complete.  The loop over r + 1 such steps is unrolled, so that every
//    accumulator has a fixed register.
//  * Rows are fetched three or more steps ahead (one step: 126 us).
// 4096^2, r = 9: 53 us for both passes; 99 us with 64 columns per warp, a row per
// step and 16-bit pixels in shared memory, 176 us for 2047 x 1531 by the block
// form that odd widths and other radii took (29 us now).  Bound: instruction
// issue and latency, about 75 instructions per row and 128 columns (the 67 MB
// that both passes move take 10 us); 16 warps per SM by registers.
#include <algorithm>

#include "internal.cuh"
#include "morph.cuh"

namespace nucseg {

MORPH_PASS(9)

// Copies a plane whose rows start on no 4-byte boundary into rows of `pitch`
// bytes (a multiple of 16), padded with 255: 16 pixels per thread.
__global__ void __launch_bounds__(256) k_morph_pad(const uint8_t* __restrict__ src, uint8_t* __restrict__ dst, int W, int H,
                                                   int pitch) {
    const int cpr = pitch >> 4;
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= (long long)cpr * H) return;
    const int y = (int)(i / cpr), x = (int)(i - (long long)y * cpr) * 16, n = W - x;
    uint4 v = load_px16(src, W, H, x, y);
    if (n < 16) {
        const uint4 k = clip_px16(make_uint4(~0u, ~0u, ~0u, ~0u), n);
        v = make_uint4(v.x | ~k.x, v.y | ~k.y, v.z | ~k.z, v.w | ~k.w);
    }
    *reinterpret_cast<uint4*>(dst + (size_t)y * pitch + x) = v;
}

typedef void (*MorphPass)(const MorphArgs&, bool, int, cudaStream_t);
template <int R>
static MorphPass pass_of(int r) {
    if constexpr (R > MORPH_RMAX) {
        return nullptr;
    } else {
        return r == R ? &morph_pass<R> : pass_of<R + 1>(r);
    }
}

static bool morph_direct(const uint8_t* src, int W) { return ((reinterpret_cast<uintptr_t>(src) | (uintptr_t)W) & 3) == 0; }

void launch_morph_open(const uint8_t* src, uint8_t* dst, uint8_t* tmp, int W, int H, int r, int sms, cudaStream_t s,
                       Profiler* pf) {
    if (r == 0) {  // the disk is one pixel
        cudaMemcpyAsync(dst, src, (size_t)W * H, cudaMemcpyDeviceToDevice, s);
        return;
    }
    const MorphPass pass = pass_of<1>(r);
    const int tp = morph_pitch(W);
    MorphArgs a{src, tmp, W, tp, W, H, (W + MS_COLS - 1) / MS_COLS, 0, 0};
    if (!morph_direct(src, W)) {
        uint8_t* padded = tmp + (((size_t)tp * H + 255) & ~(size_t)255);
        const long long items = (long long)(tp >> 4) * H;
        pf->begin("morph_pad", s);
        k_morph_pad<<<(unsigned)((items + 255) / 256), 256, 0, s>>>(src, padded, W, H, tp);
        pf->end("morph_pad", s);
        a.src = padded;
        a.sp = tp;
    }
    pf->begin("morph_erode", s);
    pass(a, false, sms, s);
    pf->end("morph_erode", s);
    a.src = tmp;
    a.dst = dst;
    a.sp = tp;
    a.dp = W;
    pf->begin("morph_dilate", s);
    pass(a, true, sms, s);
    pf->end("morph_dilate", s);
}

}  // namespace nucseg
