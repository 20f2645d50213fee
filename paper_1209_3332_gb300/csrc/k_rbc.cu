// RBC detection (Table I "RBC detection": OpenCV colour operations and
// Vincent's MR; the paper gives no definition).  The reading computed here:
//   d = R - max(G, B) per pixel (red dominance);
//   marker = d >= t_hi, mask = d >= t_lo (0 <= t_lo <= t_hi <= 255);
//   RBC = the binary reconstruction by dilation, 8-connected, of the marker
//         under the mask: the mask components that hold a marker pixel.
// k_rbc_planes writes the marker and the mask as bit planes, 64x64 work tile
// by work tile, and whether a tile holds a marker pixel; the growth
// (k_grow.cu) then starts from those tiles only.  One warp per work tile: a
// lane takes 16 consecutive pixels of a row (three 16-byte loads of
// interleaved RGB where the rows allow it) in each of 8 steps of 8 rows, so
// the tile's words leave as whole sectors.  HBM-bound: 3 B read and 1/4 B
// written per pixel.
#include "internal.cuh"

namespace nucseg {

constexpr int RB_WARPS = 8;  // work tiles per CTA

__global__ void __launch_bounds__(RB_WARPS * 32) k_rbc_planes(const __grid_constant__ GrowLaunch G,
                                                              const uint8_t* __restrict__ rgb, size_t pitch, int t_lo,
                                                              int t_hi) {
    cudaTriggerProgrammaticLaunchCompletion();  // the growth may be prepared
    const int t = blockIdx.x * RB_WARPS + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (blockIdx.x == 0 && threadIdx.x == 0) grow_reset(G);
    if (t >= G.n_rt) return;
    const int W = G.tab.near[0].W, H = G.tab.near[0].H, rtx = (W + RT - 1) / RT, ty = t / rtx, tx = t - ty * rtx;
    const int q = lane & 3, x0 = tx * RT + 16 * q;
    unsigned any = 0;
#pragma unroll 2
    for (int i = 0; i < RT / 8; i++) {
        const int r = 8 * i + (lane >> 2), y = ty * RT + r;
        unsigned mk = 0, ms = 0;  // bit p: pixel x0 + p is in the marker, the mask
        if (y < H && x0 < W) {
            const uint8_t* src = rgb + (size_t)y * pitch + (size_t)x0 * 3;
            auto px = [&](int p, uint32_t r8, uint32_t g8, uint32_t b8) {
                const int d = (int)r8 - (int)max(g8, b8);
                mk |= (unsigned)(d >= t_hi) << p;
                ms |= (unsigned)(d >= t_lo) << p;
            };
            if (x0 + 16 <= W && (reinterpret_cast<uintptr_t>(src) & 15) == 0) {
                const uint4 a = __ldcs(reinterpret_cast<const uint4*>(src));
                const uint4 b = __ldcs(reinterpret_cast<const uint4*>(src) + 1);
                const uint4 c = __ldcs(reinterpret_cast<const uint4*>(src) + 2);
                const uint32_t w[12] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w, c.x, c.y, c.z, c.w};
                auto byte_at = [&](int k) -> uint32_t { return __byte_perm(w[k >> 2], 0u, 0x4440 | (k & 3)); };
#pragma unroll
                for (int p = 0; p < 16; p++) px(p, byte_at(3 * p), byte_at(3 * p + 1), byte_at(3 * p + 2));
            } else {
                const int n = min(16, W - x0);
                for (int p = 0; p < n; p++) px(p, src[3 * p], src[3 * p + 1], src[3 * p + 2]);
            }
        }
        reinterpret_cast<uint16_t*>(G.marker + (size_t)t * RT + r)[q] = (uint16_t)mk;
        reinterpret_cast<uint16_t*>(G.mask + (size_t)t * RT + r)[q] = (uint16_t)ms;
        any |= mk;
    }
    any = __any_sync(0xffffffffu, any != 0u);
    if (lane == 0) G.any[t] = (uint8_t)any;
}

void launch_rbc_planes(const GrowLaunch& G, const uint8_t* rgb, size_t pitch, int t_lo, int t_hi, cudaStream_t s,
                       Profiler* pf) {
    pf->begin("rbc_planes", s);
    k_rbc_planes<<<(G.n_rt + RB_WARPS - 1) / RB_WARPS, RB_WARPS * 32, 0, s>>>(G, rgb, pitch, t_lo, t_hi);
    pf->end("rbc_planes", s);
}

}  // namespace nucseg
