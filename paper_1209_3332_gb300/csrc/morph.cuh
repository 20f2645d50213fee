// One pass of the opening (see k_morph.cu), a template over the radius.
#pragma once
#include "internal.cuh"

namespace nucseg {

constexpr int MS_WARPS = 4, MS_COLS = 128, MS_SEG_MIN = 16;

// Input rows start on 4-byte boundaries, and the bytes of a row's last word that
// lie beyond the image hold the neutral value (255 for a minimum, 0 for a maximum).
struct MorphArgs {
    const uint8_t* src;
    uint8_t* dst;
    int sp, dp;      // row pitches (dp > W: rows padded to 4 bytes, the padding takes zeros)
    int W, H;
    int nstrip;      // strips of MS_COLS columns
    int seg, n;      // rows per segment, strips times segments (set at the launch)
};

__device__ __forceinline__ uint32_t morph2(bool mx, uint32_t a, uint32_t b) {
    uint32_t d;
    if (mx) asm("max.u16x2 %0, %1, %2;" : "=r"(d) : "r"(a), "r"(b));
    else asm("min.u16x2 %0, %1, %2;" : "=r"(d) : "r"(a), "r"(b));
    return d;
}
__device__ __forceinline__ uint32_t morph3(bool mx, uint32_t a, uint32_t b, uint32_t c) {
    return mx ? __vimax3_u16x2(a, b, c) : __vimin3_u16x2(a, b, c);
}

// steps ahead that rows are fetched: a divisor of the R + 1 unrolled steps, so
// that the words of a step have fixed registers, and 3 or more where there is one
__host__ __device__ constexpr int morph_ahead(int R) {
    for (int d = 3; d <= R; d++)
        if ((R + 1) % d == 0) return d;
    return R + 1;
}

template <int R, bool MAX>
__global__ void __launch_bounds__(MS_WARPS * 32) k_morph_stream(const MorphArgs g) {
    constexpr int K = 2 * R + 2;               // output rows that two entering rows reach
    constexpr int NH = (R + 3) / 4, A = 4 * NH;  // halo words per side
    constexpr int NW = 2 * NH + 1;             // words a lane reads per row
    constexpr uint32_t NEUTRAL = MAX ? 0u : 0xffffffffu;
    __shared__ uint32_t buf[MS_WARPS][2][32 + 2 * NH];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int gw = blockIdx.x * MS_WARPS + warp;
    if (gw >= g.n) return;  // whole warps only
    const int strip = gw % g.nstrip, seg = gw / g.nstrip, W = g.W, H = g.H;
    const int xs = strip * MS_COLS, ys = seg * g.seg, ye = min(H, ys + g.seg);
    const int t1 = ye + R;                     // input rows [ys - R, t1) reach the segment
    const int x0 = xs + 4 * lane;
    // this lane's words of a row: its own, and on the first 2 NH lanes one of the halo
    const int hw = lane < NH ? lane : 32 + lane, hx = xs - A + 4 * hw;
    const bool in0 = x0 < W, in1 = lane < 2 * NH && hx >= 0 && hx < W;
    const uint8_t* const p0 = g.src + x0;
    const uint8_t* const p1 = g.src + hx;
    auto fetch = [&](int t, const uint8_t* p, bool in) -> uint32_t {
        return in && t >= 0 && t < H && t < t1 ? __ldg(reinterpret_cast<const uint32_t*>(p + (size_t)t * g.sp)) : NEUTRAL;
    };
    uint32_t E[K], O[K];  // accumulators: columns 4l, 4l + 2 and 4l + 1, 4l + 3
#pragma unroll
    for (int k = 0; k < K; k++) E[k] = O[k] = NEUTRAL;
    constexpr int D = morph_ahead(R);
    uint32_t nw[D][2], nh[D][2];  // the words of the next D steps
#pragma unroll
    for (int d = 0; d < D; d++)
#pragma unroll
        for (int q = 0; q < 2; q++) {
            nw[d][q] = fetch(ys - R + 2 * d + q, p0, in0);
            nh[d][q] = fetch(ys - R + 2 * d + q, p1, in1);
        }
    // output: whole words, unless the caller's rows start on no 4-byte boundary
    const bool words = ((reinterpret_cast<uintptr_t>(g.dst) | (uintptr_t)g.dp) & 3) == 0;
    const uint32_t last = x0 + 4 > W && x0 < W ? (1u << (8 * (W - x0))) - 1u : 0xffffffffu;
    // half-width of the chord at distance d
    auto half = [](int d) constexpr {
        int w = 0;
        while ((w + 1) * (w + 1) + d * d <= R * R) w++;
        return w;
    };
    for (int tb = ys - R; tb < t1; tb += K) {
#pragma unroll
        for (int u = 0; u <= R; u++) {
            const int t = tb + 2 * u;
            if (t >= t1) break;
#pragma unroll
            for (int q = 0; q < 2; q++) {
                buf[warp][q][NH + lane] = nw[u % D][q];
                if (lane < 2 * NH) buf[warp][q][hw] = nh[u % D][q];
                nw[u % D][q] = fetch(t + 2 * D + q, p0, in0);
                nh[u % D][q] = fetch(t + 2 * D + q, p1, in1);
            }
            __syncwarp();
            uint32_t CE[2][R + 1], CO[2][R + 1];
#pragma unroll
            for (int q = 0; q < 2; q++) {
                uint32_t w[NW];
#pragma unroll
                for (int k = 0; k < NW; k++) w[k] = buf[warp][q][lane + k];
                // the pair (4l + d, 4l + d + 2)
                auto pair = [&](int d) -> uint32_t {
                    const int i = d + A, k = i >> 2;
                    switch (i & 3) {
                        case 0: return w[k] * 256u;
                        case 1: return w[k];
                        case 2: return __byte_perm(w[k], w[k + 1], 0x4020);
                        default: return __byte_perm(w[k], w[k + 1], 0x5030);
                    }
                };
                CE[q][0] = pair(0);
                CO[q][0] = pair(1);
#pragma unroll
                for (int wd = 1; wd <= R; wd++) {
                    CE[q][wd] = morph3(MAX, CE[q][wd - 1], pair(-wd), pair(wd));
                    CO[q][wd] = morph3(MAX, CO[q][wd - 1], pair(1 - wd), pair(1 + wd));
                }
            }
            __syncwarp();  // every lane has read the row buffers
            // output row t - R + j: row t at distance |j - R|, row t + 1 at |j - R - 1|
#pragma unroll
            for (int j = 0; j < K; j++) {
                const int k = (2 * u + j) % K;
                const int a = half(j < R ? R - j : j - R), b = half(j < R + 1 ? R + 1 - j : j - R - 1);
                if (j == 0) {
                    E[k] = morph2(MAX, E[k], CE[0][a]);
                    O[k] = morph2(MAX, O[k], CO[0][a]);
                } else if (j == K - 1) {
                    E[k] = CE[1][b];
                    O[k] = CO[1][b];
                } else if (j == K - 2) {
                    E[k] = morph2(MAX, CE[0][a], CE[1][b]);
                    O[k] = morph2(MAX, CO[0][a], CO[1][b]);
                } else {
                    E[k] = morph3(MAX, E[k], CE[0][a], CE[1][b]);
                    O[k] = morph3(MAX, O[k], CO[0][a], CO[1][b]);
                }
            }
            // rows t - R and t - R + 1 are complete
#pragma unroll
            for (int q = 0; q < 2; q++) {
                const int y = t - R + q, k = (2 * u + q) % K;
                if (y < ys || y >= ye || x0 >= W) continue;
                const uint32_t v = __byte_perm(E[k], O[k], 0x7351) & last;
                uint8_t* p = g.dst + (size_t)y * g.dp + x0;
                if (words) {
                    *reinterpret_cast<uint32_t*>(p) = v;
                } else {
#pragma unroll
                    for (int i = 0; i < 4; i++)
                        if (x0 + i < W) p[i] = (uint8_t)(v >> (8 * i));
                }
            }
        }
    }
}

// Launches one pass.  Segments: as many as fill the resident warps once, so
// that every warp streams the same number of rows and reads as few rows twice
// as that allows (r = 9, both passes: 53 us for 4096^2 with 54 rows, 62 with 64;
// 165 us for 16384 x 4096 with 216 rows, 171 with 128), but not below 16 rows
// (2047 x 1531: 29 us, 33 with 10 rows; 512^2: 17, and 13 to 16 with 2 to 8).
template <int R, bool MAX>
void morph_launch(MorphArgs a, int sms, cudaStream_t s) {
    int per = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_morph_stream<R, MAX>, MS_WARPS * 32, 0) != cudaSuccess || per < 1)
        per = 1;
    const int most = sms * per * MS_WARPS, nseg = most / a.nstrip > 1 ? most / a.nstrip : 1;
    a.seg = (a.H + nseg - 1) / nseg;
    if (a.seg < MS_SEG_MIN) a.seg = MS_SEG_MIN;
    a.n = a.nstrip * ((a.H + a.seg - 1) / a.seg);
    k_morph_stream<R, MAX><<<(a.n + MS_WARPS - 1) / MS_WARPS, MS_WARPS * 32, 0, s>>>(a);
}

// The definitions for radii 1 .. MORPH_RMAX are spread over k_morph*.cu, so that
// they compile in parallel.
template <int R>
void morph_pass(const MorphArgs& a, bool dilate, int sms, cudaStream_t s);
#define MORPH_DECLARE(R) template <> void morph_pass<R>(const MorphArgs&, bool, int, cudaStream_t);
MORPH_DECLARE(1) MORPH_DECLARE(2) MORPH_DECLARE(3) MORPH_DECLARE(4) MORPH_DECLARE(5)
MORPH_DECLARE(6) MORPH_DECLARE(7) MORPH_DECLARE(8) MORPH_DECLARE(9) MORPH_DECLARE(10)
MORPH_DECLARE(11) MORPH_DECLARE(12) MORPH_DECLARE(13) MORPH_DECLARE(14) MORPH_DECLARE(15)
#define MORPH_PASS(R)                                                                      \
    template <>                                                                            \
    void morph_pass<R>(const MorphArgs& a, bool dilate, int sms, cudaStream_t s) {         \
        if (dilate) morph_launch<R, true>(a, sms, s);                                      \
        else morph_launch<R, false>(a, sms, s);                                            \
    }

}  // namespace nucseg
