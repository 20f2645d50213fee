// K5: exact squared Euclidean distance transform to the nearest label-0
// pixel (Table I, the distance transform of "Pre-Watershed").
//
// Separable form (as in Meijster, Roerdink, Hesselink 2000): g(y,x) is the
// distance along column x to the nearest background pixel, and
// D(y,x) = min_q (x-q)^2 + g(y,q)^2 along row y.
//
// GB300 layout: the relabel pass leaves, per 32-row chunk and column, one
// word with the chunk's 32 kept bits of that column (2 MB for a 4K tile).
// k_edt_rows handles a band of rows per CTA: for each column it finds the
// nearest background row within the chunk with bit scans, and above/below
// the chunk by walking to the nearest chunk that has background (almost
// always the adjacent one), keeps the band's g rows in shared memory and
// solves every row there, so the only full-plane traffic is the single
// int32 write of D.  Rows whose g stays
// within WMAX use an exact windowed search (a candidate at distance r costs
// at least r^2, so the search stops once r^2 >= the best value); other rows
// run Meijster's lower-envelope scan on one thread.  Shared memory holds
// only the band (4 rows of u16 for a 4096-wide tile, each padded with WMAX
// "no background" entries on both sides so that the search needs no bounds
// test), so several CTAs fit on an SM.
//
// 16 tiles of 4096^2: 265 us for 1.07 GB written (4.1 TB/s), 310 before the
// columns and the pixels were taken in fours; what bounds it is the search of
// foreground pixels in shared memory, where a warp waits for its farthest
// pixel, and the barrier between a CTA's columns and its rows.  (Limited to 40
// registers, six CTAs per SM instead of five: 258 us, but with spills, and one
// tile of 4096^2 takes 28.5 instead of 27 us.  Streaming stores: no change.)
#include "internal.cuh"

namespace nucseg {

constexpr int INFG = 32767;       // "no background in this column"
constexpr int WMAX = 128;
constexpr unsigned FULLE = 0xffffffffu;

__device__ __forceinline__ int sq(int v) { return v * v; }
__device__ __forceinline__ uint32_t below_or_at(int k) { return (2u << k) - 1u; }  // bits 0..k

// Meijster's row pass for rows whose column distances exceed WMAX (rare:
// long stretches of foreground).  The stack of (site s, start t) pairs lives
// in the output row itself, packed as (s << 16) | t: in the backward pass the
// live stack index q satisfies q <= t[q] <= u, and entry q is read before
// out[u] is written, so no scratch memory is needed.
__device__ void meijster_row(const uint16_t* g, int W, int32_t* out) {
    auto F = [&](int u, int i) -> long long { return (long long)(u - i) * (u - i) + (long long)g[i] * g[i]; };
    auto S = [&](int k) -> int { return (int)((uint32_t)out[k] >> 16); };
    auto Tt = [&](int k) -> int { return (int)(out[k] & 0xffff); };
    int q = 0;
    out[0] = 0;
    for (int u = 1; u < W; u++) {
        while (q >= 0 && F(Tt(q), S(q)) > F(Tt(q), u)) q--;
        if (q < 0) {
            q = 0;
            out[0] = (int32_t)((uint32_t)u << 16);
        } else {
            int i = S(q);
            long long num = (long long)u * u - (long long)i * i + (long long)g[u] * g[u] - (long long)g[i] * g[i];
            long long den = 2LL * (u - i);
            long long fl = num / den;
            if ((num % den != 0) && (num < 0)) fl--;
            long long w = 1 + fl;
            if (w < W) {
                q++;
                out[q] = (int32_t)(((uint32_t)u << 16) | (uint32_t)w);
            }
        }
    }
    for (int u = W - 1; u >= 0; u--) {
        const int su = S(q), tu = Tt(q);
        long long d = F(u, su);
        out[u] = d >= (long long)INFG * INFG ? 0x7fffffff : (int32_t)d;
        if (u == tu) q--;
    }
}

__global__ void __launch_bounds__(256) k_edt_rows(Launch L, int RB, int Wmax) {
    if (L.early) after_previous();
    extern __shared__ __align__(16) unsigned char smraw[];
    uint16_t* gs = reinterpret_cast<uint16_t*>(smraw);  // [RB][WMAX + Wmax + WMAX]
    const int Wp = Wmax + 2 * WMAX;
    __shared__ int rowslow[32];
    const int gbnd = blockIdx.x;
    const int ti = find_tile(L.tiles, L.ntiles, gbnd, &TileDev::row_base);
    const TileDev T = L.tiles[ti];
    if (!T.edt) return;
    const int W = T.W, H = T.H;
    const int y0 = (gbnd - T.row_base) * RB;
    const int c = y0 / CB, r0 = c * CB;
    const int nrow = min(RB, H - y0);
    const int nchunk = T.cby;
    if (threadIdx.x < 32) rowslow[threadIdx.x] = 0;
    for (int i = threadIdx.x; i < nrow * 2 * WMAX; i += blockDim.x) {
        const int j = i / (2 * WMAX), k = i - j * 2 * WMAX;
        gs[(size_t)j * Wp + (k < WMAX ? k : W + k)] = (uint16_t)INFG;
    }
    __syncthreads();
    auto rows_valid = [&](int cc) -> uint32_t {
        int k = min(CB, H - cc * CB);
        return k >= 32 ? FULLE : ((1u << k) - 1u);
    };
    const uint32_t rv = rows_valid(c);
    const uint32_t* const colbits = T.colbits;
    const int k0 = y0 - r0, k1 = y0 + nrow - 1 - r0;
    const uint32_t band = below_or_at(k1) & ~((1u << k0) - 1u);
    // nearest background row of column x above / below this chunk, where the
    // chunk (background bits bg) has none on that side of the band
    auto look_above = [&](int x, uint32_t bg) -> int {
        if (!(bg & below_or_at(k0)))
            for (int cc = c - 1; cc >= 0; cc--) {
                const uint32_t b2 = ~colbits[(size_t)cc * W + x] & rows_valid(cc);
                if (b2) return cc * CB + 31 - __clz(b2);
            }
        return -1;
    };
    auto look_below = [&](int x, uint32_t bg) -> int {
        if (!(bg & ~((1u << k1) - 1u)))
            for (int cc = c + 1; cc < nchunk; cc++) {
                const uint32_t b2 = ~colbits[(size_t)cc * W + x] & rows_valid(cc);
                if (b2) return cc * CB + __ffs(b2) - 1;
            }
        return -1;
    };
    auto g_of = [&](int y, uint32_t bg, int above, int below) -> int {
        const int k = y - r0;
        const uint32_t mu = bg & below_or_at(k);
        const int du = mu ? k - (31 - __clz(mu)) : (above >= 0 ? y - above : INFG);
        const uint32_t md = bg & ~((1u << k) - 1u);
        const int dd = md ? (__ffs(md) - 1) - k : (below >= 0 ? below - y : INFG);
        return min(min(du, dd), INFG);
    };
    // g for the band.  Widths that are a multiple of 4: four columns per
    // thread, one 16-byte load of their words (the next four are under way
    // meanwhile) and one 8-byte store per row.
    if ((W & 3) == 0 && (Wp & 3) == 0) {
        const int step = 4 * blockDim.x;
        const uint32_t* const words = colbits + (size_t)c * W;  // 16-byte aligned: the plane is, and W
        int x = 4 * threadIdx.x;
        uint4 next = make_uint4(0u, 0u, 0u, 0u);
        if (x < W) next = __ldg(reinterpret_cast<const uint4*>(words + x));
        for (; x < W; x += step) {
            const uint32_t bg[4] = {~next.x & rv, ~next.y & rv, ~next.z & rv, ~next.w & rv};
            if (x + step < W) next = __ldg(reinterpret_cast<const uint4*>(words + x + step));
            if (((bg[0] & bg[1]) & (bg[2] & bg[3]) & band) == band) {  // background on every row of the band: g = 0
                for (int j = 0; j < nrow; j++) *reinterpret_cast<uint2*>(gs + (size_t)j * Wp + WMAX + x) = make_uint2(0u, 0u);
                continue;
            }
            int above[4], below[4];
#pragma unroll
            for (int u = 0; u < 4; u++) {
                above[u] = look_above(x + u, bg[u]);
                below[u] = look_below(x + u, bg[u]);
            }
            for (int j = 0; j < nrow; j++) {
                int gv[4];
#pragma unroll
                for (int u = 0; u < 4; u++) gv[u] = g_of(y0 + j, bg[u], above[u], below[u]);
                *reinterpret_cast<uint2*>(gs + (size_t)j * Wp + WMAX + x) =
                    make_uint2((uint32_t)gv[0] | ((uint32_t)gv[1] << 16), (uint32_t)gv[2] | ((uint32_t)gv[3] << 16));
                if (max(max(gv[0], gv[1]), max(gv[2], gv[3])) > WMAX) rowslow[j] = 1;
            }
        }
    } else {
        // one column per thread; the words of four columns are loaded before
        // any is used, so their latencies overlap
        constexpr int CU = 4;
        for (int xb = threadIdx.x; xb < W; xb += CU * blockDim.x) {
            uint32_t wv[CU];
#pragma unroll
            for (int u = 0; u < CU; u++) {
                const int x = xb + u * blockDim.x;
                wv[u] = x < W ? __ldg(colbits + (size_t)c * W + x) : 0u;
            }
#pragma unroll
            for (int u = 0; u < CU; u++) {
                const int x = xb + u * blockDim.x;
                if (x >= W) break;
                const uint32_t bg = ~wv[u] & rv;
                if ((bg & band) == band) {
                    for (int j = 0; j < nrow; j++) gs[(size_t)j * Wp + WMAX + x] = 0;
                    continue;
                }
                const int above = look_above(x, bg), below = look_below(x, bg);
                for (int j = 0; j < nrow; j++) {
                    const int gv = g_of(y0 + j, bg, above, below);
                    gs[(size_t)j * Wp + WMAX + x] = (uint16_t)gv;
                    if (gv > WMAX) rowslow[j] = 1;
                }
            }
        }
    }
    __syncthreads();
    for (int j = 0; j < nrow; j++) {
        const uint16_t* g = gs + (size_t)j * Wp + WMAX;
        int32_t* out = T.edt + (size_t)(y0 + j) * W;
        if (!rowslow[j]) {
            // g <= WMAX on this row, so r < WMAX stays within the padding,
            // whose entries cost INFG^2 and never win
            auto solve = [&](int x) -> int {
                int D = sq(g[x]);
                for (int r = 1, rr = 1; rr < D; rr += 2 * r + 1, r++) {
                    D = __viaddmin_s32(sq(g[x - r]), rr, D);
                    D = __viaddmin_s32(sq(g[x + r]), rr, D);
                }
                return D;
            };
            // Four pixels per thread, searched together: the site r beyond either
            // end of the four is a candidate for each of them, so one read of g
            // serves four updates.  Every candidate is a true one, so looking as
            // far as the largest of the four values needs changes no result.
            auto solve4 = [&](int x, int g0, int g1, int g2, int g3) -> int4 {
                const int s0 = sq(g0), s1 = sq(g1), s2 = sq(g2), s3 = sq(g3);
                int d0 = min(__viaddmin_s32(s1, 1, s0), __viaddmin_s32(s2, 4, s3 + 9));
                int d1 = min(__viaddmin_s32(s0, 1, s1), __viaddmin_s32(s2, 1, s3 + 4));
                int d2 = min(__viaddmin_s32(s1, 1, s2), __viaddmin_s32(s3, 1, s0 + 4));
                int d3 = min(__viaddmin_s32(s2, 1, s3), __viaddmin_s32(s1, 4, s0 + 9));
                int a0 = 1, a1 = 4, a2 = 9, a3 = 16;  // r^2 .. (r + 3)^2
                for (int r = 1; a0 < max(max(d0, d1), max(d2, d3)); r++) {
                    const int l = sq(g[x - r]), h = sq(g[x + 3 + r]);
                    d0 = __viaddmin_s32(l, a0, __viaddmin_s32(h, a3, d0));
                    d1 = __viaddmin_s32(l, a1, __viaddmin_s32(h, a2, d1));
                    d2 = __viaddmin_s32(l, a2, __viaddmin_s32(h, a1, d2));
                    d3 = __viaddmin_s32(l, a3, __viaddmin_s32(h, a0, d3));
                    a0 = a1;
                    a1 = a2;
                    a2 = a3;
                    a3 += 2 * r + 7;
                }
                return make_int4(d0, d1, d2, d3);
            };
            if ((W & 3) == 0 && (Wp & 3) == 0 && (reinterpret_cast<uintptr_t>(out) & 15) == 0) {
                // one 8-byte read of g (8-byte aligned: WMAX, x and the row
                // stride Wp are multiples of 4), one 16-byte store; a run of
                // four background pixels needs no search at all
                for (int x = 4 * threadIdx.x; x < W; x += 4 * blockDim.x) {
                    const uint2 gq = *reinterpret_cast<const uint2*>(g + x);
                    int4 D = make_int4(0, 0, 0, 0);
                    if (gq.x | gq.y)
                        D = solve4(x, (int)(gq.x & 0xffffu), (int)(gq.x >> 16), (int)(gq.y & 0xffffu), (int)(gq.y >> 16));
                    *reinterpret_cast<int4*>(out + x) = D;
                }
            } else {
                for (int x = threadIdx.x; x < W; x += blockDim.x) out[x] = solve(x);
            }
        } else if (threadIdx.x == 0) {
            meijster_row(g, W, out);
        }
    }
}

size_t edt_rows_smem(int RB, int Wmax) { return (size_t)RB * (Wmax + 2 * WMAX) * 2; }

void launch_edt(const Launch& L, int RB, int Wmax, cudaStream_t s, Profiler* pf) {
    if (L.n_rows == 0) return;
    size_t smem = edt_rows_smem(RB, Wmax);
    cudaFuncSetAttribute(k_edt_rows, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    pf->begin("edt_rows", s);
    launch_behind(L.early && pf->overlap(), k_edt_rows, L.n_rows, 256, smem, s, L, RB, Wmax);
    pf->end("edt_rows", s);
}

}  // namespace nucseg
