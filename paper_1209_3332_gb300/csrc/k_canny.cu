// Canny edges of a uint8 plane (Sec. V-A lists Canny among the
// feature-stage transforms applied to the deconvolved image; Table I
// "Features comp.") and the per-object edge counts (Sec. II "edge"
// features).  Definition (the paper gives no parameter):
//   gx, gy = 3x3 Sobel with replicated border; m = |gx| + |gy|;
//   sector: horizontal if (ax + ay)^2 < 2 ax^2 (ay < ax tan 22.5 deg),
//     vertical if ay > ax and (ay - ax)^2 > 2 ax^2 (ay > ax tan 67.5 deg),
//     else the diagonal along (+x,+y) when gx gy > 0, (+x,-y) otherwise;
//   neighbours a, b along the sector (a on the previous row, or the left
//     one for the horizontal sector); m outside the image is 0;
//   p survives iff m(p) > m(a) and m(p) >= m(b); candidate iff it survives
//     with m > low, strong iff it survives with m > high;
//   edges = candidates 8-connected through candidates to a strong pixel.
// Every kernel takes a table of tile descriptors, so one launch covers any
// number of tiles (the plain form is the batched form of one tile), a warp
// finding its tile by binary search over the tiles' first items.
// k_canny_nms writes the strong pixels (the marker) and the candidates (the
// mask) as bit planes, 64x64 work tile by work tile; the hysteresis is the
// growth of the marker through the mask (k_grow.cu), which also writes the
// edge map as bytes.  The counts are a stencil pass over 32x32 blocks: each
// edge pixel adds one to every object with a pixel within its disk -- the
// same count as the edge pixels within each object's disk dilation, with the
// labels read only around edges.
#include "internal.cuh"

namespace nucseg {

constexpr int CT = 32;                 // block of the counts pass: CT x CT pixels
typedef unsigned long long u64;

// ---- suppression: one warp streams a strip of 128 columns (4 per lane) down
// a segment of 64 rows (one work-tile row), keeping four image rows and the
// magnitudes of three in registers ---------------------------------------------------
constexpr int NS_COLS = 128, NS_ROWS = 64;
constexpr int NS_WARPS = 4;          // warps per CTA

struct Row8 {                        // image row, columns cx0 - 2 .. cx0 + 5 (replicated border), as
    uint32_t p[4];                   // four pairs of 16-bit lanes: (-2,-1), (0,1), (2,3), (4,5)
};

// the global reads of one row for one lane: its own 4 pixels, and on the
// strip's edge lanes the two pixels beyond the strip
struct RowFetch {
    uint32_t w;
    int e0, e1;
};

__device__ __forceinline__ RowFetch ns_fetch(const uint8_t* __restrict__ I, int W, int H, int y, int cx0, bool vec,
                                             int lane) {
    const uint8_t* row = I + (size_t)min(max(y, 0), H - 1) * W;
    RowFetch f;
    if (vec && cx0 < W) {
        f.w = __ldg(reinterpret_cast<const uint32_t*>(row + cx0));
    } else {
        f.w = 0;
#pragma unroll
        for (int k = 3; k >= 0; k--) f.w = (f.w << 8) | __ldg(row + min(cx0 + k, W - 1));
    }
    f.e0 = f.e1 = 0;
    if (lane == 0) {
        f.e0 = __ldg(row + max(cx0 - 2, 0));
        f.e1 = __ldg(row + max(cx0 - 1, 0));
    } else if (lane == 31) {
        f.e0 = __ldg(row + min(cx0 + 4, W - 1));
        f.e1 = __ldg(row + min(cx0 + 5, W - 1));
    }
    return f;
}

// columns cx0 - 2 .. cx0 + 5 of a fetched row: the neighbours' pixels by shuffle
__device__ __forceinline__ Row8 ns_row(const RowFetch& f, int lane) {
    uint32_t wl = __shfl_up_sync(0xffffffffu, f.w, 1), wr = __shfl_down_sync(0xffffffffu, f.w, 1);
    if (lane == 0) wl = ((uint32_t)f.e0 << 16) | ((uint32_t)f.e1 << 24);   // bytes 2, 3: columns -2, -1
    if (lane == 31) wr = (uint32_t)f.e0 | ((uint32_t)f.e1 << 8);            // bytes 0, 1: columns 4, 5
    Row8 r;
    r.p[0] = __byte_perm(wl, 0u, 0x4342);
    r.p[1] = __byte_perm(f.w, 0u, 0x4140);
    r.p[2] = __byte_perm(f.w, 0u, 0x4342);
    r.p[3] = __byte_perm(wr, 0u, 0x4140);
    return r;
}

__device__ __forceinline__ Row8 ns_load_row(const uint8_t* __restrict__ I, int W, int H, int y, int cx0, bool vec,
                                            int lane) {
    return ns_row(ns_fetch(I, W, H, y, cx0, vec, lane), lane);
}

__device__ __forceinline__ uint32_t max2(uint32_t a, uint32_t b) {
    uint32_t d;
    asm("max.u16x2 %0, %1, %2;" : "=r"(d) : "r"(a), "r"(b));
    return d;
}
__device__ __forceinline__ uint32_t min2(uint32_t a, uint32_t b) {
    uint32_t d;
    asm("min.u16x2 %0, %1, %2;" : "=r"(d) : "r"(a), "r"(b));
    return d;
}

// Sobel of the row between A and C (rows r - 1, r, r + 1, replicated) in
// 16x2-bit lanes, for the column pairs (-1, 0), (1, 2), (3, 4): with
// vs = A + 2B + C and vd = C - A per column, gx(c) = vs(c+1) - vs(c-1) and
// gy(c) = vd(c-1) + 2 vd(c) + vd(c+1).  Signed values carry a bias (256 on
// vd, 1024 on gx and gy) so that every lane stays in [0, 2^16) and packed
// adds never borrow across lanes.
constexpr uint32_t B256 = 0x01000100u, B1024 = 0x04000400u;
struct Grad {
    uint32_t x[3], y[3];  // gx + 1024, gy + 1024
};
__device__ __forceinline__ Grad ns_grad(const Row8& A, const Row8& B, const Row8& C) {
    uint32_t V[4], Dv[4];
#pragma unroll
    for (int k = 0; k < 4; k++) {
        V[k] = A.p[k] + (B.p[k] << 1) + C.p[k];
        Dv[k] = C.p[k] + B256 - A.p[k];
    }
    Grad g;
#pragma unroll
    for (int k = 0; k < 3; k++) {
        g.x[k] = V[k + 1] + B1024 - V[k];
        g.y[k] = Dv[k] + (__byte_perm(Dv[k], Dv[k + 1], 0x5432) << 1) + Dv[k + 1];
    }
    return g;
}
__device__ __forceinline__ uint32_t abs2(uint32_t biased) { return max2(biased, B1024) - min2(biased, B1024); }

// L1 magnitudes of the three column pairs.  colmask: per pair, 0xffff on the
// lanes of columns inside the image; m is 0 elsewhere and on a row off the image.
struct Mag {
    uint32_t m[3];
    __device__ __forceinline__ int at(int j) const { return (int)((m[j >> 1] >> (16 * (j & 1))) & 0xffffu); }
};
__device__ __forceinline__ Mag ns_mag(const Grad& g, const uint32_t colmask[3], bool row_in) {
    Mag o;
#pragma unroll
    for (int k = 0; k < 3; k++) o.m[k] = row_in ? (abs2(g.x[k]) + abs2(g.y[k])) & colmask[k] : 0u;
    return o;
}

// floor(v tan 22.5 deg) for 0 <= v <= 1020, where it equals (v * 27146) >> 16
// (tan 22.5 deg is irrational, so a <= tan22(b) is a < b tan 22.5 deg for b > 0)
__device__ __forceinline__ int tan22(int v) { return (v * 27146) >> 16; }

// One warp per strip of 128 columns (two work tiles) and 64 rows (one work
// tile).  Magnitudes are computed for every pixel; the suppression itself
// runs only on rows where some lane has a magnitude above low, which leaves
// out about half of the rows on the benchmark tile (8 planes of 4096^2: 290 us,
// 502 with the suppression of every pixel and byte planes; rows fetched two
// ahead instead of one: no change).  Bound: instruction issue (1 B read and
// 1/4 B written per pixel, 25 us).  The strip's marker and mask bits are
// gathered in shared memory, four columns per lane and row.
__global__ void __launch_bounds__(32 * NS_WARPS, 6) k_canny_nms(const __grid_constant__ GrowLaunch G, int n_warps,
                                                                int low, int high) {
    __shared__ __align__(16) uint8_t bits[NS_WARPS][2][NS_ROWS][NS_COLS / 8];  // marker, mask
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int gw = blockIdx.x * NS_WARPS + warp;
    if (blockIdx.x == 0 && threadIdx.x == 0) grow_reset(G);
    if (gw >= n_warps) return;
    const CannyDesc& d = G.tab[G.tab.find(gw, &CannyDesc::nms_base)];
    const uint8_t* __restrict__ I = d.img;
    const int W = d.W, H = d.H, wi = gw - d.nms_base;
    const int strips = (W + NS_COLS - 1) / NS_COLS, nw = strips * ((H + NS_ROWS - 1) / NS_ROWS);
    const int seg = wi / strips, strip = wi - seg * strips;
    const int cx0 = strip * NS_COLS + 4 * lane, ya = seg * NS_ROWS, yb = min(ya + NS_ROWS, H);
    // this warp's share of the counts to zero
    for (long long i = (long long)wi * 32 + lane; i < d.K; i += (long long)nw * 32) d.counts[i] = 0;
#pragma unroll
    for (int i = 0; i < 2 * NS_ROWS * NS_COLS / 8 / (32 * 16); i++)
        reinterpret_cast<uint4*>(&bits[warp][0][0][0])[i * 32 + lane] = make_uint4(0, 0, 0, 0);
    __syncwarp();
    const bool vec = (W & 3) == 0 && (reinterpret_cast<uintptr_t>(I) & 3) == 0;
    uint32_t colmask[3];  // pair k holds columns cx0 + 2k - 1 and cx0 + 2k
#pragma unroll
    for (int k = 0; k < 3; k++) {
        const int x = cx0 + 2 * k - 1;
        colmask[k] = ((x >= 0 && x < W) ? 0xffffu : 0u) | ((x + 1 >= 0 && x + 1 < W) ? 0xffff0000u : 0u);
    }
    const uint32_t low2 = (uint32_t)min(low, 0xffff) * 0x00010001u;
    Row8 P = ns_load_row(I, W, H, ya - 1, cx0, vec, lane);
    Row8 Q = ns_load_row(I, W, H, ya, cx0, vec, lane);
    Row8 N = ns_load_row(I, W, H, ya + 1, cx0, vec, lane);
    Mag prev = ns_mag(ns_grad(ns_load_row(I, W, H, ya - 2, cx0, vec, lane), P, Q), colmask, ya - 1 >= 0);
    Mag cur = ns_mag(ns_grad(P, Q, N), colmask, true);
    RowFetch fn = ns_fetch(I, W, H, ya + 2, cx0, vec, lane);  // one row ahead of its use
#pragma unroll 1
    for (int y = ya; y < yb; y++) {
        const Row8 M = ns_row(fn, lane);  // rows P, Q, N, M: y - 1 .. y + 2
        fn = ns_fetch(I, W, H, y + 3, cx0, vec, lane);
        const Mag next = ns_mag(ns_grad(Q, N, M), colmask, y + 1 < H);
        // columns cx0 .. cx0 + 3 are the high lane of pair 0, pair 1, the low lane of pair 2
        const uint32_t top = max2(max2(cur.m[0] >> 16, cur.m[1]), cur.m[2] & 0xffffu);
        if (__any_sync(0xffffffffu, max2(top, low2) != low2)) {
            const Grad g = ns_grad(P, Q, N);
            unsigned v = 0;  // bits 0-3: strong, 4-7: candidates
#pragma unroll
            for (int c = 0; c < 4; c++) {
                const int j = c + 1, sh = 16 * (j & 1), m = cur.at(j);
                const int gx = (int)((g.x[j >> 1] >> sh) & 0xffffu) - 1024, gy = (int)((g.y[j >> 1] >> sh) & 0xffffu) - 1024;
                const int ax = abs(gx), ay = abs(gy);
                const bool hor = ay <= tan22(ax), ver = ax <= tan22(ay), same = (gx ^ gy) >= 0;
                // a on the previous row (left for the horizontal sector), b opposite
                const int ma = hor ? cur.at(j - 1) : ver ? prev.at(j) : same ? prev.at(j - 1) : prev.at(j + 1);
                const int mb = hor ? cur.at(j + 1) : ver ? next.at(j) : same ? next.at(j + 1) : next.at(j - 1);
                const bool keep = m > ma && m >= mb && m > low;
                v |= (keep ? 16u << c : 0u) | (keep && m > high ? 1u << c : 0u);
            }
            // bytes of 8 columns: the even lane of a pair writes the marker, the odd one the mask
            const unsigned o = __shfl_xor_sync(0xffffffffu, v, 1);
            bits[warp][lane & 1][y - ya][lane >> 1] =
                (uint8_t)((lane & 1) ? (o >> 4) | (v & 0xf0u) : (v & 15u) | (o << 4));
        }
        prev = cur;
        cur = next;
        P = Q;
        Q = N;
        N = M;
    }
    __syncwarp();
    const int rtx = (W + RT - 1) / RT;
#pragma unroll
    for (int h = 0; h < 2; h++) {  // the strip's two work tiles: rows 2 l and 2 l + 1 from lane l
        const int tx = 2 * strip + h;
        if (tx >= rtx) break;
        const size_t t = (size_t)d.rt_base + (size_t)seg * rtx + tx;
        u64 w[2][2];
#pragma unroll
        for (int q = 0; q < 2; q++)
#pragma unroll
            for (int r = 0; r < 2; r++) w[q][r] = *reinterpret_cast<const u64*>(&bits[warp][q][2 * lane + r][8 * h]);
        reinterpret_cast<ulonglong2*>(G.marker + t * RT)[lane] = make_ulonglong2(w[0][0], w[0][1]);
        reinterpret_cast<ulonglong2*>(G.mask + t * RT)[lane] = make_ulonglong2(w[1][0], w[1][1]);
        const bool any = __any_sync(0xffffffffu, (w[0][0] | w[0][1]) != 0ull);
        if (lane == 0) G.any[t] = any;
    }
}

// ---- edge counts: one warp per 32x32 block with an edge pixel ---------------------
// The warp lists the block's edge pixels (a few dozen of 1024), stages the
// labels of the rows within r of them with a 4-pixel margin (0 off the
// image, and for labels outside 1..K) and one bit per staged pixel that holds
// an object, and takes the listed pixels 32 at a time, one per lane: the
// bits under the disk's chord of each row pick the labels to look at.  Each
// edge pixel adds one to every distinct object in its disk: the first four are
// remembered in registers, the others as a bit of 64 (a hash where there are more
// objects than bits), and only an object whose bit is taken is looked for at the
// earlier disk offsets (1024^2 of noise with a label on every other pixel, disks
// of radius 4 with 25 objects: 1004 us; 2350 with every object looked for).
// 8 tiles of 4096^2: 146 us (465 with a CTA per block, a thread per pixel and a
// label read for every disk offset).  Bound: the latency of the label loads of
// the blocks that hold edges (about half; seven of a lane in flight), 24 warps
// per SM by shared memory.
constexpr int CR_MAX = 4;                 // largest disk radius of the counts
constexpr int CC_S = CT + 2 * CR_MAX;     // staged labels: the block and a CR_MAX-pixel margin (40 x 40)
// Blocks (one per warp) per CTA: most blocks hold no edge pixel and end at once, and
// a CTA keeps its warps' places until its slowest is done (8 tiles of 4096^2: 224
// us with four, 170 with two, 146 with one).
constexpr int CC_WARPS = 1;

struct CountStage {
    int32_t lab[CC_S][CC_S];
    u64 occ[CC_S];           // bit x: lab[y][x] != 0
    uint16_t list[CT * CT];  // edge pixels, y << 5 | x
};

__global__ void __launch_bounds__(CC_WARPS * 32) k_canny_counts(const __grid_constant__ GrowLaunch G, int n_blocks, int r) {
    extern __shared__ __align__(16) unsigned char cc_smem[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    CountStage& S = reinterpret_cast<CountStage*>(cc_smem)[warp];
    const int gb = blockIdx.x * CC_WARPS + warp;
    if (gb >= n_blocks) return;
    const CannyDesc& d = G.tab[G.tab.find(gb, &CannyDesc::blk_base)];
    const int K = d.K, W = d.W, H = d.H, bl = gb - d.blk_base;
    if (K <= 0) return;
    const int by = bl / d.bx, bx = bl - by * d.bx, x0 = bx * CT, y0 = by * CT;
    const size_t t = (size_t)d.rt_base + (size_t)(by >> 1) * ((W + RT - 1) / RT) + (bx >> 1);
    const uint32_t e = reinterpret_cast<const uint32_t*>(G.marker + t * RT + (by & 1) * CT + lane)[bx & 1];
    const unsigned rows = __ballot_sync(0xffffffffu, e != 0u);  // block rows with an edge pixel
    if (!rows) return;
    int at = __popc(e), n;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int v = __shfl_up_sync(0xffffffffu, at, o);
        if (lane >= o) at += v;
    }
    n = __shfl_sync(0xffffffffu, at, 31);
    at -= __popc(e);
    for (uint32_t m = e; m; m &= m - 1) S.list[at++] = (uint16_t)(lane << 5 | (__ffs(m) - 1));
    // staged rows needed: within r of a row with an edge pixel (staged row = block row + CR_MAX)
    u64 need = 0;
    for (int dy = CR_MAX - r; dy <= CR_MAX + r; dy++) need |= (u64)rows << dy;
    const bool vec = (W & 3) == 0 && (reinterpret_cast<uintptr_t>(d.labels) & 15) == 0;
    if (lane < CC_S) S.occ[lane] = 0ull;
    if (lane < CC_S - 32) S.occ[lane + 32] = 0ull;
    __syncwarp();
    constexpr int NQ = CC_S * (CC_S / 4);
    constexpr int CU = 7;  // loads of a lane in flight
#pragma unroll 1
    for (int i0 = 0; i0 < NQ; i0 += CU * 32) {
        int4 v[CU];
#pragma unroll
        for (int u = 0; u < CU; u++) {
            const int i = i0 + 32 * u + lane, ly = i / (CC_S / 4), q = i - ly * (CC_S / 4);
            const int gy = y0 - CR_MAX + ly, gx = x0 - CR_MAX + 4 * q;
            v[u] = make_int4(0, 0, 0, 0);
            if (i < NQ && ((need >> ly) & 1u) && (unsigned)gy < (unsigned)H) {
                const int32_t* src = d.labels + (size_t)gy * W + gx;
                if (vec && gx >= 0 && gx + 4 <= W) {
                    v[u] = __ldg(reinterpret_cast<const int4*>(src));
                } else {
                    int w[4];
#pragma unroll
                    for (int k = 0; k < 4; k++) w[k] = (unsigned)(gx + k) < (unsigned)W ? __ldg(src + k) : 0;
                    v[u] = make_int4(w[0], w[1], w[2], w[3]);
                }
            }
        }
#pragma unroll
        for (int u = 0; u < CU; u++) {
            const int i = i0 + 32 * u + lane, ly = i / (CC_S / 4), q = i - ly * (CC_S / 4);
            if (i >= NQ || !(v[u].x | v[u].y | v[u].z | v[u].w)) continue;
            int4 w = v[u];
            w.x = (w.x >= 1 && w.x <= K) ? w.x : 0;
            w.y = (w.y >= 1 && w.y <= K) ? w.y : 0;
            w.z = (w.z >= 1 && w.z <= K) ? w.z : 0;
            w.w = (w.w >= 1 && w.w <= K) ? w.w : 0;
            *reinterpret_cast<int4*>(&S.lab[ly][4 * q]) = w;  // read only where occ is set
            const u64 o = (u64)((w.x != 0) | (w.y != 0) << 1 | (w.z != 0) << 2 | (w.w != 0) << 3) << (4 * q);
            if (o) atomicOr(&S.occ[ly], o);
        }
    }
    __syncwarp();
    const int r2 = r * r;
    const bool exact = K <= 64;  // a bit for every object
    for (int i0 = 0; i0 < n; i0 += 32) {
        if (i0 + lane >= n) break;
        const int p = S.list[i0 + lane], ly = p >> 5, lx = p & 31;
        int seen0 = 0, seen1 = 0, seen2 = 0, seen3 = 0, nseen = 0;
        u64 seen = 0;
        // the chord of the disk in row dy: its half-width, and its pixels with an object from its left end on
        auto chord = [&](int dy, int& w) -> u64 {
            w = r;
            while (w * w + dy * dy > r2) w--;
            return (S.occ[ly + CR_MAX + dy] >> (lx + CR_MAX - w)) & ((2ull << (2 * w)) - 1ull);
        };
        for (int dy = -r; dy <= r; dy++) {
            int w;
            for (u64 m = chord(dy, w); m; m &= m - 1) {
                const int dx = __ffsll((long long)m) - 1 - w;
                const int v = S.lab[ly + CR_MAX + dy][lx + CR_MAX + dx];
                if (v == seen0 || v == seen1 || v == seen2 || v == seen3) continue;
                if (nseen >= 4) {
                    const u64 bit = 1ull << (exact ? v - 1 : (int)(((unsigned)v * 0x9e3779b1u) >> 26));
                    bool fresh = !(seen & bit);
                    if (!fresh && !exact) {  // look for v at an earlier disk offset
                        fresh = true;
                        for (int ey = -r; ey <= dy && fresh; ey++) {
                            int we;
                            u64 e = chord(ey, we);
                            if (ey == dy) e &= (1ull << (dx + w)) - 1ull;
                            for (; e && fresh; e &= e - 1)
                                fresh = S.lab[ly + CR_MAX + ey][lx + CR_MAX + __ffsll((long long)e) - 1 - we] != v;
                        }
                    }
                    if (!fresh) continue;
                    seen |= bit;
                }
                atomicAdd(&d.counts[v - 1], 1);
                if (nseen == 0) seen0 = v; else if (nseen == 1) seen1 = v; else if (nseen == 2) seen2 = v;
                else if (nseen == 3) seen3 = v;
                nseen++;
            }
        }
    }
}

int canny_blocks(int W, int H) { return ((W + CT - 1) / CT) * ((H + CT - 1) / CT); }
int canny_nms_warps(int W, int H) { return ((W + NS_COLS - 1) / NS_COLS) * ((H + NS_ROWS - 1) / NS_ROWS); }

void launch_canny_nms(const GrowLaunch& G, int warps, int low, int high, cudaStream_t s, Profiler* pf) {
    pf->begin("canny_nms", s);
    k_canny_nms<<<(warps + NS_WARPS - 1) / NS_WARPS, 32 * NS_WARPS, 0, s>>>(G, warps, low, high);
    pf->end("canny_nms", s);
}

void launch_canny_counts(const GrowLaunch& G, int blocks, int r, cudaStream_t s, Profiler* pf) {
    pf->begin("canny_counts", s);
    k_canny_counts<<<(blocks + CC_WARPS - 1) / CC_WARPS, CC_WARPS * 32, CC_WARPS * sizeof(CountStage), s>>>(G, blocks, r);
    pf->end("canny_counts", s);
}

}  // namespace nucseg
