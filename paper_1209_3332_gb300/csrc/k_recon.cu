// K2: grayscale reconstruction by dilation, 8-connected, of the h-dome
// marker under hem8 (Table I, "ReconToNuclei"; the paper's GPU version is a
// queue-based wave propagation, Sec. V-A).  R = lim R_k with
// R_{k+1} = min(dilate8(R_k), hem8), R_0 = max(hem8 - h, 0) (written by K1).
//
// Design (GB300): a persistent kernel of independent workers, each a warp, or
// in launches of few tiles a team of four (see k_recon).
// The image is cut into 64x64 work tiles; a device-wide queue holds the
// tiles that may still change.  A worker pops a tile, stages R and hem8 (M) of
// the tile and a one-pixel halo in its own shared memory, and runs rounds of
// four directional sweeps over the whole tile (down, up, right, left), each
// an exact sequential sweep along one axis:
//  * the tile is stored as 2x2-pixel blocks, one 32-bit word of R and one of
//    M per block, so that two pixels of a row and two pixels of a column are
//    equally one byte permute away from a pair of 16-bit lanes;
//  * a row sweep gives each lane two adjacent columns, a column sweep two
//    adjacent rows; the pair is updated with 16x2-bit SIMD max/min
//    (new = min(max(R, max of the three pixels of the line before), M)),
//    and the two outer neighbours come from the adjacent lanes by shuffle; the
//    halo is let into the border pixels once, before the first round;
//  * a sweep reads each block once per two lines and never reads what
//    another lane stored during it.
// After each round an exact, chain-free test decides whether another is
// needed.  The worker then writes the tile back and queues each neighbouring
// tile that one of the changed border pixels can still raise.  Values only
// grow and are bounded by hem8, so any order of tile processings reaches the
// same unique fixed point; a per-tile state machine (idle / queued / running
// / running+dirty) makes sure a tile is never processed by two workers at
// once and never misses a raise of its halo.  Every spin wait is bounded by
// the pipe's cycle budget, after which the worker records ST_TIMEOUT and
// returns.
#include <algorithm>

#include "internal.cuh"

namespace nucseg {

constexpr int NB = RT / 2;        // blocks per tile side
constexpr int BS = NB + 1;        // block row stride: 33 8-byte blocks (odd: column sweeps are conflict-free)
constexpr int HL = RT + 2;        // halo line length: index = coordinate + 1, coordinates -1..RT
constexpr int MAX_ROUNDS = 256;   // sweep rounds before a tile re-queues itself
constexpr int TEAM_MIN_BLOCKS = 8;  // resident teams per SM the register budget must allow
// Work tiles per resident warp below which teams take them: 16 tiles, 67 us by
// warps and 42 us by teams; 1024, 154 and 130; 3072, 221 and 203; 4096, 282 and
// 260; 5120, 255 and 272; 8192, 389 and 411; 16384, 507 and 672; 65536, 1822 and
// 2569 (2432 resident warps)
constexpr int TEAM_TILES = 2;
constexpr unsigned FULL = 0xffffffffu;

// A worker's staged tile.  Block (j, i) covers pixels (2j + a, 2i + b),
// a, b in {0, 1}: B[j * BS + i].x holds their R bytes and .y their M bytes,
// byte 2a + b.  The halo lines keep R as one 32-bit word per pixel: the
// first line of each pair (row -1, column -1) in bits 0-7, the second
// (row RT, column RT) in bits 16-23, which is where a pixel pair of the
// neighbouring edge lane needs it; the corners appear in a row and in a
// column line.  B0 keeps the four border lines as they were when neighbours were last
// queued for them (top, bottom, left, right).
struct WarpTile {
    uint2 B[NB * BS];
    uint32_t HRow[2][HL];
    uint32_t HC[2][HL];
    uint8_t HMr[2][HL + 2];  // M of the halo rows
    uint8_t HMc[2][HL + 2];  // M of the halo columns
    uint8_t B0[4][RT];
    int flags[9];            // neighbours to queue: up, down, left, right, UL, UR, DL, DR, self
    int msg;                 // from a team's first thread to the others
};

// The worker of a tile: one warp, or the NW warps of a CTA (the arguments are
// at k_recon).
template <int NW>
struct Worker {
    static constexpr int T = 32 * NW;
    int t, lane, warp;
    __device__ __forceinline__ Worker() : t(threadIdx.x), lane(NW == 1 ? t : t & 31), warp(NW == 1 ? 0 : t >> 5) {}
    __device__ __forceinline__ void sync() const {
        if constexpr (NW == 1) __syncwarp(); else __syncthreads();
    }
    // whether p holds for some thread; with NW > 1 also a barrier
    __device__ __forceinline__ bool any(bool p) const {
        if constexpr (NW == 1) return __any_sync(FULL, p); else return __syncthreads_or(p);
    }
    // thread 0's value
    __device__ __forceinline__ int from_first(WarpTile& S, int v) const {
        if constexpr (NW == 1) {
            return __shfl_sync(FULL, v, 0);
        } else {
            if (t == 0) S.msg = v;
            __syncthreads();
            v = *(volatile int*)&S.msg;
            __syncthreads();
            return v;
        }
    }
};

// R of halo pixel (hy, hx), and setting its R and M
__device__ __forceinline__ int halo_r(const WarpTile& S, int hy, int hx) {
    if (hy == -1) return (int)(S.HRow[0][hx + 1] & 0xffu);
    if (hy == RT) return (int)(S.HRow[1][hx + 1] >> 16);
    if (hx == -1) return (int)(S.HC[0][hy + 1] & 0xffu);
    return (int)(S.HC[1][hy + 1] >> 16);
}
__device__ __forceinline__ void set_halo_r(WarpTile& S, int hy, int hx, uint32_t r) {
    if (hy == -1) S.HRow[0][hx + 1] = r;
    if (hy == RT) S.HRow[1][hx + 1] = r << 16;
    if (hx == -1) S.HC[0][hy + 1] = r;
    if (hx == RT) S.HC[1][hy + 1] = r << 16;
}
__device__ __forceinline__ void set_halo_m(WarpTile& S, int hy, int hx, uint8_t m) {
    if (hy == -1) S.HMr[0][hx + 1] = m;
    if (hy == RT) S.HMr[1][hx + 1] = m;
    if (hx == -1) S.HMc[0][hy + 1] = m;
    if (hx == RT) S.HMc[1][hy + 1] = m;
}

// 16x2-bit SIMD helpers.  A pixel pair is two 16-bit lanes with the pixel in
// the high byte; the low bytes are left as they come, since they cannot change
// the high byte of a maximum or a minimum, so no permute has to clear them.
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
// byte permutes: a block word -> the pixel pair of row a (ROW0/ROW1) or of
// column 0 (COL0; the pair of column 1 is the word itself); two row or column
// pairs -> a block word
constexpr uint32_t ROW0 = 0x1404, ROW1 = 0x3424, COL0 = 0x2404;
constexpr uint32_t PACK_ROWS = 0x7531, PACK_COLS = 0x7351;
// the two chains' pairs as one word for the shuffles: bytes 0 and 2 of the
// first, 1 and 3 of the second; and back: (left neighbour's second pixel, own
// first) and (own second, right neighbour's first) of either chain
constexpr uint32_t PACK_CHAINS = 0x7351;
constexpr uint32_t LEFT_A = 0x4020, RIGHT_A = 0x4020, LEFT_B = 0x5030, RIGHT_B = 0x5030;

__device__ __forceinline__ int ld_vol(const int* p) { return *(const volatile int*)p; }

__device__ __forceinline__ bool budget_over(long long t0, long long budget) {
    return clock64() - t0 > budget;
}

// ---- worklist -----------------------------------------------------------------
// A ticket queue: producers and consumers take indices with atomicAdd (no
// compare-and-swap retries under contention).  Slot k is one 64-bit word,
// sequence << 32 | item: sequence i means "free for producer index i",
// i + 1 means "holds the item of index i"; the consumer of index i hands the
// slot to producer index i + cap.  One word per slot, so an item and its
// sequence number become visible together.  An item is the image index
// << ITEM_BITS | the work tile's index within its image, with bit 31 set on
// the tile's first visit (queued by k_wl_init).  The tail and the
// count of queued-or-running tiles (pending) share one 64-bit word, so a push
// moves both with one atomic, and a visit's pushes and the release of its tile
// are one atomic together: the workers' atomics on one word are served one
// after the other, about 2.8 ns each, and head and tail lie in lines of their
// own.  A consumer holding a ticket waits until its item arrives or until no
// tile is queued or running any more.

constexpr int ITEM_BITS = 18;  // work tiles per image <= (16384 / 64)^2 = 2^16 < 2^18
constexpr unsigned ITEM_MASK = (1u << ITEM_BITS) - 1;
constexpr unsigned ITEM_FIRST = 1u << 31;
constexpr unsigned ITEM_IMAGE_MASK = (1u << (31 - ITEM_BITS)) - 1;  // up to 8192 images

__device__ __forceinline__ unsigned long long ld_vol64(const unsigned long long* p) {
    return *(const volatile unsigned long long*)p;
}
__device__ __forceinline__ void st_vol64(unsigned long long* p, unsigned long long v) {
    *(volatile unsigned long long*)p = v;
}

// puts item into position i of the queue
__device__ void wl_put(const Launch& L, unsigned i, unsigned item) {
    const unsigned cap = (unsigned)L.n_rt;
    unsigned long long* slot = L.wl_slots + i % cap;
    long long t0 = clock64();
    while ((unsigned)(ld_vol64(slot) >> 32) != i) {
        if (budget_over(t0, L.wait_budget)) { wait_over(&L.sh->err, L.status); return; }
        __nanosleep(32);
    }
    st_vol64(slot, ((unsigned long long)(i + 1) << 32) | item);
}

// marks work tile t (global index) as wanted; true if the caller has to queue it
__device__ bool wl_want(const Launch& L, int t) {
    for (int it = 0; it < 1024; it++) {
        int s = atomicCAS(&L.wl_state[t], WL_IDLE, WL_QUEUED);
        if (s == WL_IDLE) return true;
        if (s == WL_QUEUED || s == WL_DIRTY) return false;
        if (atomicCAS(&L.wl_state[t], WL_RUNNING, WL_DIRTY) == WL_RUNNING) return false;
    }
    wait_over(&L.sh->err, L.status);
    return false;
}

// takes the next item; false when the queue is drained (or on error)
__device__ bool wl_pop(const Launch& L, unsigned* item) {
    const unsigned cap = (unsigned)L.n_rt;
    const unsigned h = (unsigned)atomicAdd(&L.sh->head, 1);
    unsigned long long* slot = L.wl_slots + h % cap;
    long long t0 = clock64();
    for (;;) {
        const unsigned long long v = ld_vol64(slot);
        if ((unsigned)(v >> 32) == h + 1) {
            st_vol64(slot, (unsigned long long)(h + cap) << 32);
            *item = (unsigned)v;
            return true;
        }
        if ((unsigned)ld_vol64(&L.sh->tp) == 0u || ld_vol(&L.sh->err)) return false;
        if (budget_over(t0, L.wait_budget)) { wait_over(&L.sh->err, L.status); return false; }
        __nanosleep(64);
    }
}

// ---- initial queue, by groups of ORDER_GROUP images: within a group the
// work tiles that hold a strong marker first (a nucleus: its first visit
// raises the background around it, so that the tiles without one start from
// raised halos), and within each of the two classes four colours by the
// parities of tx and ty -- (even, even), (odd, odd), (odd, even), (even,
// odd) -- so that no two tiles of a colour touch, not even at a corner, and a
// tile of the last colour starts with all eight neighbours visited (3136
// tiles/s per batched step against 3101 for a checkerboard of two).  The later the tiles without
// a source come, the fewer visits (per image: 3.04 ms per 16 tiles of 4096^2,
// one group of 16: 2.45 ms); groups of four keep the time of one group with a
// fifth less DRAM traffic, since fewer images' planes are in use at once.  Places within a class are taken by atomics: the
// order inside a class is not fixed, and the result does not depend on it.
// The per-image class counters live in the tile descriptors and are zeroed
// by k_wl_reset at the start of every launch. --------------------------------------
constexpr int ORDER_GROUP = 4;   // images per ordering group: all their sources before their other tiles

__device__ __forceinline__ int order_class(const Launch& L, int i, int* ti_out, int* k_out) {
    const int ti = find_tile(L.tiles, L.ntiles, i, &TileDev::rt_base);
    const TileDev& T = L.tiles[ti];
    const int k = i - T.rt_base, ty = k / T.rtx, tx = k - ty * T.rtx;
    *ti_out = ti;
    *k_out = k;
    // four colours: (even, even), (odd, odd), (odd, even), (even, odd) -- no two
    // tiles of one colour touch, not even at a corner
    const int col = ((tx & 1) == (ty & 1)) ? (tx & 1) : 2 + (tx & 1);
    return (L.rt_src[i] ? 0 : 4) + col;
}

__global__ void k_wl_reset(Launch L) {
    if (L.early) after_previous();
    for (int t = threadIdx.x; t < L.ntiles; t += blockDim.x)
#pragma unroll
        for (int j = 0; j < 8; j++) L.tiles[t].cls[j] = L.tiles[t].cls_pos[j] = 0;
}

// Counts and places are taken once per group of lanes with the same image
// and class, so the counters see one atomic per group instead of one per
// work tile.
__global__ void k_wl_count(Launch L) {
    if (L.early) after_previous();
    const int i = blockIdx.x * blockDim.x + threadIdx.x, lane = threadIdx.x & 31;
    int ti = -1, k = 0, c = 0;
    if (i < L.n_rt) c = order_class(L, i, &ti, &k);
    const int g0 = ti < 0 ? -1 : (ti / ORDER_GROUP) * ORDER_GROUP;  // the group's first image keeps its counters
    const unsigned grp = __match_any_sync(FULL, g0 * 8 + c);
    if (ti >= 0 && lane == __ffs(grp) - 1) atomicAdd(&L.tiles[g0].cls[c], __popc(grp));
}

__global__ void k_wl_init(Launch L) {
    if (L.early) after_previous();
    const int i = blockIdx.x * blockDim.x + threadIdx.x, lane = threadIdx.x & 31;
    if (i == 0) {
        L.sh->head = 0;
        L.sh->tp = ((unsigned long long)(unsigned)L.n_rt << 32) | (unsigned)L.n_rt;
        L.sh->err = 0;
        L.sh->processed = 0;
    }
    int ti = -1, k = 0, c = 0;
    if (i < L.n_rt) c = order_class(L, i, &ti, &k);
    const int g0 = ti < 0 ? -1 : (ti / ORDER_GROUP) * ORDER_GROUP;
    const unsigned grp = __match_any_sync(FULL, g0 * 8 + c);
    const int leader = __ffs(grp) - 1;
    int first = 0;
    if (ti >= 0 && lane == leader) {
        TileDev& T = L.tiles[g0];
        int base = T.rt_base;
        for (int q = 0; q < c; q++) base += T.cls[q];
        first = base + atomicAdd(&T.cls_pos[c], __popc(grp));
    }
    first = __shfl_sync(FULL, first, leader);
    if (ti < 0) return;
    const int pos = first + __popc(grp & ((1u << lane) - 1u));
    L.wl_slots[pos] = ((unsigned long long)(unsigned)(pos + 1) << 32) |
                      (ITEM_FIRST | ((unsigned)ti << ITEM_BITS) | (unsigned)k);
    L.wl_state[i] = WL_QUEUED;
}


// ---- staging ----------------------------------------------------------------------
// Halo pixels of a thread.  One warp: q (0..8) 0-1 top row (-1, 2l + q), 2-3
// bottom row (RT, 2l + q - 2), 4-5 left column (2l + q - 4, -1), 6-7 right column
// (2l + q - 6, RT), 8 the corners, one each on lanes 0-3.  Four warps: q 0 the
// rows, 1 the columns, 2 the corners.
template <int NW>
__host__ __device__ constexpr int halo_count() { return NW == 1 ? 9 : 3; }
template <int NW>
__device__ __forceinline__ void halo_coord(int q, int t, int& hy, int& hx) {
    if constexpr (NW == 1) {
        if (q < 2) { hy = -1; hx = 2 * t + q; }
        else if (q < 4) { hy = RT; hx = 2 * t + q - 2; }
        else if (q < 6) { hy = 2 * t + q - 4; hx = -1; }
        else if (q < 8) { hy = 2 * t + q - 6; hx = RT; }
        else { hy = (t & 2) ? RT : -1; hx = (t & 1) ? RT : -1; }
    } else {
        static_assert(NW == 4, "two lines of 64 pixels per turn");
        const int far = t >> 6, i = t & 63;
        if (q == 0) { hy = far ? RT : -1; hx = i; }
        else if (q == 1) { hy = i; hx = far ? RT : -1; }
        else { hy = (t & 2) ? RT : -1; hx = (t & 1) ? RT : -1; }
    }
}
template <int NW>
__device__ __forceinline__ bool halo_lane(int q, int t) { return q < halo_count<NW>() - 1 || t < 4; }

// the image of a visit, in registers (a descriptor in memory would be read
// again after every fence)
struct Img {
    uint8_t* R;
    const uint8_t* hem8;
    int W, H, rp;
};

// R (and M) of this thread's halo pixels, 0 outside the image
template <int NW>
__device__ __forceinline__ void load_halo(uint8_t* hr, uint8_t* hm, const Img& T, int x0, int y0, int t) {
#pragma unroll
    for (int q = 0; q < halo_count<NW>(); q++) {
        int hy, hx;
        halo_coord<NW>(q, t, hy, hx);
        const int gy = y0 + hy, gx = x0 + hx;
        const bool in = gy >= 0 && gy < T.H && gx >= 0 && gx < T.W && halo_lane<NW>(q, t);
        hr[q] = in ? __ldcg(T.R + (size_t)gy * T.rp + gx) : (uint8_t)0;
        if (hm) hm[q] = in ? __ldg(T.hem8 + (size_t)gy * T.W + gx) : (uint8_t)0;
    }
}

// Stages the tile.  Thread: block row jj of a group of 8 NW, 16-pixel segment seg;
// rows 2j and 2j + 1 of R and M, eight blocks built from them.  R's rows are
// 16-byte aligned; hem8's are where W is a multiple of 16 (odd widths read the
// aligned words around them: with byte loads for both planes a 1025 x 2049
// image took 381 us).
template <int NW>
__device__ __forceinline__ void load_tile(WarpTile& S, const Img& T, int x0, int y0, int t) {
    uint8_t hr[halo_count<NW>()], hm[halo_count<NW>()];
    load_halo<NW>(hr, hm, T, x0, y0, t);
    const uint8_t* const Rg = T.R;
    const uint8_t* const Mg = T.hem8;
    const int W = T.W, H = T.H;
    const int jj = t >> 2, seg = t & 3, x = x0 + seg * 16;
    const uint4 z = make_uint4(0, 0, 0, 0);
    auto put = [&](int j, uint4 rt, uint4 rb, uint4 mt, uint4 mb) {
        const uint32_t rtw[4] = {rt.x, rt.y, rt.z, rt.w}, rbw[4] = {rb.x, rb.y, rb.z, rb.w};
        const uint32_t mtw[4] = {mt.x, mt.y, mt.z, mt.w}, mbw[4] = {mb.x, mb.y, mb.z, mb.w};
#pragma unroll
        for (int u = 0; u < 4; u++) {
            uint2* d = &S.B[j * BS + seg * 8 + 2 * u];
            d[0] = make_uint2(__byte_perm(rtw[u], rbw[u], 0x5410), __byte_perm(mtw[u], mbw[u], 0x5410));
            d[1] = make_uint2(__byte_perm(rtw[u], rbw[u], 0x7632), __byte_perm(mtw[u], mbw[u], 0x7632));
        }
    };
    if ((W & 15) == 0 && x0 + RT <= W && (reinterpret_cast<uintptr_t>(Mg) & 15) == 0) {
#pragma unroll 2
        for (int g = 0; g < NB / (8 * NW); g++) {
            const int j = g * 8 * NW + jj, gy = y0 + 2 * j;
            const size_t o = (size_t)gy * W + x;
            const uint4 rt = gy < H ? __ldcg(reinterpret_cast<const uint4*>(Rg + o)) : z;
            const uint4 rb = gy + 1 < H ? __ldcg(reinterpret_cast<const uint4*>(Rg + o + W)) : z;
            const uint4 mt = gy < H ? __ldg(reinterpret_cast<const uint4*>(Mg + o)) : z;
            const uint4 mb = gy + 1 < H ? __ldg(reinterpret_cast<const uint4*>(Mg + o + W)) : z;
            put(j, rt, rb, mt, mb);
        }
    } else {
#pragma unroll 1
        for (int g = 0; g < NB / (8 * NW); g++) {
            const int j = g * 8 * NW + jj, gy = y0 + 2 * j;
            const bool in0 = x < W && gy < H, in1 = x < W && gy + 1 < H;
            const uint8_t* r = Rg + (size_t)gy * T.rp + x;
            uint4 rt = in0 ? __ldcg(reinterpret_cast<const uint4*>(r)) : z;
            uint4 rb = in1 ? __ldcg(reinterpret_cast<const uint4*>(r + T.rp)) : z;
            const uint4 mt = in0 ? load_px16(Mg, W, H, x, gy) : z, mb = in1 ? load_px16(Mg, W, H, x, gy + 1) : z;
            if (W - x < 16) {  // R's row padding
                rt = clip_px16(rt, max(W - x, 0));
                rb = clip_px16(rb, max(W - x, 0));
            }
            put(j, rt, rb, mt, mb);
        }
    }
#pragma unroll
    for (int q = 0; q < halo_count<NW>(); q++) {
        if (!halo_lane<NW>(q, t)) continue;
        int hy, hx;
        halo_coord<NW>(q, t, hy, hx);
        set_halo_r(S, hy, hx, hr[q]);
        set_halo_m(S, hy, hx, hm[q]);
    }
}

// Writes the tile's R back (row padding takes zeros).
template <int NW>
__device__ __forceinline__ void store_tile(WarpTile& S, const Img& T, int x0, int y0, int t) {
    const int jj = t >> 2, seg = t & 3, x = x0 + seg * 16;
    if (x >= T.W) return;
#pragma unroll 1
    for (int g = 0; g < NB / (8 * NW); g++) {
        const int j = g * 8 * NW + jj, gy = y0 + 2 * j;
        uint32_t top[4], bot[4];
#pragma unroll
        for (int u = 0; u < 4; u++) {
            const uint2* s = &S.B[j * BS + seg * 8 + 2 * u];
            const uint32_t a = s[0].x, b = s[1].x;
            top[u] = __byte_perm(a, b, 0x5410);
            bot[u] = __byte_perm(a, b, 0x7632);
        }
        uint8_t* const r = T.R + (size_t)gy * T.rp + x;
        if (gy < T.H) __stcg(reinterpret_cast<uint4*>(r), make_uint4(top[0], top[1], top[2], top[3]));
        if (gy + 1 < T.H) __stcg(reinterpret_cast<uint4*>(r + T.rp), make_uint4(bot[0], bot[1], bot[2], bot[3]));
    }
}

// Raises the staged halo pixels to the values just read; true if any grew.
template <int NW>
__device__ __forceinline__ bool merge_halo(WarpTile& S, const uint8_t* hr, int t) {
    bool grew = false;
#pragma unroll
    for (int q = 0; q < halo_count<NW>(); q++) {
        if (!halo_lane<NW>(q, t)) continue;
        int hy, hx;
        halo_coord<NW>(q, t, hy, hx);
        if (hr[q] > halo_r(S, hy, hx)) {
            set_halo_r(S, hy, hx, hr[q]);
            grew = true;
        }
    }
    return grew;
}

// ---- sweeps -------------------------------------------------------------------------
// With R <= M everywhere, max(R, min(m, M)) = min(max(R, m), M).

// A row sweep pair: the down sweep (rows 0 -> RT-1) and the up sweep
// (rows RT-1 -> 0) run at once as two chains, one block row of each per step.
// Lane l owns block column l in both chains, so every store to a block comes
// from the one thread that also loads it.  The next block rows are loaded
// before a step; after the step in which the chains meet, each takes over the
// word that the other has just stored there.  Each chain is one full
// directional sweep (every row after the line before it), so a round of the
// two pairs propagates as the four sweeps do, and values only grow towards the
// unique fixed point whatever the order.  Unrolled by four: 1794 us per 16
// tiles of 4096^2 (by two 1877, three 1855, six 1867, eight 1791); one body for
// rows and columns with the permutes in registers takes 1830.
// A and B are the two chains' pixel pairs of the line before; their outer
// neighbours come from lanes l - 1 and l + 1, both chains in one word per
// direction (the edge lanes get their own pair back: its far pixel is a
// neighbour too).  The halo takes no part: it has been let into the border
// pixels before (let_in_halo).
__device__ __forceinline__ void line_step(uint32_t& A, uint32_t& B, uint32_t RA, uint32_t MA, uint32_t RB, uint32_t MB) {
    const uint32_t P = __byte_perm(A, B, PACK_CHAINS);
    const uint32_t L = __shfl_up_sync(FULL, P, 1), Rt = __shfl_down_sync(FULL, P, 1);
    A = min2(__vimax3_u16x2(__byte_perm(L, P, LEFT_A), __byte_perm(P, Rt, RIGHT_A), max2(A, RA)), MA);
    B = min2(__vimax3_u16x2(__byte_perm(L, P, LEFT_B), __byte_perm(P, Rt, RIGHT_B), max2(B, RB)), MB);
}

// With several warps, each takes a band of block rows, and its chains start from
// the lines beside the band as they are (whatever the neighbouring warp has made
// of them meanwhile: any value there is a lower bound).
template <int NW>
__device__ __forceinline__ void row_sweeps(WarpTile& S, int lane, int warp) {
    constexpr int N = NB / NW;
    const int j0 = warp * N;
    uint32_t Pd = 0u, Pu = 0u;
    if (NW > 1 && warp > 0) Pd = __byte_perm(S.B[(j0 - 1) * BS + lane].x, 0u, ROW1);
    if (NW > 1 && warp < NW - 1) Pu = __byte_perm(S.B[(j0 + N) * BS + lane].x, 0u, ROW0);
    uint2 bd = S.B[j0 * BS + lane], bu = S.B[(j0 + N - 1) * BS + lane];
#pragma unroll 4
    for (int k = 0; k < N; k++) {  // down: rows 2jd, 2jd + 1; up: rows 2ju + 1, 2ju
        const int jd = j0 + k, ju = j0 + N - 1 - k;
        uint2 nd = S.B[min(jd + 1, j0 + N - 1) * BS + lane], nu = S.B[max(ju - 1, j0) * BS + lane];
        line_step(Pd, Pu, __byte_perm(bd.x, 0u, ROW0), __byte_perm(bd.y, 0u, ROW0), __byte_perm(bu.x, 0u, ROW1),
                  __byte_perm(bu.y, 0u, ROW1));
        const uint32_t d0 = Pd, u1 = Pu;
        line_step(Pd, Pu, __byte_perm(bd.x, 0u, ROW1), __byte_perm(bd.y, 0u, ROW1), __byte_perm(bu.x, 0u, ROW0),
                  __byte_perm(bu.y, 0u, ROW0));
        const uint32_t wd = __byte_perm(d0, Pd, PACK_ROWS), wu = __byte_perm(Pu, u1, PACK_ROWS);
        S.B[jd * BS + lane].x = wd;
        S.B[ju * BS + lane].x = wu;
        if (k == N / 2 - 1) { nd.x = wu; nu.x = wd; }
        bd = nd;
        bu = nu;
    }
}

// The column sweep pair: right (columns 0 -> RT-1) and left (RT-1 -> 0) at
// once, lane l owning block row l (rows 2l, 2l + 1) in both chains.
template <int NW>
__device__ __forceinline__ void col_sweeps(WarpTile& S, int lane, int warp) {
    constexpr int N = NB / NW;
    const int i0 = warp * N;
    uint32_t Cr = 0u, Cl = 0u;
    uint2* const B = S.B + lane * BS;
    if (NW > 1 && warp > 0) Cr = B[i0 - 1].x;
    if (NW > 1 && warp < NW - 1) Cl = __byte_perm(B[i0 + N].x, 0u, COL0);
    uint2 br = B[i0], bl = B[i0 + N - 1];
#pragma unroll 4
    for (int k = 0; k < N; k++) {
        const int ir = i0 + k, il = i0 + N - 1 - k;
        uint2 nr = B[min(ir + 1, i0 + N - 1)], nl = B[max(il - 1, i0)];
        line_step(Cr, Cl, __byte_perm(br.x, 0u, COL0), __byte_perm(br.y, 0u, COL0), bl.x, bl.y);
        const uint32_t r0 = Cr, l1 = Cl;
        line_step(Cr, Cl, br.x, br.y, __byte_perm(bl.x, 0u, COL0), __byte_perm(bl.y, 0u, COL0));
        const uint32_t wr = __byte_perm(r0, Cr, PACK_COLS), wl = __byte_perm(Cl, l1, PACK_COLS);
        B[ir].x = wr;
        B[il].x = wl;
        if (k == N / 2 - 1) { nr.x = wl; nl.x = wr; }
        br = nr;
        bl = nl;
    }
}

// One round: the row sweep pair, then the column sweep pair.  __syncwarp
// orders each pair's stores before the next pair's loads (the pairs map
// lanes to blocks differently).
template <int NW>
__device__ __forceinline__ void sweep_round(WarpTile& S, const Worker<NW>& me) {
    row_sweeps<NW>(S, me.lane, me.warp);
    me.sync();
    col_sweeps<NW>(S, me.lane, me.warp);
    me.sync();
}

// Whether some pixel of the tile can still be raised by one of its 8
// neighbours in the tile: the exact convergence test, two pixels per lane and
// row, with no dependent chain; it stops at the first 16-row group that has one.
// With several warps, each looks at its band of block rows, and they agree.
template <int NW>
__device__ __forceinline__ bool can_raise(const WarpTile& S, const Worker<NW>& me) {
    const int lane = me.lane, warp = me.warp;
    constexpr int N = NB / NW;
    const int j0 = warp * N;
    // maxima of R over the three columns around each pixel, for the two rows
    // of a block row: the neighbours' block words hold both rows
    auto hmax = [&](uint32_t w, uint32_t& top, uint32_t& bot) {
        const uint32_t L = __shfl_up_sync(FULL, w, 1), Rt = __shfl_down_sync(FULL, w, 1);
        top = __vimax3_u16x2(__byte_perm(L, w, 0x4010), __byte_perm(w, Rt, 0x4010), __byte_perm(w, 0u, ROW0));
        bot = __vimax3_u16x2(__byte_perm(L, w, 0x6030), __byte_perm(w, Rt, 0x6030), __byte_perm(w, 0u, ROW1));
    };
    uint32_t hp = 0u, h0, h1;  // maxima of the row before block row j, and of its two rows
    if (NW > 1 && warp > 0) hmax(S.B[(j0 - 1) * BS + lane].x, h0, hp);
    uint2 b = S.B[j0 * BS + lane];
    hmax(b.x, h0, h1);
    uint32_t v = 0u;
#pragma unroll 1
    for (int g = 0; g < N / 8; g++) {
#pragma unroll
        for (int jj = 0; jj < 8; jj++) {
            const int j = j0 + g * 8 + jj;
            uint2 nb = make_uint2(0u, 0u);
            uint32_t n0 = 0u, n1 = 0u;
            if (j + 1 < NB) {
                nb = S.B[(j + 1) * BS + lane];
                hmax(nb.x, n0, n1);
            }
            const uint32_t r0 = min2(__vimax3_u16x2(hp, h0, h1), __byte_perm(b.y, 0u, ROW0));
            const uint32_t r1 = min2(__vimax3_u16x2(h0, h1, n0), __byte_perm(b.y, 0u, ROW1));
            v |= __byte_perm(r0, r1, PACK_ROWS) ^ b.x;
            hp = h1;
            h0 = n0;
            h1 = n1;
            b = nb;
        }
        if constexpr (NW == 1)
            if (__any_sync(FULL, v != 0u)) return true;
    }
    if constexpr (NW == 1) return false; else return me.any(v != 0u);
}

// Lets the halo into the tile: raises each border pixel by the halo pixels
// around it; true if one grew.  The halo only acts through the border, so the
// sweeps and the test need not look at it (they read a halo word per line
// before), and when the tile was at a fixed point before the halo grew, no
// pixel can be raised if no border pixel grew here.
template <int NW>
__device__ __forceinline__ bool let_in_halo(WarpTile& S, const Worker<NW>& me) {
    const int lane = me.lane, warp = me.warp;
    // lane l: border pixels 2l and 2l + 1 of a side in one block word, and the
    // four halo pixels around them (the halo lines hold the corners too, with
    // the same values as the halo rows)
    const int i = 2 * lane;
    bool v = false;
    // pixels at bits s0 and s1 of w.x, under the halo values a, b, c, d
    auto raise = [&](uint2* w, int a, int b, int c, int d, int s0, int s1) {
        const uint2 q = *w;
        const int r0 = (int)((q.x >> s0) & 0xffu), r1 = (int)((q.x >> s1) & 0xffu);
        const int n0 = max(r0, min(max(max(a, b), c), (int)((q.y >> s0) & 0xffu)));
        const int n1 = max(r1, min(max(max(b, c), d), (int)((q.y >> s1) & 0xffu)));
        if (n0 != r0 || n1 != r1) {
            w->x = q.x + ((uint32_t)(n0 - r0) << s0) + ((uint32_t)(n1 - r1) << s1);
            v = true;
        }
    };
    if (NW == 1 || warp == 0)
        raise(&S.B[lane], S.HRow[0][i] & 0xff, S.HRow[0][i + 1] & 0xff, S.HRow[0][i + 2] & 0xff, S.HRow[0][i + 3] & 0xff, 0, 8);
    if (NW == 1 || warp == 1)
        raise(&S.B[(NB - 1) * BS + lane], S.HRow[1][i] >> 16, S.HRow[1][i + 1] >> 16, S.HRow[1][i + 2] >> 16,
              S.HRow[1][i + 3] >> 16, 16, 24);
    me.sync();  // the corner blocks belong to a row and to a column
    if (NW == 1 || warp == 2)
        raise(&S.B[lane * BS], S.HC[0][i] & 0xff, S.HC[0][i + 1] & 0xff, S.HC[0][i + 2] & 0xff, S.HC[0][i + 3] & 0xff, 0, 16);
    if (NW == 1 || warp == 3)
        raise(&S.B[lane * BS + NB - 1], S.HC[1][i] >> 16, S.HC[1][i + 1] >> 16, S.HC[1][i + 2] >> 16, S.HC[1][i + 3] >> 16, 8, 24);
    const bool any = me.any(v);
    me.sync();
    return any;
}

// ---- neighbour requests ---------------------------------------------------------------
// Side s (0 top, 1 bottom, 2 left, 3 right) of the tile, after the tile is at
// a fixed point: halo pixel h of the side (h = -1..RT along it) needs its
// tile queued when a border pixel changed since the last requests and next
// to h can raise it.  h = -1 and h = RT are the halo corners, which belong
// to the diagonal neighbours.  The side's border then becomes the reference
// for the next requests.
// With four warps, each takes a side.
template <int NW>
__device__ __forceinline__ void side_requests(WarpTile& S, const Worker<NW>& me) {
    // lane l holds border pixels 2l and 2l + 1 of every side: one block word
    // of R (top: block (0, l) bytes 0, 1; bottom: block (NB-1, l) bytes 2, 3;
    // left: block (l, 0) bytes 0, 2; right: block (l, NB-1) bytes 1, 3); the
    // changed values of the pixels beyond its pair come from the next lanes
    const int lane = me.lane;
    const int p0 = 2 * lane, p1 = 2 * lane + 1;
    // (one warp: the four loads are in flight together)
    const uint32_t wt = S.B[lane].x, wb = S.B[(NB - 1) * BS + lane].x;
    const uint32_t wl = S.B[lane * BS].x, wr = S.B[lane * BS + NB - 1].x;
#pragma unroll
    for (int s = 0; s < 4; s++) {
        if (NW > 1 && s != me.warp) continue;
        const uint32_t w = s == 0 ? wt : s == 1 ? wb : s == 2 ? wl : wr;
        const int sh0 = s == 0 ? 0 : s == 1 ? 16 : s == 2 ? 0 : 8;
        const int sh1 = s == 0 ? 8 : s == 1 ? 24 : s == 2 ? 16 : 24;
        const int v0 = (int)((w >> sh0) & 0xffu), v1 = (int)((w >> sh1) & 0xffu);
        // border values changed since the last requests (else 0)
        const int c0 = v0 != (int)S.B0[s][p0] ? v0 : 0, c1 = v1 != (int)S.B0[s][p1] ? v1 : 0;
        int cl = __shfl_up_sync(FULL, c1, 1), cr = __shfl_down_sync(FULL, c0, 1);
        if (lane == 0) cl = 0;
        if (lane == 31) cr = 0;
        const int m0 = max(max(cl, c0), c1), m1 = max(max(c0, c1), cr);
        // the halo pixels facing p0, p1: R and M
        int hr0, hr1, hm0, hm1;
        if (s == 0) {
            hr0 = (int)(S.HRow[0][p0 + 1] & 0xffu); hr1 = (int)(S.HRow[0][p1 + 1] & 0xffu);
            hm0 = S.HMr[0][p0 + 1]; hm1 = S.HMr[0][p1 + 1];
        } else if (s == 1) {
            hr0 = (int)(S.HRow[1][p0 + 1] >> 16); hr1 = (int)(S.HRow[1][p1 + 1] >> 16);
            hm0 = S.HMr[1][p0 + 1]; hm1 = S.HMr[1][p1 + 1];
        } else if (s == 2) {
            hr0 = (int)(S.HC[0][p0 + 1] & 0xffu); hr1 = (int)(S.HC[0][p1 + 1] & 0xffu);
            hm0 = S.HMc[0][p0 + 1]; hm1 = S.HMc[0][p1 + 1];
        } else {
            hr0 = (int)(S.HC[1][p0 + 1] >> 16); hr1 = (int)(S.HC[1][p1 + 1] >> 16);
            hm0 = S.HMc[1][p0 + 1]; hm1 = S.HMc[1][p1 + 1];
        }
        const bool line = min(m0, hm0) > hr0 || min(m1, hm1) > hr1;
        // the corners (-1 and RT along the side) belong to the diagonal
        // neighbours; corner pixels are read from the halo rows
        const int kl = s == 1 ? 1 : 0, kh = s == 0 ? 0 : 1;        // halo row of the low / high corner
        const int il = s == 3 ? RT + 1 : 0, ih = s == 2 ? 0 : RT + 1;  // its index in that row
        bool lo = false, hi = false;
        if (lane == 0) {
            const int r = kl ? (int)(S.HRow[1][il] >> 16) : (int)(S.HRow[0][il] & 0xffu);
            lo = min(c0, (int)S.HMr[kl][il]) > r;
        }
        if (lane == 31) {
            const int r = kh ? (int)(S.HRow[1][ih] >> 16) : (int)(S.HRow[0][ih] & 0xffu);
            hi = min(c1, (int)S.HMr[kh][ih]) > r;
        }
        const bool anyl = __any_sync(FULL, line), anylo = __any_sync(FULL, lo), anyhi = __any_sync(FULL, hi);
        if (lane == 0) {
            // corners: top -> UL, UR; bottom -> DL, DR; left -> UL, DL; right -> UR, DR
            const int fl = s == 0 ? 4 : s == 1 ? 6 : s == 2 ? 4 : 5;
            const int fh = s == 0 ? 5 : s == 1 ? 7 : s == 2 ? 6 : 7;
            if (anyl) S.flags[s] = 1;
            if (anylo) S.flags[fl] = 1;
            if (anyhi) S.flags[fh] = 1;
        }
        // the side's border becomes the reference for the next requests
        S.B0[s][p0] = (uint8_t)v0;
        S.B0[s][p1] = (uint8_t)v1;
    }
    me.sync();
}

// A worker is a warp where each has many tiles to do (a warp needs no barriers,
// and the workers hide one another's latency), and a CTA of four warps where
// not: then the longest row of dependent visits sets the time, and a visit is
// serial.  A round of sweeps is 64 steps of two shuffles and a few dependent
// operations for a warp, 11500 clocks with its test, of which a visit takes two
// or so, and 16 steps in four bands of 16 lines for a team, 3600 clocks with the
// barriers; what has to cross bands costs more rounds (of 64 tiles, 6 rounds per
// tile in all by warps, 10 by teams).  The team's warps also share the loads, the
// requests and the write-back.  512^2: 141 -> 85 us; 1025 x 2049: 158 -> 107 us;
// 4096^2: 282 -> 260 us.
template <int NW>
__global__ void __launch_bounds__(32 * NW, NW == 1 ? RECON_MIN_BLOCKS : TEAM_MIN_BLOCKS) k_recon(Launch L) {
    if (L.early) after_previous();
    extern __shared__ __align__(16) unsigned char smraw[];
    WarpTile& S = *reinterpret_cast<WarpTile*>(smraw);
    const Worker<NW> me;
    const int t = me.t, lane = me.lane;
    int visits = 0;  // tile processings of this worker (diagnostic), added once at exit
    if (t < 9) S.flags[t] = 0;
    me.sync();
    for (;;) {
        unsigned item = 0;
        int ok = 0;
        if (t == 0) ok = wl_pop(L, &item) ? 1 : 0;
        ok = me.from_first(S, ok);
        if (!ok) break;
        item = (unsigned)me.from_first(S, (int)item);
        const int ti = (int)((item >> ITEM_BITS) & ITEM_IMAGE_MASK), k = (int)(item & ITEM_MASK);
        // a tile released by a visit was at a fixed point, so on later visits
        // only its border can have become raisable; its first visit starts
        // from the marker and sweeps at once
        bool sweep_now = (item & ITEM_FIRST) != 0, full_check = false;
        const TileDev& D = L.tiles[ti];
        const Img T{D.R, D.hem8, D.W, D.H, D.rp};
        const int rx = D.rtx, ry = D.rty, base = D.rt_base;
        const int tile = base + k, ty = k / rx, tx = k - ty * rx;
        const int x0 = tx * RT, y0 = ty * RT;
        if (t == 0) atomicExch(&L.wl_state[tile], WL_RUNNING);
        visits++;
        __threadfence();
        me.sync();
        load_tile<NW>(S, T, x0, y0, t);
        me.sync();
        // the border as loaded is the reference for the first requests (lane l:
        // border pixels 2l, 2l + 1 of each side, from one block word per side)
        if (NW == 1 || me.warp == 0) {
            const uint32_t wt = S.B[lane].x, wb = S.B[(NB - 1) * BS + lane].x;
            const uint32_t wl = S.B[lane * BS].x, wr = S.B[lane * BS + NB - 1].x;
            S.B0[0][2 * lane] = (uint8_t)wt;
            S.B0[0][2 * lane + 1] = (uint8_t)(wt >> 8);
            S.B0[1][2 * lane] = (uint8_t)(wb >> 16);
            S.B0[1][2 * lane + 1] = (uint8_t)(wb >> 24);
            S.B0[2][2 * lane] = (uint8_t)wl;
            S.B0[2][2 * lane + 1] = (uint8_t)(wl >> 16);
            S.B0[3][2 * lane] = (uint8_t)(wr >> 8);
            S.B0[3][2 * lane + 1] = (uint8_t)(wr >> 24);
        }
        me.sync();
        for (;;) {
            int nr = 0, queue = -1;
            bool more = false;
            bool go = let_in_halo<NW>(S, me) || sweep_now || (full_check && can_raise<NW>(S, me));
            sweep_now = false;
            while (go) {
                if (nr >= MAX_ROUNDS) { more = true; break; }
                sweep_round<NW>(S, me);
                nr++;
                go = can_raise<NW>(S, me);
            }
            full_check = more;  // otherwise the interior is at a fixed point now
            bool grew = false;
            if (nr > 0) {
                // the halo read only decides which neighbours to queue; it is
                // issued before the write-back so that the two overlap (a stale
                // value can only cause a needless request)
                uint8_t hr[halo_count<NW>()];
                load_halo<NW>(hr, nullptr, T, x0, y0, t);
                store_tile<NW>(S, T, x0, y0, t);
                // the stores drain while the requests are worked out in shared memory
                grew = me.any(merge_halo<NW>(S, hr, t));
                me.sync();
                side_requests<NW>(S, me);
                if (more && t == 0) S.flags[8] = 1;  // not converged within MAX_ROUNDS: run again
                __threadfence();  // this tile's pixels before any request
                me.sync();
                if (t < 9 && S.flags[t]) {
                    int target = -1;
                    switch (t) {
                        case 0: if (ty > 0) target = k - rx; break;
                        case 1: if (ty + 1 < ry) target = k + rx; break;
                        case 2: if (tx > 0) target = k - 1; break;
                        case 3: if (tx + 1 < rx) target = k + 1; break;
                        case 4: if (ty > 0 && tx > 0) target = k - rx - 1; break;
                        case 5: if (ty > 0 && tx + 1 < rx) target = k - rx + 1; break;
                        case 6: if (ty + 1 < ry && tx > 0) target = k + rx - 1; break;
                        case 7: if (ty + 1 < ry && tx + 1 < rx) target = k + rx + 1; break;
                        default: target = k; break;
                    }
                    S.flags[t] = 0;
                    if (target >= 0 && wl_want(L, base + target)) queue = target;
                }
            }
            // The tile is released (unless its fresher halo is to be looked at
            // again) before the wanted neighbours enter the queue; until the one
            // atomic that adds them and takes the tile off, it counts as pending.
            // No fence is needed before the release: every write-back above was
            // followed by one.
            int again = grew ? 1 : 0;
            if (NW == 1 || me.warp == 0) {
                const unsigned qm = __ballot_sync(FULL, queue >= 0);
                unsigned at = 0;
                if (lane == 0) {
                    if (!grew && atomicCAS(&L.wl_state[tile], WL_RUNNING, WL_IDLE) != WL_RUNNING) {
                        atomicExch(&L.wl_state[tile], WL_RUNNING);  // a neighbour raised the halo meanwhile
                        again = 2;
                    }
                    const int n = __popc(qm), less = again ? 0 : 1;
                    if (n || less)
                        at = (unsigned)(atomicAdd(&L.sh->tp, ((unsigned long long)n << 32) + (unsigned long long)(long long)(n - less)) >> 32);
                }
                at = __shfl_sync(FULL, at, 0);
                if (queue >= 0) wl_put(L, at + __popc(qm & ((1u << lane) - 1u)), ((unsigned)ti << ITEM_BITS) | (unsigned)queue);
            }
            again = me.from_first(S, again);
            me.sync();
            if (again == 1) continue;  // the fresher halo may raise pixels: check again
            if (!again) break;
            visits++;
            __threadfence();
            if (me.any(ld_vol(&L.sh->err) != 0)) break;
            // only the halo can have changed: the interior belongs to this worker
            uint8_t hr[halo_count<NW>()];
            load_halo<NW>(hr, nullptr, T, x0, y0, t);
            merge_halo<NW>(S, hr, t);
            me.sync();
        }
        me.sync();
    }
    if (t == 0 && visits) atomicAdd(&L.sh->processed, visits);
}

template <int NW>
static int recon_resident(int sms) {
    int per = 0;
    cudaFuncSetAttribute(k_recon<NW>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(WarpTile));
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_recon<NW>, 32 * NW, sizeof(WarpTile));
    return sms * (per < 1 ? 1 : per);
}

// resident workers of the reconstruction kernels: warps, and teams
void recon_grid(int device, int* warps, int* teams) {
    int sms = 0;
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device);
    *warps = recon_resident<1>(sms);
    *teams = recon_resident<4>(sms);
}

void launch_recon(const Launch& L, int warps, int warps_cap, int teams_cap, cudaStream_t s, Profiler* pf) {
    if (L.n_rt == 0) return;
    pf->begin("recon_init", s);
    launch_behind(L.early && pf->overlap(), k_wl_reset, 1, 256, 0, s, L);
    launch_behind(L.early && pf->overlap(), k_wl_count, (L.n_rt + 255) / 256, 256, 0, s, L);
    launch_behind(L.early && pf->overlap(), k_wl_init, (L.n_rt + 255) / 256, 256, 0, s, L);
    pf->end("recon_init", s);
    pf->begin("recon", s);
    if (L.n_rt < TEAM_TILES * warps_cap) {  // as many teams of all as `warps` is of all warps
        const int teams = std::max(1, (int)((long long)teams_cap * warps / warps_cap));
        launch_behind(L.early && pf->overlap(), k_recon<4>, std::min(L.n_rt, teams), 128, sizeof(WarpTile), s, L);
    } else {
        launch_behind(L.early && pf->overlap(), k_recon<1>, std::min(L.n_rt, warps), 32, sizeof(WarpTile), s, L);
    }
    pf->end("recon", s);
}

}  // namespace nucseg
