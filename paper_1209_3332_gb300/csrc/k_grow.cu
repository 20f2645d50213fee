// Growth of a binary marker through a binary mask, 8-connected (the
// hysteresis of the Canny edges; Table I "RBC detection", Vincent's MR on 0/1
// planes): out = the mask components that hold a marker pixel.
//
// Both planes are bits, tile-major: a 64x64 work tile is 64 words of 64 bits
// (row r, bit x), 512 contiguous bytes, so one warp holds a tile's marker
// and mask in registers, two rows per lane.  A step spreads the marker to the
// rows above and below (shuffles) and along whole runs of the mask inside a
// row: adding the marker to the mask carries through each run from its first
// marker bit upwards, and the same on bit-reversed words fills downwards.
// Steps repeat until none changes a bit; where 16 were not enough in a mask of a
// quarter of the tile and more, whole runs of the columns are filled between
// further steps, by doubling over the lanes: one marker pixel in a mask of 2048^2,
// 279 us by steps alone and 173 so (152 from the eighth step on, but then eight
// edge planes of 4096^2, whose tiles need few, take 1 % longer; thin masks that
// wind through a tile gain nothing from it).
//
// The tiles are driven by a ticket queue as in the reconstruction (k_recon.cu):
// workers first draw groups of tiles from a counter and process those whose
// marker is not empty; a processed tile queues each neighbour that holds a
// mask pixel beside one of its marker pixels that is not marked yet.  pending
// counts groups not finished and tiles queued or running; a worker leaves when
// it reaches zero, so the work never depends on which workers are resident.
// Every spin wait is bounded by the pipe's cycle budget (ST_TIMEOUT).
//
// Bound: the latency of a visit (loads, up to about twenty steps, fence and state
// atomics) and of a few dependent visits; the planes are 2/8 B per pixel in,
// 1 B out by k_grow_out.  Eight 4096^2 edge planes: 177 us and 31 for the bytes,
// one red blood cell plane 28 and 9 (414 and 54 us on bytes with the grayscale
// reconstruction kernel).
#include <algorithm>

#include "internal.cuh"

namespace nucseg {

constexpr unsigned FULLG = 0xffffffffu;
typedef unsigned long long u64;

__device__ __forceinline__ u64 vol64(const u64* p) { return *(const volatile u64*)p; }

// ---- queue ------------------------------------------------------------------------
// Slot k of the ring (one per tile) holds lap << 32 | item: 2 l means free for
// lap l, 2 l + 1 holds the item of lap l, so a zeroed ring is free for lap 0.
// Puts item into position i of the queue.
__device__ void grow_put(const GrowLaunch& G, unsigned i, unsigned item) {
    const unsigned cap = (unsigned)G.n_rt, lap = i / cap;
    u64* slot = G.slots + (i - lap * cap);
    const long long t0 = clock64();
    while ((unsigned)(vol64(slot) >> 32) != 2u * lap) {
        if (clock64() - t0 > G.wait_budget) { wait_over(&G.sh->err, G.status); return; }
        __nanosleep(32);
    }
    *(volatile u64*)slot = ((u64)(2u * lap + 1u) << 32) | item;
}

// Marks tile t as wanted; true if the caller has to queue it.
__device__ bool grow_want(const GrowLaunch& G, int t) {
    for (int it = 0; it < 1024; it++) {
        const int s = atomicCAS(&G.state[t], WL_IDLE, WL_QUEUED);
        if (s == WL_IDLE) return true;
        if (s == WL_QUEUED || s == WL_DIRTY) return false;
        if (atomicCAS(&G.state[t], WL_RUNNING, WL_DIRTY) == WL_RUNNING) return false;
    }
    wait_over(&G.sh->err, G.status);
    return false;
}

// the next queued tile, or -1 when nothing is left (or on an error)
__device__ int grow_pop(const GrowLaunch& G) {
    const unsigned h = (unsigned)atomicAdd(&G.sh->head, 1), cap = (unsigned)G.n_rt, lap = h / cap;
    u64* slot = G.slots + (h - lap * cap);
    const long long t0 = clock64();
    for (;;) {
        const u64 v = vol64(slot);
        if ((unsigned)(v >> 32) == 2u * lap + 1u) {
            *(volatile u64*)slot = (u64)(2u * lap + 2u) << 32;
            return (int)(unsigned)v;
        }
        if ((unsigned)vol64(&G.sh->tp) == 0u || *(const volatile int*)&G.sh->err) return -1;
        if (clock64() - t0 > G.wait_budget) { wait_over(&G.sh->err, G.status); return -1; }
        __nanosleep(64);
    }
}

// ---- one tile ----------------------------------------------------------------------
// the runs of c that hold a bit of s (s within c), from that bit upwards
__device__ __forceinline__ u64 fill_up(u64 s, u64 c) { return (c & ~(c + s)) | s; }
// rc = c bit-reversed
__device__ __forceinline__ u64 fill_runs(u64 s, u64 c, u64 rc) {
    s = fill_up(s, c);
    return __brevll(fill_up(__brevll(s), rc));
}
__device__ __forceinline__ u64 spread(u64 v) { return v | (v << 1) | (v >> 1); }
// The same along the columns: rows 2 l and 2 l + 1 in lane l, runs joined over
// 1, 2, 4, 8 and 16 lanes in either direction.
__device__ __forceinline__ void fill_columns(u64& s0, u64& s1, const ulonglong2 c, int lane) {
#pragma unroll
    for (int up = 0; up < 2; up++) {
        // the row of the lane that the next lane looks at: its marker, and whether it lets through
        u64 g = up ? s0 | (c.x & s1) : s1 | (c.y & s0), p = c.x & c.y;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const u64 gn = up ? __shfl_down_sync(FULLG, g, d) : __shfl_up_sync(FULLG, g, d);
            const u64 pn = up ? __shfl_down_sync(FULLG, p, d) : __shfl_up_sync(FULLG, p, d);
            if (up ? lane + d < 32 : lane >= d) {
                g |= p & gn;
                p &= pn;
            }
        }
        u64 in = up ? __shfl_down_sync(FULLG, g, 1) : __shfl_up_sync(FULLG, g, 1);
        if (lane == (up ? 31 : 0)) in = 0ull;
        if (up) {
            s1 |= c.y & in;
            s0 |= c.x & s1;
        } else {
            s0 |= c.x & in;
            s1 |= c.y & s0;
        }
    }
}
__device__ __forceinline__ ulonglong2 rows2(const u64* plane, int t, int lane) {
    return __ldcg(reinterpret_cast<const ulonglong2*>(plane + (size_t)t * RT) + lane);
}

// Grows tile t (state WL_RUNNING) to its fixed point, queues neighbours, and
// releases it.  drop: what the release takes from the pending count (0 or 1),
// in the same atomic that adds the queued neighbours: every worker's atomics
// meet at this one word, at about 2.8 ns each.
__device__ void grow_tile(const GrowLaunch& G, int t, int drop, int lane) {
    const CannyDesc& d = G.tab[G.tab.find(t, &CannyDesc::rt_base)];
    const int rx = (d.W + RT - 1) / RT, ry = (d.H + RT - 1) / RT, k = t - d.rt_base, ty = k / rx, tx = k - ty * rx;
    const bool hu = ty > 0, hd = ty + 1 < ry, hl = tx > 0, hr = tx + 1 < rx;
    const ulonglong2 c = rows2(G.mask, t, lane);
    const u64 rc0 = __brevll(c.x), rc1 = __brevll(c.y);
    const ulonglong2 z = make_ulonglong2(0, 0);
    // mask of the neighbours' facing pixels: rows 2 l, 2 l + 1 of the columns, lanes 0 / 31 the rows and corners
    const ulonglong2 cl = hl ? rows2(G.mask, t - 1, lane) : z, cr = hr ? rows2(G.mask, t + 1, lane) : z;
    auto word = [&](const u64* plane, bool in, int tt, int row) -> u64 { return in ? __ldcg(plane + (size_t)tt * RT + row) : 0ull; };
    // lane 0 looks after the row above, lane 31 after the row below
    const bool up = lane == 0, edge = lane == 0 || lane == 31;
    const bool hv = up ? hu : hd;
    const int tv = up ? t - rx : t + rx, rowv = up ? RT - 1 : 0;
    const u64 cv = word(G.mask, edge && hv, tv, rowv);
    const u64 cvl = word(G.mask, edge && hv && hl, tv - 1, rowv), cvr = word(G.mask, edge && hv && hr, tv + 1, rowv);
    for (int visit = 0;; visit++) {
        const ulonglong2 s = rows2(G.marker, t, lane);
        const ulonglong2 sl = hl ? rows2(G.marker, t - 1, lane) : z, sr = hr ? rows2(G.marker, t + 1, lane) : z;
        const u64 sv = word(G.marker, edge && hv, tv, rowv);
        const u64 svl = word(G.marker, edge && hv && hl, tv - 1, rowv), svr = word(G.marker, edge && hv && hr, tv + 1, rowv);
        // marker pixels of the left (right) column beside rows 2 l and 2 l + 1
        unsigned l0 = (unsigned)(sl.x >> 63), l1 = (unsigned)(sl.y >> 63), r0 = (unsigned)(sr.x & 1), r1 = (unsigned)(sr.y & 1);
        unsigned la = __shfl_up_sync(FULLG, l1, 1), lb = __shfl_down_sync(FULLG, l0, 1);
        unsigned ra = __shfl_up_sync(FULLG, r1, 1), rb = __shfl_down_sync(FULLG, r0, 1);
        if (lane == 0) { la = (unsigned)(svl >> 63); ra = (unsigned)(svr & 1); }
        if (lane == 31) { lb = (unsigned)(svl >> 63); rb = (unsigned)(svr & 1); }
        const u64 in0 = (u64)(la | l0 | l1) | ((u64)(ra | r0 | r1) << 63);
        const u64 in1 = (u64)(l0 | l1 | lb) | ((u64)(r0 | r1 | rb) << 63);
        u64 s0 = s.x, s1 = s.y;
        auto step = [&]() -> bool {
            u64 a = __shfl_up_sync(FULLG, s1, 1), b = __shfl_down_sync(FULLG, s0, 1);
            if (lane == 0) a = sv;
            if (lane == 31) b = sv;
            const u64 n0 = fill_runs(s0 | ((spread(a | s0 | s1) | in0) & c.x), c.x, rc0);
            const u64 n1 = fill_runs(s1 | ((spread(n0 | s1 | b) | in1) & c.y), c.y, rc1);
            const bool ch = ((n0 ^ s0) | (n1 ^ s1)) != 0ull;
            s0 = n0;
            s1 = n1;
            return __any_sync(FULLG, ch);
        };
        bool go = true;
#pragma unroll 1
        for (int i = 0; go && i < 16; i++) go = step();
        if (go) {
            const bool wide = __reduce_add_sync(FULLG, (unsigned)(__popcll(c.x) + __popcll(c.y))) >= RT * RT / 4;
#pragma unroll 1
            do {
                if (wide) fill_columns(s0, s1, c, lane);
#pragma unroll 1
                for (int i = 0; go && i < 8; i++) go = step();
            } while (go);
        }
        if (__any_sync(FULLG, ((s0 ^ s.x) | (s1 ^ s.y)) != 0ull))
            __stcg(reinterpret_cast<ulonglong2*>(G.marker + (size_t)t * RT) + lane, make_ulonglong2(s0, s1));
        // open mask pixels of the neighbours beside a marker pixel of this tile
        // (their marker as loaded: stale values only cause needless requests)
        unsigned b0 = (unsigned)(s0 & 1), b1 = (unsigned)(s1 & 1), e0 = (unsigned)(s0 >> 63), e1 = (unsigned)(s1 >> 63);
        unsigned ba = __shfl_up_sync(FULLG, b1, 1), bb = __shfl_down_sync(FULLG, b0, 1);
        unsigned ea = __shfl_up_sync(FULLG, e1, 1), eb = __shfl_down_sync(FULLG, e0, 1);
        if (lane == 0) ba = ea = 0;
        if (lane == 31) bb = eb = 0;
        const u64 ol0 = cl.x & ~sl.x, ol1 = cl.y & ~sl.y, or0 = cr.x & ~sr.x, or1 = cr.y & ~sr.y;
        const bool wl = ((ba | b0 | b1) & (unsigned)(ol0 >> 63)) | ((b0 | b1 | bb) & (unsigned)(ol1 >> 63));
        const bool wr = ((ea | e0 | e1) & (unsigned)(or0 & 1)) | ((e0 | e1 | eb) & (unsigned)(or1 & 1));
        const u64 line = up ? s0 : s1;  // this tile's row that faces the row above / below
        unsigned want = 0;              // lanes 0 and 31: bit 0 the tile there, 1 and 2 its left and right corner
        if (edge)
            want = (unsigned)((spread(line) & cv & ~sv) != 0ull) | (unsigned)((line & 1) & ((cvl & ~svl) >> 63)) << 1 |
                   (unsigned)((line >> 63) & (cvr & ~svr) & 1) << 2;
        const unsigned wu = __shfl_sync(FULLG, want, 0), wd = __shfl_sync(FULLG, want, 31);
        const unsigned mask9 = (wu & 1) | (wd & 1) << 1 | (unsigned)__any_sync(FULLG, wl) << 2 |
                               (unsigned)__any_sync(FULLG, wr) << 3 | (wu >> 1) << 4 | (wd >> 1) << 6;
        __threadfence();  // this tile's marker before any request
        __syncwarp();
        bool queue = false;
        int off = 0;
        if (lane < 8 && ((mask9 >> lane) & 1u)) {
            // up, down, left, right, up-left, up-right, down-left, down-right
            const int dt[8] = {-rx, rx, -1, 1, -rx - 1, -rx + 1, rx - 1, rx + 1};
#pragma unroll
            for (int q = 0; q < 8; q++)
                if (q == lane) off = dt[q];
            queue = grow_want(G, t + off);
        }
        const unsigned qm = __ballot_sync(FULLG, queue);
        // the tile is released before its neighbours enter the queue; until
        // then it still counts as pending
        int again = 0;
        unsigned at = 0;
        if (lane == 0) {
            if (atomicCAS(&G.state[t], WL_RUNNING, WL_IDLE) != WL_RUNNING) {
                atomicExch(&G.state[t], WL_RUNNING);  // a neighbour grew meanwhile: once more
                again = 1;
            }
            const int n = __popc(qm), less = again ? 0 : drop;
            if (n || less) at = (unsigned)(atomicAdd(&G.sh->tp, ((u64)n << 32) + (u64)(long long)(n - less)) >> 32);
        }
        at = __shfl_sync(FULLG, at, 0);
        if (queue) grow_put(G, at + __popc(qm & ((1u << lane) - 1u)), (unsigned)(t + off));
        if (!__shfl_sync(FULLG, again, 0)) return;
        __threadfence();
        if (__any_sync(FULLG, *(const volatile int*)&G.sh->err != 0)) return;
    }
}

constexpr int GROW_WARPS = 4, GROW_CTAS = 2;  // per CTA, per SM (grow_grid)

__global__ void __launch_bounds__(GROW_WARPS * 32, GROW_CTAS) k_grow(const __grid_constant__ GrowLaunch G) {
    after_previous();
    const int lane = threadIdx.x & 31;
    int groups = 0;
    for (;; groups++) {  // the tiles of a group that hold a marker pixel
        int g = 0;
        if (lane == 0) g = atomicAdd(&G.sh->next, 1);
        g = __shfl_sync(FULLG, g, 0);
        const int t0 = g * G.group;
        if (t0 >= G.n_rt) break;
        unsigned todo = __ballot_sync(FULLG, lane < G.group && t0 + lane < G.n_rt && G.any[t0 + lane]);
        for (; todo; todo &= todo - 1) {
            const int t = t0 + __ffs(todo) - 1;
            int mine = 0;  // a tile that a neighbour has queued is left to the queue
            if (lane == 0) mine = atomicCAS(&G.state[t], WL_IDLE, WL_RUNNING) == WL_IDLE;
            if (!__shfl_sync(FULLG, mine, 0)) continue;
            __threadfence();
            __syncwarp();
            grow_tile(G, t, 0, lane);
        }
    }
    __syncwarp();
    if (lane == 0 && groups) atomicAdd(&G.sh->tp, (u64)(-(long long)groups));  // pending
    for (;;) {
        int t = 0;
        if (lane == 0) {
            t = grow_pop(G);
            if (t >= 0) atomicExch(&G.state[t], WL_RUNNING);
        }
        t = __shfl_sync(FULLG, t, 0);
        if (t < 0) break;
        __threadfence();
        __syncwarp();
        grow_tile(G, t, 1, lane);
        __syncwarp();
    }
}

// ---- bits to bytes: one warp per work tile ---------------------------------------------
// Rows of 16-byte aligned planes are written 8 at a time, 16 pixels per lane;
// other planes one row at a time, a byte per lane and half row.
__device__ __forceinline__ uint32_t nibble_bytes(unsigned b) { return (b * 0x00204081u) & 0x01010101u; }

__global__ void __launch_bounds__(256) k_grow_out(const __grid_constant__ GrowLaunch G) {
    after_previous();
    const int t = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (t >= G.n_rt) return;
    const CannyDesc& d = G.tab[G.tab.find(t, &CannyDesc::rt_base)];
    const int W = d.W, H = d.H, rx = (W + RT - 1) / RT, k = t - d.rt_base, ty = k / rx, tx = k - ty * rx;
    const u64* src = G.marker + (size_t)t * RT;
    const int x0 = tx * RT, y0 = ty * RT, nr = min(RT, H - y0);
    uint8_t* dst = d.edges + (size_t)y0 * W + x0;
    if ((W & 15) == 0 && (reinterpret_cast<uintptr_t>(d.edges) & 15) == 0) {
        const int q = lane & 3;
        if (x0 + 16 * q >= W) return;
#pragma unroll
        for (int i = 0; i < RT / 8; i++) {
            const int r = 8 * i + (lane >> 2);
            if (r >= nr) break;
            const unsigned b = reinterpret_cast<const uint16_t*>(src + r)[q];
            *reinterpret_cast<uint4*>(dst + (size_t)r * W + 16 * q) =
                make_uint4(nibble_bytes(b & 15u), nibble_bytes((b >> 4) & 15u), nibble_bytes((b >> 8) & 15u), nibble_bytes(b >> 12));
        }
    } else {
        const bool p0 = x0 + lane < W, p1 = x0 + 32 + lane < W;
        for (int r = 0; r < nr; r++) {
            const u64 w = src[r];
            if (p0) dst[(size_t)r * W + lane] = (uint8_t)((w >> lane) & 1u);
            if (p1) dst[(size_t)r * W + 32 + lane] = (uint8_t)((w >> (32 + lane)) & 1u);
        }
    }
}

// descriptors beyond those that fit in the launch parameters reach the
// device through the parameters of small launches (no host buffer has to
// outlive the call)
struct CannyDescPack {
    CannyDesc d[CannyTab::NEAR];
    int n, first;
};
__global__ void k_set_canny_desc(CannyDesc* dst, const __grid_constant__ CannyDescPack p) {
    if (threadIdx.x < p.n) dst[p.first + threadIdx.x] = p.d[threadIdx.x];
}

CannyTab make_canny_tab(const std::vector<CannyDesc>& v, CannyDesc* far, cudaStream_t s) {
    CannyTab tab;
    tab.n = (int)v.size();
    tab.far = far;
    if (tab.n <= CannyTab::NEAR) {
        for (int i = 0; i < tab.n; i++) tab.near[i] = v[i];
        return tab;
    }
    for (int i = 0; i < tab.n; i += CannyTab::NEAR) {
        CannyDescPack pk;
        pk.first = i;
        pk.n = std::min((int)CannyTab::NEAR, tab.n - i);
        for (int k = 0; k < pk.n; k++) pk.d[k] = v[i + k];
        k_set_canny_desc<<<1, 32, 0, s>>>(far, pk);
    }
    return tab;
}

// Tiles per draw: the draws of a large launch meet at one counter, while in a
// small one a worker should not hold several tiles (one 512^2 edge plane: 11 us
// with one tile per draw, 19 us with four; one 4096^2 red blood cell plane 28,
// 27 and 29 us with one, two and four; eight 4096^2 edge planes 192, 184, 176).
int grow_group(int n_rt) { return n_rt < 2048 ? 1 : n_rt < 16384 ? 2 : 4; }

// Two CTAs (8 warps) per SM: more workers draw from the counters and wait on
// the queue without being needed (rbc 28 us; with 16, 24 and 32 warps per SM
// 36, 45 and 49; the edge planes 176, 174, 187, 202).
int grow_grid(int device) {
    int sms = 0, per = 0;
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_grow, GROW_WARPS * 32, 0);
    return sms * std::min(std::max(per, 1), GROW_CTAS);
}

void launch_grow(const GrowLaunch& G, int grid_cap, cudaStream_t s, Profiler* pf) {
    pf->begin("grow", s);
    launch_behind(pf->overlap(), k_grow, std::min((G.n_rt + GROW_WARPS - 1) / GROW_WARPS, grid_cap), GROW_WARPS * 32, 0, s, G);
    pf->end("grow", s);
    pf->begin("grow_out", s);
    launch_behind(pf->overlap(), k_grow_out, (G.n_rt + 7) / 8, 256, 0, s, G);
    pf->end("grow_out", s);
}

}  // namespace nucseg
