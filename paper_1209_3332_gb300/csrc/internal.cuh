// Internal declarations shared by the CUDA translation units of libpipe.
// Nothing here is part of the C ABI (include/pipe.h).
#pragma once
#include <type_traits>
#include <cuda_runtime.h>
#include <stdint.h>
#include <stddef.h>
#include <vector>

namespace nucseg {

// ---- geometry ---------------------------------------------------------------
constexpr int RT = 64;            // reconstruction work tile: RT x RT pixels, one warp
constexpr int RECON_MIN_BLOCKS = 16;  // resident reconstruction workers (one-warp CTAs) per SM the register budget must allow
constexpr int CB = 32;            // labelling block: CB x CB pixels (one bitmap word per row)
constexpr int CCL_WARPS = 4;      // labelling blocks (one per warp) per CTA
constexpr int RL_CAP = 512;       // root-list slots per labelling block
constexpr int NFEAT = 15;
constexpr int MAX_SIDE = 16384;   // largest width and height of an image
constexpr int MAX_TILES = 4096;   // tiles of a batched call
constexpr int MORPH_RMAX = 15;   // largest disk radius of the opening (chords of up to 31 pixels)

// worklist tile states
constexpr int WL_IDLE = 0, WL_QUEUED = 1, WL_RUNNING = 2, WL_DIRTY = 3;

// device status codes (same values as pipe_status)
constexpr int ST_TIMEOUT = 5, ST_OVERFLOW = 6;

// One image of a launch: pointers into caller buffers and the pipe's arena.
struct TileDev {
    int W, H;
    size_t pitch;                 // RGB row pitch in bytes
    const uint8_t* rgb;
    uint8_t* hem8;                // H*W
    uint8_t* R;                   // reconstruction (workspace), rows of rp bytes
    int rp;                       // W rounded up to 16: R's rows start on 16-byte boundaries
    int32_t* labels;              // H*W
    int32_t* edt;                 // H*W (may be null: EDT skipped)
    int32_t* n_objects;           // [1]
    float* feats;                 // [feats_cap][15] (batched form)
    int feats_cap;
    uint32_t* fgbits;             // bitmaps, block-major: CB words (rows) per labelling block
    uint32_t* filledbits;
    uint32_t* rootbits;           // kept component roots, row-major: H rows of wpr words
    int32_t* wordprefix;          // exclusive popcount prefix of rootbits words
    int32_t* chunksum;            // per scan chunk
    int32_t* P;                   // union-find parents (sparse, H*W)
    int32_t* A;                   // per-root payload (sparse, H*W)
    int32_t* border;              // per labelling block: 4*CB local roots
    int32_t* rootlist;            // local roots, RL_CAP per labelling block
    int32_t* blkroots;            // local roots recorded per labelling block
    int4* bbox;                   // per object: xmin, ymin, xmax, ymax
    uint32_t* colbits;            // per 32-row chunk and column: kept bits of the 32 rows
    int wpr;                      // bitmap words per row = ceil(W/32)
    int rtx, rty, rt_base;        // reconstruction tiles and global base id
    int cbx, cby, cb_base;        // labelling blocks and global base id
    int nchunks, chunk_base;      // scan chunks (of SCAN_CHUNK words)
    int row_base;                 // EDT rows base
    int px_base;                  // deconvolution work items base
    int obj_base;                 // first object item of this tile (batched features)
    int cls[8], cls_pos[8];       // reconstruction queue order: work tiles per class, and placed so far
};

constexpr int SCAN_THREADS = 1024;           // threads of a scan CTA, four bitmap words each
constexpr int SCAN_CHUNK = 4 * SCAN_THREADS;  // bitmap words per scan chunk
constexpr int LAUNCH_TAB = 64;    // tiles whose block bases travel in the launch parameters

// Shared state of one launch sequence (device memory).
struct Shared {
    unsigned long long tp;              // reconstruction worklist: tail << 32 | pending
    alignas(256) int head;              // worklist head
    alignas(256) int next_obj;          // the batched feature pass draws its objects from this counter
    alignas(256) int nobj;              // object items of a batched feature pass
    int err;                            // first error of this launch: ends its waits
    int processed;                      // tile processings (diagnostic)
};

struct Launch {
    TileDev* tiles;        // device array [ntiles]
    int ntiles;
    unsigned long long* wl_slots;  // [n_rt] queue ring: sequence << 32 | item
    int* wl_state;         // [n_rt] per-tile state
    int* rt_src;           // [n_rt] work tiles holding a strong marker (queued first)
    Shared* sh;
    int* tile_status;      // [ntiles]
    int* status;           // the pipe's status word (set_status); null for served groups, whose results carry theirs
    // totals (host-computed) for grid sizing
    int n_rt, n_cb, n_chunks, n_rows, n_px;
    int early;             // each kernel is launched before the one ahead of it is complete (launch_behind)
    long long wait_budget;
    int h, thr, amin, amax;
    // first labelling block of each of the first LAUNCH_TAB tiles (kernel
    // parameters live in the constant bank, so a search over them is cheap)
    int cb_first[LAUNCH_TAB];
};

// ---- small device helpers ----------------------------------------------------
__device__ __forceinline__ int find_tile(const TileDev* t, int n, int gid, int TileDev::*base) {
    int lo = 0, hi = n - 1;
    while (lo < hi) {
        int mid = (lo + hi + 1) >> 1;
        if (t[mid].*base <= gid) lo = mid; else hi = mid - 1;
    }
    return lo;
}

// The pipe's status word keeps the first error of any call until the host reads
// it: no launch clears it.
__device__ __forceinline__ void set_status(int* status, int code) {
    if (status) atomicCAS(status, 0, code);
}
// A wait of a launch whose error word is err ran out.
__device__ __forceinline__ void wait_over(int* err, int* status) {
    atomicCAS(err, 0, ST_TIMEOUT);
    set_status(status, ST_TIMEOUT);
}

// 4 N consecutive bytes from p on, any alignment, from N + 1 aligned words; all
// of [p - 3, p + 4 N + 4) must be readable.
template <int N>
__device__ __forceinline__ void load_unaligned(const uint8_t* p, uint32_t (&out)[N]) {
    const uintptr_t a = reinterpret_cast<uintptr_t>(p);
    const uint32_t* w = reinterpret_cast<const uint32_t*>(a & ~(uintptr_t)3);
    const uint32_t sel = 0x3210u + 0x1111u * (uint32_t)(a & 3);
    uint32_t v[N + 1];
#pragma unroll
    for (int i = 0; i <= N; i++) v[i] = __ldg(w + i);
#pragma unroll
    for (int i = 0; i < N; i++) out[i] = __byte_perm(v[i], v[i + 1], sel);
}

// zeroes the pixels from n on (n < 16)
__device__ __forceinline__ uint4 clip_px16(uint4 v, int n) {
    uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
    for (int i = 0; i < 4; i++) w[i] &= n >= 4 * i + 4 ? 0xffffffffu : n <= 4 * i ? 0u : (1u << (8 * (n - 4 * i))) - 1u;
    return make_uint4(w[0], w[1], w[2], w[3]);
}

// Pixels x .. x + 15 of row y of a W x H byte plane, 0 beyond the row's end: a
// 16-byte load where that is aligned, the aligned words that hold them where
// these lie within the plane, bytes otherwise.  x < W, y < H.
__device__ __forceinline__ uint4 load_px16(const uint8_t* __restrict__ plane, int W, int H, int x, int y) {
    const uint8_t* p = plane + (size_t)y * W + x;
    const int n = W - x;  // valid pixels
    if (n >= 16 && (reinterpret_cast<uintptr_t>(p) & 15) == 0) return __ldg(reinterpret_cast<const uint4*>(p));
    uint32_t w[4] = {0, 0, 0, 0};
    const size_t left = (size_t)(H - y) * W - x;  // bytes of the plane from p on
    if (left >= 20 && p >= plane + 3) {
        load_unaligned<4>(p, w);
        if (n < 16) return clip_px16(make_uint4(w[0], w[1], w[2], w[3]), n);
    } else {
#pragma unroll
        for (int k = 0; k < 16; k++)
            if (k < n) w[k >> 2] |= (uint32_t)__ldg(p + k) << (8 * (k & 3));
    }
    return make_uint4(w[0], w[1], w[2], w[3]);
}
// Object boxes from one row segment of FB_SEG labels, one warp: each lane
// reads 4 labels at a time; the lanes holding the same label (one
// __match_any_sync group per label value) combine their column range and
// one lane updates the box with atomics.  Labels outside 1..K are ignored.
constexpr int FB_STEPS = 8;
constexpr int FB_SEG = 32 * 4 * FB_STEPS;
__device__ __forceinline__ void bbox_segment(const int32_t* __restrict__ row, int W, int K, int y, int xs,
                                             int4* bbox, int lane) {
    const unsigned full = 0xffffffffu;
    const bool vec = (W & 3) == 0;
    for (int step = 0; step < FB_STEPS; step++) {
        const int x0 = xs + (step * 32 + lane) * 4;
        int v[4] = {0, 0, 0, 0};
        if (vec && x0 + 3 < W) {
            int4 q = __ldcs(reinterpret_cast<const int4*>(row + x0));
            v[0] = q.x; v[1] = q.y; v[2] = q.z; v[3] = q.w;
        } else {
            for (int k = 0; k < 4; k++) v[k] = x0 + k < W ? __ldcs(row + x0 + k) : 0;
        }
        if (__ballot_sync(full, (v[0] | v[1] | v[2] | v[3]) != 0) == 0) continue;
#pragma unroll
        for (int k = 0; k < 4; k++) {
            int lab = (v[k] >= 1 && v[k] <= K) ? v[k] : 0;
            // the other pixels of this lane with the same label join this update
            int mn = 0x7fffffff, mx = -1;
            if (lab) {
                for (int j = k; j < 4; j++)
                    if (v[j] == lab) { mn = min(mn, x0 + j); mx = max(mx, x0 + j); v[j] = 0; }
            }
            unsigned grp = __match_any_sync(full, lab);
            if (lab) {
                int gmn = __reduce_min_sync(grp, (unsigned)mn), gmx = __reduce_max_sync(grp, (unsigned)mx);
                if (lane == __ffs(grp) - 1) {
                    int4* b = bbox + (lab - 1);
                    atomicMin(&b->x, gmn);
                    atomicMax(&b->z, gmx);
                    atomicMin(&b->y, y);
                    atomicMax(&b->w, y);
                }
            }
        }
    }
}

// ---- launchers (one per translation unit) -----------------------------------
// Profiler hook: every kernel launch is bracketed by begin/end with its name;
// the pipe counts launches and, when enabled, records CUDA events.
struct Profiler {
    virtual void begin(const char* name, cudaStream_t s) = 0;
    virtual void end(const char* name, cudaStream_t s) = 0;
    virtual bool overlap() const { return true; }  // whether kernels may be launched early
    virtual ~Profiler() {}
};

// A kernel launched right behind another one of the same stream.  The device
// prepares it while that one still runs, and its blocks become resident as soon
// as all blocks of that one have started and left room; its first statement is
// after_previous(), which waits until that one is complete and its writes can
// be seen, so that no access comes before it (what such a kernel reads through
// __ldg lies behind a pointer that it loads from a descriptor first).  As every
// kernel waits so before the next one may be prepared, completion is transitive.
// The plain form launches its kernels so: 512^2, 233 -> 195 us; 1024^2, 250 -> 212;
// 4096^2, 490 -> 458; 8192^2, 1054 -> 1029 us.  In a graph it gains nothing (1, 4 and
// 16 tiles of 4096^2 per batch: 486, 1072 and 3515 us without, 486, 1087 and 3550
// with), so that the batched and the served forms do without (Launch::early).
template <typename... P>
inline void launch_behind(bool early, void (*kernel)(P...), unsigned grid, unsigned block, size_t smem, cudaStream_t s,
                          typename std::common_type<P>::type... args) {
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t c{};
    c.gridDim = grid;
    c.blockDim = block;
    c.dynamicSmemBytes = smem;
    c.stream = s;
    c.attrs = &at;
    c.numAttrs = early ? 1 : 0;
    cudaLaunchKernelEx(&c, kernel, args...);
}
// The first statement of a kernel that is launched so, or that another one so
// launched follows (which may then be prepared from here on).
__device__ __forceinline__ void after_previous() {
    cudaGridDependencySynchronize();
    cudaTriggerProgrammaticLaunchCompletion();
}

void upload_deconv_tables(const int32_t* lut256, const int32_t* wq3);
void launch_deconv(const Launch& L, cudaStream_t s, Profiler* pf);
void recon_grid(int device, int* warps, int* teams);
// warps: resident one-warp workers to use, of warps_cap; launches with few work
// tiles per worker use teams of four warps instead, the same share of teams_cap
void launch_recon(const Launch& L, int warps, int warps_cap, int teams_cap, cudaStream_t s, Profiler* pf);
void launch_label(const Launch& L, int want_bbox, int sms, cudaStream_t s, Profiler* pf);
size_t edt_rows_smem(int RB, int Wmax);
void launch_edt(const Launch& L, int RB, int Wmax, cudaStream_t s, Profiler* pf);
// The opening (1 <= r <= MORPH_RMAX in two passes through tmp, morph_scratch bytes).
inline int morph_pitch(int W) { return (W + 15) & ~15; }  // rows of its scratch planes
// The scratch of any plane of up to `px` pixels, whatever its shape and alignment, so
// that a call allocates only where it has more pixels than every one before: two
// planes of padded rows, which are at most W + W / 16 bytes from W = 240 on, and 240
// bytes below.
inline size_t morph_scratch(size_t px) {
    const size_t narrow = (size_t)240 * MAX_SIDE, plane = px + px / 16 > narrow ? px + px / 16 : narrow;
    return 2 * ((plane + 255) & ~(size_t)255);
}
void launch_morph_open(const uint8_t* src, uint8_t* dst, uint8_t* tmp, int W, int H, int r, int sms, cudaStream_t s,
                       Profiler* pf);
void launch_features_plain(const uint8_t* hem8, const int32_t* labels, int W, int H, int K, float* feats,
                           int4* bbox, int sms, cudaStream_t s, Profiler* pf);
void launch_features_batched(const Launch& L, int grid, int sms, cudaStream_t s, Profiler* pf);
// One tile of a Canny launch (plain: one tile; batched: many), or of another
// growth of a binary marker through a binary mask.
struct CannyDesc {
    const uint8_t* img;      // W x H plane
    const int32_t* labels;   // W x H labels (may be null when K == 0)
    uint8_t* edges;          // the grown marker as bytes (0/1)
    int32_t* counts;         // K edge counts
    int W, H, K;
    int bx;                  // 32-pixel blocks per row
    int blk_base;            // first 32x32 block of this tile in the counts launch
    int nms_base;            // first warp of this tile in the suppression launch
    int rt_base;             // first work tile of this tile
};
// The descriptors of a launch: up to NEAR travel in the launch parameters,
// more are in device memory.
struct CannyTab {
    static constexpr int NEAR = 8;
    int n;
    const CannyDesc* far;
    CannyDesc near[NEAR];
    __device__ __forceinline__ const CannyDesc& operator[](int i) const { return n <= NEAR ? near[i] : far[i]; }
    // the tile of launch item b, by the tiles' first items
    __device__ __forceinline__ int find(int b, int CannyDesc::*base) const {
        int lo = 0, hi = n - 1;
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if ((*this)[mid].*base <= b) lo = mid; else hi = mid - 1;
        }
        return lo;
    }
};
CannyTab make_canny_tab(const std::vector<CannyDesc>& v, CannyDesc* far, cudaStream_t s);
// Growth of a marker through a mask (k_grow.cu): bit planes of 64 64-bit words
// per work tile, and the state of its queue.
struct GrowShared {  // the words that every worker's atomics meet at, in lines of their own
    unsigned long long tp;          // tail << 32 | groups not finished and tiles queued or running
    int err;                        // first error of this launch: ends its waits
    alignas(256) int head;          // queue head
    alignas(256) int next;          // next group of tiles
};
struct GrowLaunch {
    CannyTab tab;
    unsigned long long *mask, *marker;  // the marker grows in place
    unsigned long long* slots;          // [n_rt], zeroed before the launches
    int* state;                         // [n_rt], zeroed
    uint8_t* any;                       // [n_rt] the work tile holds a marker pixel
    GrowShared* sh;
    int* status;                        // the pipe's status word
    int n_rt;
    int group;                          // work tiles drawn at a time at the start, 1 to 32
    long long wait_budget;
};
// by one thread of the kernel that writes the planes
__device__ __forceinline__ void grow_reset(const GrowLaunch& G) {
    G.sh->tp = (unsigned long long)((G.n_rt + G.group - 1) / G.group);
    G.sh->head = G.sh->err = G.sh->next = 0;
}
int grow_grid(int device);
int grow_group(int n_rt);  // GrowLaunch::group for a launch of n_rt work tiles
// grows the marker and writes it to every tile's edges as bytes
void launch_grow(const GrowLaunch& G, int grid_cap, cudaStream_t s, Profiler* pf);
// Blocks (32 x 32 pixels) and suppression warps of a tile in the Canny launches.
int canny_blocks(int W, int H);
int canny_nms_warps(int W, int H);
// Zeroes the counts; writes the strong pixels into the marker and the
// candidates into the mask.
void launch_canny_nms(const GrowLaunch& G, int warps, int low, int high, cudaStream_t s, Profiler* pf);
// Edge counts of every tile: each edge pixel adds one to every object 1..K
// with a pixel within its disk of radius r (the disk dilation of the object).
void launch_canny_counts(const GrowLaunch& G, int blocks, int r, cudaStream_t s, Profiler* pf);
// One tile of a batched watershed split.
struct WsDesc {
    const int32_t* labels;
    const int32_t* edt;
    int32_t* out;
    int32_t* n_basins;
    long long px_base;    // first pixel of this tile in the scratch planes
    int W, H, K;
    int obj_base;         // first object item of this tile
    int seg_base;         // first box row segment of this tile
};
// descs: host copy; d_descs: device array of the same length; cnt: an int per
// object (basin counts, then their exclusive prefix); next: WS_COUNTERS ints and
// an int per object (draw counters and lists, set up by the launcher); status: a
// device int; side: a second stream for the larger boxes (fork and join through
// the two events)
constexpr int WS_COUNTERS = 5;
void launch_watershed_batch(const std::vector<WsDesc>& descs, WsDesc* d_descs, int h, int4* bbox, int* cnt,
                            int* next, void* scratch, size_t scratch_px, int* status, int sms, cudaStream_t s,
                            cudaStream_t side, cudaEvent_t fork, cudaEvent_t join, Profiler* pf);
// RBC detection planes: d = R - max(G, B); marker = d >= t_hi, mask = d >= t_lo.
void launch_rbc_planes(const GrowLaunch& G, const uint8_t* rgb, size_t pitch, int t_lo, int t_hi, cudaStream_t s,
                       Profiler* pf);
void launch_unpack_bits(const uint32_t* bits, int W, int H, int cbx, uint8_t* out, cudaStream_t s,
                        Profiler* pf);

}  // namespace nucseg
