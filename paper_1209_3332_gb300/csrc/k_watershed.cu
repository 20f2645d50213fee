// Watershed split of labelled objects on the distance transform (Table I:
// "Pre-Watershed" -- the distance transform and the markers -- and
// "Watershed").  The paper names the operations only; the definition built
// here, for each object k of the label plane:
//   d  = min(255, floor(sqrt(edt))) on the object's pixels;
//   R  = reconstruction by dilation, 8-connected, of max(d - h, 0) under d
//        (the h-maxima of d);
//   markers = maximal 8-connected plateaus of equal R with no 8-neighbour in
//        the object of larger R, each named by its first pixel in raster order;
//   flooding in synchronous waves: with F the unnamed object pixels that have
//        a named 8-neighbour and L = max d over F, every pixel of F with
//        d >= L takes, in one wave, the name of its named neighbour of largest
//        edt (then smallest name); waves repeat at L while any pixel is named,
//        then L is taken again from the new F;
//   out = basins numbered object by object in label order, within an object
//        by the raster order of each basin's first pixel; 0 off the objects.
//
// Objects are independent: two labels are never 8-adjacent (they would be
// one component), and d = 0 off the object keeps R, the plateaus and the
// flooding inside it.  So a team of threads owns one object: its bounding box
// plus a 1-px margin is staged in shared memory (d, R and later flags in one
// 16-bit word per pixel, edt, and one 32-bit work word), and every step runs
// there with a barrier between passes:
//   1. relaxation passes, alternately in raster and anti-raster order, update
//      R in place until a pass changes nothing (monotone updates from below,
//      so the fixed point reached is the reconstruction);
//   2. markers: what a few passes cannot rule out is joined by union-find over
//      the work words (roots are the smallest index, i.e. the first pixel);
//   3. flooding: the work word holds (wave stamp, name); a pass names the
//      pixels of F at level L with stamp = wave, and only neighbours with an
//      older stamp count, so a pass is exactly one synchronous wave.  F itself
//      is kept as a list (double-buffered, pixels entered once through an
//      atomic flag), so a wave costs the frontier, not the box;
//   4. each basin's first pixel by atomicMin on its root's word, a ballot
//      prefix over the box in raster order for the ranks.
// Boxes up to WS_STAGE pixels (with margin) are split by one warp; larger ones
// by the four warps of a CTA, with a stage of WS_MIDDLE pixels or a larger one,
// launched on a side stream so that the few large objects overlap the many
// small ones; boxes beyond that stage run the same steps (with a full-box scan
// per wave) on image-sized scratch planes in global memory.  A scan of the
// per-object basin counts and a pass adding each object's offset finish the
// numbering.
// Bound: the latency of an object's chain of passes over shared memory; the
// zeros of the split plane, the boxes and the offsets (about 250 us of the 596
// for 8 tiles of 4096^2) move the labels and the plane once each.
#include <algorithm>

#include "internal.cuh"

namespace nucseg {

constexpr int WS_WARPS = 4;      // warps per CTA: one object each (small boxes) or one together
constexpr int WS_STAGE = 384;    // staged box (with margin) capacity per warp of the small-box kernel, pixels
// Staged box capacity of a CTA with the small stage.  The large stage leaves room
// for two CTAs per SM and waits for that room behind the small boxes, so it is
// kept for the rare boxes beyond this (8 tiles of 4096^2, and 4 with chains of
// nuclei: 691 and 917 us at 1024, 592 and 943 at 1536, 609 and 946 at 2048, 596
// and 812 at 3072).
constexpr int WS_MIDDLE = 3072;
constexpr int WS_PX_BYTES = 14;  // stage bytes per pixel: e 4, w 4, dr 2, two frontier lists 2 + 2
constexpr int WS_LARGE_SMEM = 96 * 1024;  // dynamic stage of a CTA with the large stage
constexpr int WS_OUT_PASSES = 8;  // passes that spread "on no marker" before the union-find
constexpr unsigned WFULL = 0xffffffffu;

__device__ __forceinline__ int ws_isqrt(int v) {  // floor(sqrt(v)), exact
    if (v <= 0) return 0;
    int r = (int)sqrtf((float)v);
    while ((long long)r * r > v) r--;
    while ((long long)(r + 1) * (r + 1) <= v) r++;
    return r;
}

// The threads that split one object: a warp, or the NW warps of a CTA.
template <int NW>
struct Team {
    static constexpr int N = 32 * NW;
    int t;    // thread of the team
    int* sh;  // NW > 1: shared, the lengths of the two frontier lists, a result, and a word per warp
    __device__ __forceinline__ int lane() const { return t & 31; }
    __device__ __forceinline__ void sync() const {
        if constexpr (NW == 1) __syncwarp(); else __syncthreads();
    }
    // sync, and whether p held for some thread
    __device__ __forceinline__ bool any(bool p) const {
        if constexpr (NW == 1) { __syncwarp(); return __any_sync(WFULL, p); }
        else return __syncthreads_or(p);
    }
    // the largest v >= 0
    __device__ __forceinline__ int max_of(int v) const {
        v = (int)__reduce_max_sync(WFULL, (unsigned)v);
        if constexpr (NW > 1) {
            __syncthreads();
            if (lane() == 0) sh[3 + (t >> 5)] = v;
            __syncthreads();
#pragma unroll
            for (int i = 0; i < NW; i++) v = max(v, sh[3 + i]);
        }
        return v;
    }
};

// Flat positions f = f0, f0 + STEP, ... of a row-major box of width ww, with
// (y, x) of f kept without a division per step.
template <int STEP>
struct WalkBy {
    int f, y, x, qy, qx, ww;
    __device__ __forceinline__ WalkBy(int f0, int ww_) : f(f0), ww(ww_) {
        y = f0 / ww;
        x = f0 - y * ww;
        qy = STEP / ww;
        qx = STEP - qy * ww;
    }
    __device__ __forceinline__ void next() {
        f += STEP;
        x += qx;
        y += qy;
        if (x >= ww) { x -= ww; y++; }
    }
    __device__ __forceinline__ void prev() {
        f -= STEP;
        x -= qx;
        y -= qy;
        if (x < 0) { x += ww; y--; }
    }
};

// Shared-memory box: the object's box plus a 1-px margin, row stride ww.
// Pixels off the object (margin, background, other objects) are staged with
// dr = 0 and w = all ones, so neighbour reads need no bounds or label tests.
struct SBox {
    using Wt = uint32_t;
    static constexpr bool GLOBAL = false;
    static constexpr int SH = 16;               // name bits (indices < 2^16)
    volatile uint16_t* dr;                      // d | R << 8; later bit 8 marker, 9 first pixel, 10 in F once
    volatile int32_t* e;                        // edt
    volatile Wt* w;                             // work word
    volatile uint16_t *la, *lb;                 // frontier lists, n entries each
    int ww, n;                                  // walk width, flat size
    int gx0, gy0, W;                            // image position of flat (0, 0)
    template <class WK>
    __device__ __forceinline__ int stor(const WK& it) const { return it.f; }
    __device__ __forceinline__ bool in(int s) const { return (dr[s] & 0xFF) != 0; }
    template <class WK>
    __device__ __forceinline__ int nb(const WK&, int s, int dy, int dx) const { return s + dy * ww + dx; }
    template <class WK>
    __device__ __forceinline__ size_t gidx(const WK& it) const {
        return (size_t)(gy0 + it.y) * W + (gx0 + it.x);
    }
};

// Global box: the object's box (no margin) inside image-sized scratch planes
// (row stride W); membership from the label plane, bounds tested.
struct GBox {
    using Wt = unsigned long long;
    static constexpr bool GLOBAL = true;
    static constexpr int SH = 32;
    volatile uint16_t* dr;
    const int32_t* e;
    volatile Wt* w;
    const int32_t* lab;
    int k;
    int ww, bh, n;
    int gx0, gy0, W;
    template <class WK>
    __device__ __forceinline__ int stor(const WK& it) const { return it.y * W + it.x; }
    __device__ __forceinline__ bool in(int s) const { return lab[s] == k; }
    template <class WK>
    __device__ __forceinline__ int nb(const WK& it, int s, int dy, int dx) const {
        return ((unsigned)(it.y + dy) < (unsigned)bh && (unsigned)(it.x + dx) < (unsigned)ww) ? s + dy * W + dx
                                                                                              : -1;
    }
    template <class WK>
    __device__ __forceinline__ size_t gidx(const WK& it) const {
        return (size_t)(gy0 + it.y) * W + (gx0 + it.x);
    }
};

template <class B>
__device__ __forceinline__ bool ws_nb_in(const B& b, int q) {
    if constexpr (B::GLOBAL) return q >= 0 && b.in(q);
    else return b.in(q);
}

// neighbour j (0..7, raster order) of pixel s of a shared-memory box
__device__ __forceinline__ int ws_nb8(const SBox& b, int s, int j) {
    const int k = j < 4 ? j : j + 1;
    return s + (k / 3 - 1) * b.ww + (k % 3 - 1);
}

template <class B>
__device__ __forceinline__ int ws_find(const B& b, int x) {
    // path halving: a non-root is pointed at its grandparent (an ancestor,
    // whatever concurrent unions do, so the forest stays valid); without it
    // the walks over a plateau of a thousand pixels grow with its size
    constexpr typename B::Wt IDX = ((typename B::Wt)1 << B::SH) - 1;
    for (;;) {
        const int p = (int)(b.w[x] & IDX);
        if (p == x) return x;
        const int gp = (int)(b.w[p] & IDX);
        if (gp != p) b.w[x] = (typename B::Wt)gp;
        x = gp;
    }
}

// The root of x without shortening links: while other warps replace links by
// roots, a shortcut written late could put an older ancestor over a root.
template <class B>
__device__ __forceinline__ int ws_root(const B& b, int x) {
    constexpr typename B::Wt IDX = ((typename B::Wt)1 << B::SH) - 1;
    for (;;) {
        const int p = (int)(b.w[x] & IDX);
        if (p == x) return x;
        x = p;
    }
}

// Union of the plateaus of a and b; the larger root is linked under the
// smaller, so every root is its set's first pixel.
template <class B>
__device__ __forceinline__ void ws_unite(const B& b, int a, int c) {
    using Wt = typename B::Wt;
    for (;;) {
        a = ws_find(b, a);
        c = ws_find(b, c);
        if (a == c) return;
        if (a < c) { const int t = a; a = c; c = t; }
        const Wt old = atomicCAS((Wt*)(b.w + a), (Wt)a, (Wt)c);
        if (old == (Wt)a) return;
    }
}

// The four steps on one object.  Returns the number of basins (0 on a wave
// count beyond the cap, after setting the status word).
template <class B, int NW>
__device__ int ws_object(const B& b, const Team<NW>& team, int32_t* out, int* status) {
    using Wt = typename B::Wt;
    using Walk = WalkBy<Team<NW>::N>;
    const int t = team.t, lane = team.lane();
    constexpr Wt IDX = ((Wt)1 << B::SH) - 1;
    constexpr Wt FLAG = (Wt)1 << (sizeof(Wt) * 8 - 1);
    constexpr Wt UNNAMED = ~(Wt)0;

    // 1. R: relaxation passes until one changes nothing
    for (int pass = 0;; pass++) {
        bool ch = false;
        auto relax = [&](const Walk& it) {
            const int s = b.stor(it);
            if (!b.in(s)) return;
            const unsigned v = b.dr[s];
            const int d = v & 0xFF, r = v >> 8;
            int m = r;
#pragma unroll
            for (int j = 0; j < 9; j++) {
                if (j == 4) continue;
                const int q = b.nb(it, s, j / 3 - 1, j % 3 - 1);
                if constexpr (B::GLOBAL) {
                    if (!ws_nb_in(b, q)) continue;
                }
                m = max(m, (int)(b.dr[q] >> 8));
            }
            m = min(m, d);
            if (m != r) {
                b.dr[s] = (uint16_t)(d | (m << 8));
                ch = true;
            }
        };
        if ((pass & 1) == 0) {
            for (Walk it(t, b.ww); it.f < b.n; it.next()) relax(it);
        } else {
            const int last = b.n - 1 - t;
            if (last >= 0)
                for (Walk it(last, b.ww); it.f >= 0; it.prev()) relax(it);
        }
        if (!team.any(ch)) break;
    }

    // 2. markers.  Pixels with a higher neighbour are on no marker, and neither
    // are pixels of equal R beside one of those: a few passes of that leave
    // little but the markers themselves.  What is left is joined by union-find
    // (adjacent pixels left over have equal R: of two different ones the lower
    // has a higher neighbour), and a component beside a pixel of equal R that
    // was left out is no marker either (only possible if the passes were cut
    // short, by a plateau longer than they reach).
    constexpr Wt OUT = UNNAMED - 1;  // on no marker
    for (Walk it(t, b.ww); it.f < b.n; it.next()) {
        const int s = b.stor(it);
        if (!b.in(s)) continue;
        const int r = b.dr[s] >> 8;
        bool higher = false;
#pragma unroll
        for (int j = 0; j < 9; j++) {
            if (j == 4) continue;
            const int q = b.nb(it, s, j / 3 - 1, j % 3 - 1);
            if constexpr (B::GLOBAL) {
                if (!ws_nb_in(b, q)) continue;
            }
            higher |= (int)(b.dr[q] >> 8) > r;  // 0 off the object
        }
        b.w[s] = higher ? OUT : (Wt)s;
    }
    team.sync();
    // Whether a pixel left over touches one of equal R that is out.  In shared
    // memory all sixteen words are read at once and then compared (branches
    // between them cost about 2000 cycles per pixel instead of 300).
    auto beside_out = [&](const Walk& it, int s) -> bool {
        const int r = b.dr[s] >> 8;
        bool out = false;
        if constexpr (B::GLOBAL) {
#pragma unroll
            for (int j = 0; j < 9; j++) {
                if (j == 4) continue;
                const int q = b.nb(it, s, j / 3 - 1, j % 3 - 1);
                if (!ws_nb_in(b, q)) continue;
                out |= (int)(b.dr[q] >> 8) == r && b.w[q] == OUT;
            }
        } else {
            unsigned dq[8];
            Wt wq[8];
#pragma unroll
            for (int j = 0; j < 8; j++) {
                const int q = ws_nb8(b, s, j);
                dq[j] = b.dr[q];
                wq[j] = b.w[q];
            }
#pragma unroll
            for (int j = 0; j < 8; j++) out |= ((int)(dq[j] >> 8) == r) & (wq[j] == OUT);
        }
        return out;
    };
    bool settled = false;
    for (int pass = 0; pass < WS_OUT_PASSES && !settled; pass++) {
        bool ch = false;
        for (Walk it(t, b.ww); it.f < b.n; it.next()) {
            const int s = b.stor(it);
            if (!b.in(s) || b.w[s] == OUT || !beside_out(it, s)) continue;
            b.w[s] = OUT;
            ch = true;
        }
        settled = !team.any(ch);
    }
    for (Walk it(t, b.ww); it.f < b.n; it.next()) {
        const int s = b.stor(it);
        if (!b.in(s) || b.w[s] == OUT) continue;
        unsigned with = 0;  // the neighbours before s in raster order to join
#pragma unroll
        for (int j = 0; j < 4; j++) {
            const int q = b.nb(it, s, j < 3 ? -1 : 0, j < 3 ? j - 1 : -1);
            if constexpr (B::GLOBAL) {
                if (!ws_nb_in(b, q) || b.w[q] == OUT) continue;
                with |= 1u << j;
            } else {
                with |= (unsigned)(b.in(q) & (b.w[q] != OUT)) << j;
            }
        }
        for (; with; with &= with - 1) {
            const int j = __ffs(with) - 1;
            ws_unite(b, s, b.nb(it, s, j < 3 ? -1 : 0, j < 3 ? j - 1 : -1));
        }
    }
    team.sync();
    for (Walk it(t, b.ww); it.f < b.n; it.next()) {
        const int s = b.stor(it);
        if (b.in(s) && b.w[s] != OUT) b.w[s] = (Wt)ws_root(b, s);
    }
    team.sync();
    if (!settled) {
        for (Walk it(t, b.ww); it.f < b.n; it.next()) {
            const int s = b.stor(it);
            if (!b.in(s) || b.w[s] == OUT || !beside_out(it, s)) continue;
            atomicOr((Wt*)(b.w + (int)(b.w[s] & IDX)), FLAG);
        }
        team.sync();
    }
    for (Walk it(t, b.ww); it.f < b.n; it.next()) {  // bit 8 of dr: a marker pixel (R no longer needed)
        const int s = b.stor(it);
        if (!b.in(s)) continue;
        const Wt w = b.w[s];
        const bool mk = w != OUT && !(b.w[(int)(w & IDX)] & FLAG);
        b.dr[s] = (uint16_t)((b.dr[s] & 0xFF) | (mk ? 0x100 : 0));
    }
    team.sync();
    for (Walk it(t, b.ww); it.f < b.n; it.next()) {  // markers: stamp 0, name = root
        const int s = b.stor(it);
        if (!b.in(s)) continue;
        b.w[s] = (b.dr[s] & 0x100) ? (b.w[s] & IDX) : UNNAMED;
    }
    team.sync();

    // 3. flooding in synchronous waves
    {
        const unsigned cap = (unsigned)min((long long)b.n + 300, (long long)IDX - 1);
        if constexpr (B::GLOBAL) {
            // full-box scan per wave (boxes beyond every stage: rare)
            int L = 256;  // above every d: the first pass only measures F
            for (unsigned wave = 1;; wave++) {
                if (wave >= cap) {
                    if (t == 0) set_status(status, ST_OVERFLOW);
                    return 0;
                }
                int named = 0, fmax = -1;
                for (Walk it(t, b.ww); it.f < b.n; it.next()) {
                    const int s = b.stor(it);
                    if (!b.in(s) || b.w[s] != UNNAMED) continue;
                    int be = 0;
                    Wt bn = IDX;
#pragma unroll
                    for (int j = 0; j < 9; j++) {
                        if (j == 4) continue;
                        const int q = b.nb(it, s, j / 3 - 1, j % 3 - 1);
                        if (!ws_nb_in(b, q)) continue;
                        const Wt wq = b.w[q];
                        if ((wq >> B::SH) >= (Wt)wave) continue;  // unnamed, or named in this wave
                        const int eq = b.e[q];
                        const Wt nq = wq & IDX;
                        if (eq > be || (eq == be && nq < bn)) {
                            be = eq;
                            bn = nq;
                        }
                    }
                    if (be > 0) {
                        const int d = b.dr[s] & 0xFF;
                        fmax = max(fmax, d);
                        if (d >= L) {
                            b.w[s] = ((Wt)wave << B::SH) | bn;
                            named++;
                        }
                    }
                }
                const bool some = team.any(named > 0);
                fmax = team.max_of(fmax + 1) - 1;
                if (!some) {
                    if (fmax < 0) break;
                    L = fmax;
                }
            }
        } else {
            // F as a list: entries enter once (bit 10 of dr, set atomically on
            // the 32-bit word holding it; nothing else writes dr meanwhile)
            auto enter = [&](int q) -> bool {
                const uintptr_t a = (uintptr_t)(b.dr + q);
                const unsigned sh = (unsigned)(a & 2) * 8;
                const unsigned old = atomicOr((unsigned*)(a & ~(uintptr_t)3), 0x400u << sh);
                return !((old >> sh) & 0x400u);
            };
            // Puts `self` (if keep) and, if named, the unnamed object pixels around
            // s that are not in F yet into list `to`; the lanes of a warp call it
            // together.  The list's length is in len (a warp alone) or shared.
            int len = 0;
            auto append = [&](bool keep, bool named, int s, volatile uint16_t* to, int which) {
                unsigned open = 0, mine = 0;
                if (named) {
                    Wt wq[8];
                    unsigned dq[8];
#pragma unroll
                    for (int j = 0; j < 8; j++) {
                        const int q = ws_nb8(b, s, j);
                        wq[j] = b.w[q];
                        dq[j] = b.dr[q];
                    }
#pragma unroll
                    for (int j = 0; j < 8; j++)
                        open |= (unsigned)((wq[j] == UNNAMED) & ((dq[j] & 0xFF) != 0) & !(dq[j] & 0x400)) << j;
                }
                for (; open; open &= open - 1) {
                    const int j = __ffs(open) - 1;
                    if (enter(ws_nb8(b, s, j))) mine |= 1u << j;
                }
                const int c = __popc(mine) + (keep ? 1 : 0);
                int at = c;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const int v = __shfl_up_sync(WFULL, at, o);
                    if (lane >= o) at += v;
                }
                const int total = __shfl_sync(WFULL, at, 31);
                int base = len;
                if constexpr (NW > 1) {
                    if (lane == 0) base = atomicAdd(&team.sh[which], total);
                    base = __shfl_sync(WFULL, base, 0);
                } else {
                    len += total;
                }
                at += base - c;
                if (keep) to[at++] = (uint16_t)s;
                for (; mine; mine &= mine - 1) to[at++] = (uint16_t)ws_nb8(b, s, __ffs(mine) - 1);
            };
            // the length of list `which` after all appends; the other one starts empty
            auto length = [&](int which) -> int {
                team.sync();
                if constexpr (NW > 1) {
                    const int m = *(volatile int*)&team.sh[which];
                    if (t == 0) team.sh[1 - which] = 0;  // seen before the next append: a wave's max_of lies between
                    return m;
                } else {
                    const int m = len;
                    len = 0;
                    return m;
                }
            };
            volatile uint16_t* cur = b.la;
            volatile uint16_t* nxt = b.lb;
            int which = 0;
            if constexpr (NW > 1) {
                if (t == 0) team.sh[0] = 0;
                team.sync();
            }
            for (int f0 = t - lane; f0 < b.n; f0 += Team<NW>::N) {  // neighbours of the markers
                const int s = f0 + lane;
                const bool mk = s < b.n && b.w[s] != UNNAMED;
                if (__any_sync(WFULL, mk)) append(false, mk, s, cur, which);
            }
            int m = length(which);
            // every entry has a neighbour named in an earlier wave, so the next L
            // is known before a wave: no wave names nothing
            int L = 256;
            for (unsigned wave = 1; m > 0; wave++) {
                if (wave >= cap) {
                    if (t == 0) set_status(status, ST_OVERFLOW);
                    return 0;
                }
                int fmax = 0;
                for (int i = t; i < m; i += Team<NW>::N) fmax = max(fmax, (int)(b.dr[cur[i]] & 0xFF));
                L = min(L, team.max_of(fmax));
                which = 1 - which;
                for (int i0 = t - lane; i0 < m; i0 += Team<NW>::N) {
                    const int i = i0 + lane;
                    const int s = i < m ? (int)cur[i] : -1;
                    const bool took = s >= 0 && (int)(b.dr[s] & 0xFF) >= L;
                    if (took) {
                        int be = 0;
                        Wt bn = IDX;
                        Wt wq[8];
                        int eq[8];
#pragma unroll
                        for (int j = 0; j < 8; j++) {
                            const int q = ws_nb8(b, s, j);
                            wq[j] = b.w[q];
                            eq[j] = b.e[q];
                        }
#pragma unroll
                        for (int j = 0; j < 8; j++) {
                            const bool old = (wq[j] >> B::SH) < (Wt)wave;  // named in an earlier wave
                            const Wt nq = wq[j] & IDX;
                            if (old & ((eq[j] > be) | ((eq[j] == be) & (nq < bn)))) {
                                be = eq[j];
                                bn = nq;
                            }
                        }
                        b.w[s] = ((Wt)wave << B::SH) | bn;
                    }
                    append(s >= 0 && !took, took, s, nxt, which);
                }
                m = length(which);
                volatile uint16_t* sw = cur;
                cur = nxt;
                nxt = sw;
            }
        }
    }

    // 4. ranks of the basins by first pixel
    for (Walk it(t, b.ww); it.f < b.n; it.next()) {  // roots: first-pixel field to "none"
        const int s = b.stor(it);
        if (b.in(s) && (int)(b.w[s] & IDX) == s) b.w[s] = (IDX << B::SH) | (Wt)s;
    }
    team.sync();
    for (Walk it(t, b.ww); it.f < b.n; it.next()) {
        const int s = b.stor(it);
        if (!b.in(s)) continue;
        const Wt nm = b.w[s] & IDX;
        atomicMin((Wt*)(b.w + (int)nm), ((Wt)s << B::SH) | nm);
    }
    team.sync();
    for (Walk it(t, b.ww); it.f < b.n; it.next()) {  // bit 9 of dr: the first pixel of its basin
        const int s = b.stor(it);
        if (!b.in(s)) continue;
        const int nm = (int)(b.w[s] & IDX);
        if ((int)(b.w[nm] >> B::SH) == s) b.dr[s] = (uint16_t)(b.dr[s] | 0x200);
    }
    team.sync();
    int run = 0;
    if (t < 32) {
        for (int f0 = 0; f0 < b.n; f0 += 32) {  // raster order: rank = first pixels up to this one
            const int f = f0 + lane;
            bool first = false;
            int s = 0;
            if (f < b.n) {
                const Walk it(f, b.ww);
                s = b.stor(it);
                first = b.in(s) && (b.dr[s] & 0x200);
            }
            const unsigned bal = __ballot_sync(WFULL, first);
            if (first) {
                const Wt nm = b.w[s] & IDX;
                const int rank = run + __popc(bal & ((1u << lane) - 1)) + 1;
                b.w[(int)nm] = ((Wt)rank << B::SH) | nm;
            }
            run += __popc(bal);
        }
    }
    team.sync();
    for (Walk it(t, b.ww); it.f < b.n; it.next()) {
        const int s = b.stor(it);
        if (!b.in(s)) continue;
        out[b.gidx(it)] = (int32_t)(b.w[(int)(b.w[s] & IDX)] >> B::SH);
    }
    return run;
}

// Large boxes: the same steps on global scratch planes, kept out of line.
template <int NW>
__device__ __noinline__ int ws_object_global(const int32_t* labels, const int32_t* edt, int W, int k, int4 bx,
                                             int h, uint16_t* gdr, unsigned long long* gw, int32_t* out,
                                             int* status, const Team<NW>& team) {
    using Walk = WalkBy<Team<NW>::N>;
    GBox b;
    const size_t o = (size_t)bx.y * W + bx.x;
    b.dr = gdr + o;
    b.e = edt + o;
    b.w = gw + o;
    b.lab = labels + o;
    b.k = k;
    b.ww = bx.z - bx.x + 1;
    b.bh = bx.w - bx.y + 1;
    b.n = b.ww * b.bh;
    b.gx0 = bx.x;
    b.gy0 = bx.y;
    b.W = W;
    for (Walk it(team.t, b.ww); it.f < b.n; it.next()) {
        const int s = b.stor(it);
        if (!b.in(s)) continue;
        const int d = min(255, ws_isqrt(b.e[s]));
        b.dr[s] = (uint16_t)(d | ((d > h ? d - h : 0) << 8));
    }
    team.sync();
    return ws_object(b, team, out, status);
}

// Stages one object's box plus margin into a shared-memory stage of `cap`
// pixels (e, w, dr and the two frontier lists, laid out back to back) and
// splits it there.
template <int NW>
__device__ __forceinline__ int ws_staged(const int32_t* __restrict__ labels, const int32_t* __restrict__ edt,
                                         int W, int H, int k, int4 bx, int h, char* stage, int cap,
                                         int32_t* out, int* status, const Team<NW>& team) {
    using Walk = WalkBy<Team<NW>::N>;
    const int BW = bx.z - bx.x + 3, BH = bx.w - bx.y + 3;
    SBox b;
    b.e = (int32_t*)stage;
    b.w = (uint32_t*)(stage + 4 * cap);
    b.dr = (uint16_t*)(stage + 8 * cap);
    b.la = (uint16_t*)(stage + 10 * cap);
    b.lb = (uint16_t*)(stage + 12 * cap);
    b.ww = BW;
    b.n = BW * BH;
    b.gx0 = bx.x - 1;
    b.gy0 = bx.y - 1;
    b.W = W;
    for (Walk it(team.t, BW); it.f < b.n; it.next()) {
        const int gy = b.gy0 + it.y, gx = b.gx0 + it.x;
        int ev = 0;
        if ((unsigned)gy < (unsigned)H && (unsigned)gx < (unsigned)W) {
            const size_t g = (size_t)gy * W + gx;
            if (labels[g] == k) ev = edt[g];
        }
        const int d = ev > 0 ? min(255, ws_isqrt(ev)) : 0;
        b.dr[it.f] = (uint16_t)(d | ((d > h ? d - h : 0) << 8));
        b.e[it.f] = ev;
        b.w[it.f] = 0xffffffffu;
    }
    team.sync();
    return ws_object(b, team, out, status);
}

__device__ __forceinline__ int ws_box_px(int4 bx) { return (bx.z - bx.x + 3) * (bx.w - bx.y + 3); }

// The next entry for this team from a launch-wide counter (entries go to
// whichever team is free, so one that drew a slow object takes no more).
template <int NW>
__device__ __forceinline__ int ws_next(int* next, const Team<NW>& team) {
    int v = 0;
    if constexpr (NW == 1) {
        if (team.t == 0) v = atomicAdd(next, 1);
        return __shfl_sync(WFULL, v, 0);
    } else {
        __syncthreads();
        if (team.t == 0) team.sh[2] = atomicAdd(next, 1);
        __syncthreads();
        return *(volatile int*)&team.sh[2];
    }
}

// Sorts the objects before the object kernels.  An absent object (empty box)
// gets count 0.  By its box an object goes to a warp (k_ws_objects), or to a CTA
// with a small or a large stage (k_ws_team), listed from the front and from the
// back of `list`: next[1] and next[4] entries.
// next: large drawn, large listed, small drawn, middle drawn, middle listed
__global__ void k_ws_classify(const int4* __restrict__ bbox, int total, int* cnt, int* next, int* list) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= total) return;
    const int4 bx = bbox[i];
    if (bx.z < bx.x) cnt[i] = 0;
    else if (ws_box_px(bx) > WS_MIDDLE) list[atomicAdd(next + 1, 1)] = i;
    else if (ws_box_px(bx) > WS_STAGE) list[total - 1 - atomicAdd(next + 4, 1)] = i;
}

// The objects of one tile or of many: items are objects numbered across the
// tiles; the tile of an item is the last descriptor whose obj_base is <= the
// item (seg_base likewise for box segments).
__device__ __forceinline__ int ws_desc_of(const WsDesc* __restrict__ D, int n, int item, bool by_seg) {
    int lo = 0, hi = n - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if ((by_seg ? D[mid].seg_base : D[mid].obj_base) <= item) lo = mid; else hi = mid - 1;
    }
    return lo;
}

// Small boxes: persistent warps drawing objects from a launch-wide counter
// (next[2]), WS_STAGE pixels of stage each.  Writes the basin's rank inside
// the object to out and the basin count to cnt[object]; absent objects and
// larger boxes were sorted out by k_ws_classify.
__global__ void __launch_bounds__(WS_WARPS * 32) k_ws_objects(const WsDesc* __restrict__ D, int n, int total, int h,
                                                               const int4* __restrict__ bbox, int* cnt, int* next,
                                                               int* status) {
    extern __shared__ __align__(16) char ws_smem[];
    const int warp = threadIdx.x >> 5;
    const Team<1> team{(int)threadIdx.x & 31, nullptr};
    char* stage = ws_smem + (size_t)warp * WS_STAGE * WS_PX_BYTES;
    for (int item = ws_next(next + 2, team); item < total; item = ws_next(next + 2, team)) {
        const int4 bx = bbox[item];
        if (bx.z < bx.x || ws_box_px(bx) > WS_STAGE) continue;
        const WsDesc& T = D[ws_desc_of(D, n, item, false)];
        const int c = ws_staged(T.labels, T.edt, T.W, T.H, item - T.obj_base + 1, bx, h, stage, WS_STAGE, T.out,
                                status, team);
        if (team.t == 0) cnt[item] = c;
        __syncwarp();
    }
}

// Larger boxes: the warps of a CTA split one object, with a stage of `cap`
// pixels; drawn from a list (entries list[0], list[step], ...); boxes beyond the
// stage run on the global scratch planes.
__global__ void __launch_bounds__(WS_WARPS * 32) k_ws_team(const WsDesc* __restrict__ D, int n, int h,
                                                           const int4* __restrict__ bbox, int* cnt, int cap,
                                                           uint16_t* gdr, unsigned long long* gw, int* draw,
                                                           const int* __restrict__ listed, const int* __restrict__ list,
                                                           int step, int* status) {
    extern __shared__ __align__(16) char ws_smem[];
    __shared__ int sh[3 + WS_WARPS];
    const Team<WS_WARPS> team{(int)threadIdx.x, sh};
    const int nl = *listed;
    for (int i = ws_next(draw, team); i < nl; i = ws_next(draw, team)) {
        const int item = list[i * step];
        const int4 bx = bbox[item];
        const WsDesc& T = D[ws_desc_of(D, n, item, false)];
        const int k = item - T.obj_base + 1;
        const int c = ws_box_px(bx) <= cap
                          ? ws_staged(T.labels, T.edt, T.W, T.H, k, bx, h, ws_smem, cap, T.out, status, team)
                          : ws_object_global(T.labels, T.edt, T.W, k, bx, h, gdr + T.px_base, gw + T.px_base,
                                             T.out, status, team);
        if (team.t == 0) cnt[item] = c;
    }
}

// In place: cnt[i] -> exclusive prefix; total -> *n_basins (one CTA of 1024).
__device__ __forceinline__ void ws_scan_block(int* cnt, int K, int32_t* n_basins) {
    __shared__ int wsum[32];
    __shared__ int carry;
    const int t = threadIdx.x, lane = t & 31, wid = t >> 5;
    if (t == 0) carry = 0;
    __syncthreads();
    for (int base = 0; base < K; base += 1024) {
        const int i = base + t;
        const int v = i < K ? cnt[i] : 0;
        int x = v;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(WFULL, x, o);
            if (lane >= o) x += y;
        }
        if (lane == 31) wsum[wid] = x;
        __syncthreads();
        if (wid == 0) {
            int s = wsum[lane];
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int y = __shfl_up_sync(WFULL, s, o);
                if (lane >= o) s += y;
            }
            wsum[lane] = s;
        }
        __syncthreads();
        const int excl = carry + (wid ? wsum[wid - 1] : 0) + x - v;
        if (i < K) cnt[i] = excl;
        __syncthreads();
        if (t == 1023) carry = excl + v;
        __syncthreads();
    }
    if (t == 0) *n_basins = carry;
}

// out += o on the pixels of object k inside box bx (one warp).
__device__ __forceinline__ void ws_offset_obj(const int32_t* __restrict__ labels, int W, int k, int4 bx, int o,
                                              int32_t* out, int lane) {
    const int bw = bx.z - bx.x + 1, n = bw * (bx.w - bx.y + 1);
    for (WalkBy<32> it(lane, bw); it.f < n; it.next()) {
        const size_t g = (size_t)(bx.y + it.y) * W + (bx.x + it.x);
        if (labels[g] == k) out[g] += o;
    }
}

constexpr int WS_DESC_PACK = 16;
struct WsDescPack {
    int first, n;
    WsDesc d[WS_DESC_PACK];
};

// Writes the descriptors pk; the launch with the first ones also empties the boxes
// and the counters: a call of up to 16 tiles starts with one launch (64 objects of
// 1 x 1 in 2048^2: 41.5 us, 43.4 to 47.7 with three).
__global__ void __launch_bounds__(256) k_ws_start(WsDesc* dst, const __grid_constant__ WsDescPack pk, int4* bbox, int total,
                                                  int* next) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < pk.n) dst[pk.first + i] = pk.d[i];
    if (pk.first > 0) return;
    if (i < WS_COUNTERS) next[i] = 0;
    if (i < total) bbox[i] = make_int4(0x7fffffff, 0x7fffffff, -1, -1);
}

__global__ void __launch_bounds__(256) k_ws_bbox(const WsDesc* __restrict__ D, int n, int total_segs,
                                                   int4* bbox) {
    const int lane = threadIdx.x & 31;
    const int gw = (int)(((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5);
    if (gw >= total_segs) return;
    const WsDesc& T = D[ws_desc_of(D, n, gw, true)];
    const int k = gw - T.seg_base, spr = (T.W + FB_SEG - 1) / FB_SEG;
    const int y = k / spr, xs = (k - y * spr) * FB_SEG;
    bbox_segment(T.labels + (size_t)y * T.W, T.W, T.K, y, xs, bbox + T.obj_base, lane);
}

__global__ void __launch_bounds__(1024) k_ws_scan(const WsDesc* __restrict__ D, int* cnt) {
    const WsDesc& T = D[blockIdx.x];
    ws_scan_block(cnt + T.obj_base, T.K, T.n_basins);
}

__global__ void __launch_bounds__(256) k_ws_offset(const WsDesc* __restrict__ D, int n, int total,
                                                     const int4* __restrict__ bbox, const int* __restrict__ off) {
    const int lane = threadIdx.x & 31;
    const int nw = gridDim.x * (blockDim.x >> 5);
    for (int item = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); item < total; item += nw) {
        const int o = off[item];
        const int4 bx = bbox[item];
        if (o == 0 || bx.z < bx.x) continue;
        const WsDesc& T = D[ws_desc_of(D, n, item, false)];
        ws_offset_obj(T.labels, T.W, item - T.obj_base + 1, bx, o, T.out, lane);
    }
}

void launch_watershed_batch(const std::vector<WsDesc>& descs, WsDesc* d_descs, int h, int4* bbox, int* cnt,
                            int* next, void* scratch, size_t scratch_px, int* status, int sms, cudaStream_t s,
                            cudaStream_t side, cudaEvent_t fork, cudaEvent_t join, Profiler* pf) {
    static bool attrs[64] = {};  // opt-in shared memory above 48 KB, once per device
    const int small_smem = WS_WARPS * WS_STAGE * WS_PX_BYTES, mid_smem = WS_MIDDLE * WS_PX_BYTES;
    int dev = 0;
    cudaGetDevice(&dev);
    if (dev < 0 || dev >= 64 || !attrs[dev]) {
        cudaFuncSetAttribute(k_ws_objects, cudaFuncAttributeMaxDynamicSharedMemorySize, small_smem);
        cudaFuncSetAttribute(k_ws_team, cudaFuncAttributeMaxDynamicSharedMemorySize, WS_LARGE_SMEM);
        if (dev >= 0 && dev < 64) attrs[dev] = true;
    }
    const int n = (int)descs.size();
    int total = 0, segs = 0;
    for (const WsDesc& d : descs) {
        cudaMemsetAsync(d.out, 0, (size_t)d.W * d.H * sizeof(int32_t), s);
        total += d.K;
        segs += (d.W + FB_SEG - 1) / FB_SEG * d.H;
    }
    if (n == 1 && total == 0) {  // one tile without objects: 10 us, 15 with the launches below
        cudaMemsetAsync(descs[0].n_basins, 0, sizeof(int32_t), s);
        return;
    }
    for (int i = 0; i < n; i += WS_DESC_PACK) {
        WsDescPack pk;
        pk.first = i;
        pk.n = n - i < WS_DESC_PACK ? n - i : WS_DESC_PACK;
        for (int k = 0; k < pk.n; k++) pk.d[k] = descs[i + k];
        pf->begin("ws_start", s);
        k_ws_start<<<i ? 1 : std::max(1, (total + 255) / 256), 256, 0, s>>>(d_descs, pk, bbox, total, next);
        pf->end("ws_start", s);
    }
    if (total > 0) {
        unsigned long long* gw = (unsigned long long*)scratch;
        uint16_t* gdr = (uint16_t*)(gw + scratch_px);
        pf->begin("ws_bbox", s);
        k_ws_bbox<<<(unsigned)(((long long)segs * 32 + 255) / 256), 256, 0, s>>>(d_descs, n, segs, bbox);
        pf->end("ws_bbox", s);
        int* list = next + WS_COUNTERS;
        pf->begin("ws_classify", s);
        k_ws_classify<<<(total + 255) / 256, 256, 0, s>>>(bbox, total, cnt, next, list);
        pf->end("ws_classify", s);
        // The larger boxes on the (higher-priority) side stream, overlapping the small
        // ones; those of the small stage behind the rare ones of the large stage.  (On
        // a stream each: one tile of 4096^2 232 -> 223 us, but 64 objects of one pixel
        // 41.5 -> 43.5 and 3000 of 14 x 14 109 -> 117, for the joins and the order in
        // which the launches get their room.)
        cudaEventRecord(fork, s);
        cudaStreamWaitEvent(side, fork, 0);
        pf->begin("ws_large", side);
        k_ws_team<<<std::min(total, sms * 2), WS_WARPS * 32, WS_LARGE_SMEM, side>>>(
            d_descs, n, h, bbox, cnt, WS_LARGE_SMEM / WS_PX_BYTES, gdr, gw, next, next + 1, list, 1, status);
        pf->end("ws_large", side);
        pf->begin("ws_middle", side);
        // (five of these CTAs fit on an SM; those that come later find what is left to draw)
        k_ws_team<<<std::min(total, sms * 8), WS_WARPS * 32, mid_smem, side>>>(
            d_descs, n, h, bbox, cnt, WS_MIDDLE, gdr, gw, next + 3, next + 4, list + total - 1, -1, status);
        pf->end("ws_middle", side);
        cudaEventRecord(join, side);
        const int ctas = (total + WS_WARPS - 1) / WS_WARPS;
        pf->begin("ws_objects", s);
        k_ws_objects<<<std::min(ctas, sms * 10), WS_WARPS * 32, small_smem, s>>>(d_descs, n, total, h, bbox, cnt, next, status);
        pf->end("ws_objects", s);
        cudaStreamWaitEvent(s, join, 0);
    }
    pf->begin("ws_scan", s);
    k_ws_scan<<<n, 1024, 0, s>>>(d_descs, cnt);
    pf->end("ws_scan", s);
    if (total > 0) {
        const int octas = (total + 7) / 8;
        pf->begin("ws_offset", s);
        k_ws_offset<<<octas < sms * 8 ? octas : sms * 8, 256, 0, s>>>(d_descs, n, total, bbox, cnt);
        pf->end("ws_offset", s);
    }
}

}  // namespace nucseg
