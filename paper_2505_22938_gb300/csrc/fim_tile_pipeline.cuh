#pragma once
// The tile pipeline: one Tx x Ty output tile filtered by one tile group (a CTA, or part of a
// batch CTA) (Sec. 3.3, Sec. 4.2). The single-image and batch kernels include this file.
//
// Phases of one tile, separated by group barriers:
//   1. ordinal transform - the rounded-rectangle footprint (Fig. 10) is read with clamp-to-edge
//                        and key-value sorted by value, giving the omnigram Omega (Sec. 3.3):
//                          8-bit, and 16-bit data in 1024-thread CTAs: counting sort over 256 /
//                                         65536 shared-memory bins, the bucket construction of
//                                         Eq. 5 run by all threads;
//                          float in 1024-thread CTAs, and float and 16-bit data in the 256- and
//                                         512-thread CTAs of larger tiles, where the tile's box
//                                         lies inside the image: counting sort by equalised
//                                         16-bit codes, ties settled at the output;
//                          float otherwise, and 16-bit data in smaller CTAs: LSD radix sort of
//                                         order-preserving keys (Sec. 4.1 float key): for float in
//                                         1024-thread CTAs with room for its bins a 16-bit and
//                                         two 8-bit passes, else 8-bit passes (four / two).
//   2. ordinal image   - I(Omega[v]) = v (Eq. 4), exact 16-bit ranks.
//   3. seed solve      - RB*G seed windows, one warp each: coarse histogram of I over the
//                        window, then a ballot scan of Omega to the exact median (Sec. 4.2).
//                        With a learned bracket (an extension), a block-wide MLP proposes a
//                        rank bracket per seed and exact counts at its ends replace the histogram.
//   4. seed rows       - one warp per (seed, direction) slides the window left/right; lanes
//                        split the kernel rows and reduce the count change (Sec. 3.3 step 4).
//   5. vertical sweep  - one thread per (column, band, direction) slides its window up or
//                        down (Fig. 7), sharing packed compares with its neighbour's window, and
//                        refines it by scanning Omega itself in 64-byte blocks; the last few
//                        lanes of a warp hand very long scans to warp ballots (Sec. 4.1, Eq. 2).
//   6. output          - out = C[m] through the omnigram: the input value at Omega[m].
// Pivots are exact previous medians (Huang's choice, Sec. 3.1): after each solve the count
// below the pivot is exactly the target rank, and a slide only adds the change.
//
// W selects the omnigram encoding: W = 0 packs a location as two int8 coordinates (footprint
// box up to 256 x 256 with one side below 256, Sec. 4.1; -128 marks padding); W = 1 uses two
// int16 coordinates. OG = 1 keeps the omnigram in the CTA's global scratch slice when shared
// memory cannot hold it.
#include <stdint.h>

#include <algorithm>
#include <type_traits>

#include "fim_internal.h"

namespace fim {
namespace {

// First device-side error since the last fim_sync_status(). Each translation unit that includes
// this file has its own word (internal linkage); the host reads and clears all of them.
__device__ int g_status;

constexpr unsigned kFull = 0xffffffffu;

template <int DT>
struct Traits;
template <>
struct Traits<FIM_U8> {
    using T = uint8_t;
    __device__ static uint32_t key(T v) { return v; }
};
template <>
struct Traits<FIM_U16> {
    using T = uint16_t;
    __device__ static uint32_t key(T v) { return v; }
};
template <>
struct Traits<FIM_F32> {
    using T = float;
    // Sign-magnitude to unsigned order (Sec. 4.1): negative values have all bits flipped,
    // non-negative values only the sign bit, so unsigned comparison is IEEE totalOrder.
    __device__ static uint32_t key(T v) {
        const uint32_t b = __float_as_uint(v);
        return b ^ ((uint32_t)((int32_t)b >> 31) | 0x80000000u);
    }
};

// Omnigram entry encodings (locations relative to the footprint box centre cx0, cy0).
template <int W>
struct Loc;
template <>
struct Loc<0> {
    using E = uint16_t;    // entry
    using Pos = uint16_t;  // bounding-box position in the radix lists
    static constexpr int kGroup = 8;  // entries per 128-bit load
    static constexpr E kSentinel = 0x8080;  // (-128, -128): a box side below 256 keeps it out of every window
    __device__ static E pack(int u, int v, int cx0, int cy0) {
        return (E)((uint32_t)(uint8_t)(int8_t)(u - cx0) | ((uint32_t)(uint8_t)(int8_t)(v - cy0) << 8));
    }
    __device__ static int x(uint32_t e) { return (int)(int8_t)(e & 0xffu); }
    __device__ static int y(uint32_t e) { return (int)(int8_t)((e >> 8) & 0xffu); }
};
template <>
struct Loc<1> {
    using E = uint32_t;
    using Pos = uint32_t;
    static constexpr int kGroup = 4;
    static constexpr E kSentinel = 0xC000C000u;  // (-16384, -16384): far outside every window
    __device__ static E pack(int u, int v, int cx0, int cy0) {
        return (E)((uint32_t)(uint16_t)(int16_t)(u - cx0) | ((uint32_t)(uint16_t)(int16_t)(v - cy0) << 16));
    }
    __device__ static int x(uint32_t e) { return (int)(int16_t)(e & 0xffffu); }
    __device__ static int y(uint32_t e) { return (int)(int16_t)(e >> 16); }
};

__device__ __forceinline__ uint32_t lanemask_lt() {
    uint32_t m;
    asm("mov.u32 %0, %%lanemask_lt;" : "=r"(m));
    return m;
}
__device__ __forceinline__ uint32_t lanemask_le() {
    uint32_t m;
    asm("mov.u32 %0, %%lanemask_le;" : "=r"(m));
    return m;
}
__device__ __forceinline__ uint32_t lanemask_ge() {
    uint32_t m;
    asm("mov.u32 %0, %%lanemask_ge;" : "=r"(m));
    return m;
}

__device__ __forceinline__ void set_status(int code) { atomicCAS(&g_status, 0, code); }

// This translation unit's device status word, read and cleared by the host.
inline fim_status read_and_clear_unit_status() {
    int v = 0;
    if (cudaMemcpyFromSymbol(&v, g_status, sizeof(int)) != cudaSuccess) return FIM_ERR_CUDA;
    const int zero = 0;
    if (v != 0 && cudaMemcpyToSymbol(g_status, &zero, sizeof(int)) != cudaSuccess) return FIM_ERR_CUDA;
    return (fim_status)v;
}

__device__ __forceinline__ int clampi(int v, int lo, int hi) { return min(max(v, lo), hi); }

// A tile group: the threads that run one tile's pipeline. A CTA holds one group (single-image
// launches) or several equal groups (batches of small configurations), each with its own
// named barrier and its own partition of shared memory (everything after the kernel tables).
struct Grp {
    int tid, lane, warp;  // group-local indices
    int nthreads;         // group size (the plan's CTA size)
    int bar;              // named barrier; 0 is the whole CTA
    int shift;            // byte shift of this group's shared-memory partition
    __device__ __forceinline__ void sync() const {
        if (bar == 0)
            __syncthreads();
        else
            asm volatile("bar.sync %0, %1;" ::"r"(bar), "r"(nthreads) : "memory");
    }
};

// Diagnostics: thread 0 records clock64() at phase boundaries when a buffer is attached. The
// stamps collect in the group's scan scratch (words 48..63, which no phase uses) and go to the
// buffer together at the end of the tile, so that no stamp waits behind the tile's own global
// stores.
__device__ __forceinline__ void stamp(const Plan& P, int tile, int phase, const Grp& G) {
    if (P.phase_clock != nullptr && G.tid == 0 && tile < P.phase_tiles) {
        extern __shared__ __align__(128) unsigned char smem_base[];
        unsigned long long* st = reinterpret_cast<unsigned long long*>(smem_base + G.shift + P.off_misc + 48 * 4);
        st[phase] = clock64();
        if (phase == 7)
            for (int i = 0; i < 8; ++i) P.phase_clock[tile * 8 + i] = st[i];
    }
}

__device__ __forceinline__ int span_lo(int s) { return (int)(int16_t)(s & 0xffff); }
__device__ __forceinline__ int span_hi(int s) { return s >> 16; }

// The kernel as the membership tests need it (Eq. 2, Eq. 3).
template <int SHAPE, int W>
struct Member;

template <int W>
struct Member<kShapeDisk, W> {
    int r2;  // dx^2 + dy^2 <= r2
};

template <int W>
struct Member<kShapeSpans, W> {
    const uint32_t* test;  // shared memory: the rows' test words (see WordTest)
    int xmin, ymin, nrows;
};

// Membership of the omnigram entries held in one 32-bit word (two 16-bit entries, or one 32-bit
// entry), for a fixed window whose centre (px, py) is given in the entries' coordinate frame:
// bit k of operator() is entry k of the word.
template <int SHAPE, int W>
struct WordTest;

// Disk with 8-bit coordinates: (x-px)^2 + (y-py)^2 <= r2 is evaluated as the sign of
// x^2 + y^2 - 2(x px + y py) + px^2 + py^2 - r2 - 1, two byte dot products per entry on the packed
// pair. The plan keeps -2px and -2py in a signed byte (px, py in [-63, 64]).
template <>
struct WordTest<kShapeDisk, 0> {
    int nR;        // px^2 + py^2 - r2 - 1
    int plo, phi;  // (-2px, -2py, 0, 0) and (0, 0, -2px, -2py) as signed bytes
    __device__ __forceinline__ void init(const Member<kShapeDisk, 0>& mm, int px, int py) {
        nR = px * px + py * py - mm.r2 - 1;
        const uint32_t b = (uint32_t)((-2 * px) & 0xff) | ((uint32_t)((-2 * py) & 0xff) << 8);
        plo = (int)b;
        phi = (int)(b << 16);
    }
    // negative iff the low / high entry of the word is a member
    __device__ __forceinline__ int lo(uint32_t w) const {
        return __dp4a((int)w, plo, __dp4a((int)(w & 0xffffu), (int)w, nR));
    }
    __device__ __forceinline__ int hi(uint32_t w) const {
        return __dp4a((int)w, phi, __dp4a((int)(w & 0xffff0000u), (int)w, nR));
    }
    __device__ __forceinline__ uint32_t operator()(uint32_t w) const {
        return ((uint32_t)lo(w) >> 31) | (((uint32_t)hi(w) >> 31) << 1);
    }
};

// Any convex shape. A kernel row's columns [lo, hi] (counted from the kernel's first column, plus
// 256) stand in one word (0x8000 - lo, 0x7fff - hi): added to the entry's column in both halves,
// bit 31 says "from lo on" and bit 15 "past hi", so that an entry takes two dot products that pick
// its coordinates, a row clamp, a table load, a multiply-add and two bit operations. Row nrows
// stands for every row outside the kernel and holds no column. The entries a warp tests at once
// lie in unrelated rows: eight copies of the table, side by side for the lanes modulo 8, halve the
// bank conflicts of their loads (3.5 -> 2.1 wavefronts on random rows).
template <int W>
struct WordTest<kShapeSpans, W> {
    const uint32_t* test;
    int cx, cy, nrows;
    __device__ __forceinline__ void init(const Member<kShapeSpans, W>& mm, int px, int py) {
        test = mm.test + (threadIdx.x & (kSpanCopies - 1));
        cx = 256 - mm.xmin - px;
        cy = -mm.ymin - py;
        nrows = mm.nrows;
    }
    __device__ __forceinline__ int column(int x, int y) const {
        const uint32_t e = (uint32_t)x * 65537u + test[min((uint32_t)y, (uint32_t)nrows) * kSpanCopies];
        return (int)(e & ~(e << 16));
    }
    // negative iff the low / high entry of the word (W = 0), or the word (W = 1), is a member
    __device__ __forceinline__ int lo(uint32_t w) const {
        if constexpr (W == 0) return column(__dp4a((int)w, 0x00000001, cx), __dp4a((int)w, 0x00000100, cy));
        else return column(__dp2a_lo((int)w, 0x0001, cx), __dp2a_lo((int)w, 0x0100, cy));
    }
    __device__ __forceinline__ int hi(uint32_t w) const {
        return column(__dp4a((int)w, 0x00010000, cx), __dp4a((int)w, 0x01000000, cy));
    }
    __device__ __forceinline__ uint32_t operator()(uint32_t w) const {
        if constexpr (W == 0) return ((uint32_t)lo(w) >> 31) | (((uint32_t)hi(w) >> 31) << 1);
        else return (uint32_t)lo(w) >> 31;
    }
};

// A disk with 16-bit coordinates.
template <>
struct WordTest<kShapeDisk, 1> {
    int r2, px, py;
    __device__ __forceinline__ void init(const Member<kShapeDisk, 1>& mm, int x, int y) {
        r2 = mm.r2;
        px = x;
        py = y;
    }
    __device__ __forceinline__ int lo(uint32_t w) const {  // negative iff the entry is a member
        const int dx = Loc<1>::x(w) - px, dy = Loc<1>::y(w) - py;
        return dx * dx + dy * dy - r2 - 1;
    }
    __device__ __forceinline__ uint32_t operator()(uint32_t w) const { return (uint32_t)lo(w) >> 31; }
};

// Appends the word's membership bits below `mask` (mask moves up by the entries of a word): the
// sign of each entry's test shifts straight in, one funnel shift per entry.
template <int SHAPE, int W>
__device__ __forceinline__ uint32_t push_word(uint32_t mask, const WordTest<SHAPE, W>& wt, uint32_t w) {
    if constexpr (W == 0) mask = __funnelshift_l((uint32_t)wt.hi(w), mask, 1);
    return __funnelshift_l((uint32_t)wt.lo(w), mask, 1);
}

// Membership of the entries of one 64-byte block of the omnigram (32 entries of 16 bits, 16 of 32
// bits): bit k is entry k. Every lane reads its own block. All lanes starting with their block's
// first 16 bytes would meet in two of the eight bank quads per load; lane l instead reads its
// quads in the order k ^ (l & 3), so that a load's eight lanes cover four quads of one half, and
// the order is undone when the four part masks are joined (measured on random blocks: 13.7
// cycles per 128-bit load unordered). The four parts are also independent shift chains.
template <int SHAPE, int W>
__device__ __forceinline__ uint32_t block_mask(const uint4* om128, int b, const WordTest<SHAPE, W>& wt) {
    const int l3 = threadIdx.x & 3;
    const uint4* blk = om128 + 4 * b;
    uint4 q[4];
    uint32_t part[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) q[k] = blk[k ^ l3];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        uint32_t m = push_word(0u, wt, q[k].w);
        m = push_word(m, wt, q[k].z);
        m = push_word(m, wt, q[k].y);
        part[k] = push_word(m, wt, q[k].x);
    }
    if constexpr (W == 0) {  // one byte per part
        const uint32_t s0 = l3 & 1 ? 0x1104u : 0x1140u, s1 = l3 & 2 ? 0x1054u : 0x5410u;
        return __byte_perm(__byte_perm(part[0], part[1], s0), __byte_perm(part[2], part[3], s0), s1);
    } else {
        uint32_t m = 0;
#pragma unroll
        for (int k = 0; k < 4; ++k) m |= part[k] << (4 * (k ^ l3));
        return m;
    }
}

// Position of the k-th lowest set bit (k >= 1) of a mask that holds at least k.
__device__ __forceinline__ int nth_bit(uint32_t m, int k) {
    int pos = 0;
    int c = __popc(m & 0xffffu);
    if (k > c) {
        k -= c;
        m >>= 16;
        pos = 16;
    }
    c = __popc(m & 0xffu);
    if (k > c) {
        k -= c;
        m >>= 8;
        pos += 8;
    }
    for (; k > 1; --k) m &= m - 1;
    return pos + 31 - __clz(m & (0u - m));
}

// Exact selection by ballot scans of the omnigram (Sec. 4.1, Sec. 4.2), one window for the whole
// warp, 32 entries a step. Given a pivot rank p and c = #{window members with rank < p}, returns the
// rank m of the window element with window-rank `target`. All 32 lanes pass the same arguments and
// get the same result; -1 means the counts were inconsistent (never expected). (Two or four
// entries per lane and step take fewer steps but more population counts, whose rate is an eighth
// of an addition's: the seed rows' phase 31k -> 36k and 47k cycles per u16 r = 48 tile.)
template <int SHAPE, int W>
__device__ __forceinline__ int warp_select(const typename Loc<W>::E* __restrict__ om, int N, int p, int c,
                                           int target, int px, int py, const Member<SHAPE, W>& member) {
    const int lane = threadIdx.x & 31;
    WordTest<SHAPE, W> wt;
    wt.init(member, px, py);
    if (c <= target) {  // the answer is at or above p
        int need = target - c + 1;
        for (int v0 = p; v0 < N; v0 += 32) {
            const int v = v0 + lane;
            const bool in = v < N && wt.lo(om[v]) < 0;
            const uint32_t mask = __ballot_sync(kFull, in);
            const int cnt = __popc(mask);
            if (cnt >= need) {
                const uint32_t hit = __ballot_sync(kFull, in && __popc(mask & lanemask_le()) == need);
                return v0 + 31 - __clz(hit);
            }
            need -= cnt;
        }
    } else {  // the answer is below p: walk down, the need-th member met is the answer
        int need = c - target;
        for (int v1 = p; v1 > 0; v1 -= 32) {
            const int v = v1 - 32 + lane;
            const bool in = v >= 0 && wt.lo(om[v]) < 0;
            const uint32_t mask = __ballot_sync(kFull, in);
            const int cnt = __popc(mask);
            if (cnt >= need) {
                const uint32_t hit = __ballot_sync(kFull, in && __popc(mask & lanemask_ge()) == need);
                return v1 - 1 - __clz(hit);
            }
            need -= cnt;
        }
    }
    return -1;
}

// Warp-cooperative exact selection for long walks (seed windows): the same contract as
// warp_select, but every lane tests two consecutive aligned 128-bit groups of entries per
// step, so a warp covers 64 groups (512 entries of 16 bits) per step. A warp reduction of the
// per-lane member counts says whether the step holds the target; only that last step takes the
// warp prefix sum that finds the lane, and the lane picks the entry. Entries past N up to the
// last group are sentinels, never members; groups outside the omnigram count nothing. The loop is
// bounded by the omnigram length.
template <int SHAPE, int W>
__device__ __forceinline__ int wide_select(const typename Loc<W>::E* __restrict__ om, int N, int p, int c,
                                           int target, int px, int py, const Member<SHAPE, W>& member) {
    constexpr int G = Loc<W>::kGroup;
    constexpr int kShift = G == 8 ? 3 : 2;
    constexpr int kb = G / 4;  // entries per 32-bit word
    constexpr uint32_t kAll = (1u << G) - 1;
    const int lane = threadIdx.x & 31;
    WordTest<SHAPE, W> wt;
    wt.init(member, px, py);
    const uint4* om128 = reinterpret_cast<const uint4*>(om);
    const bool up = c <= target;
    int need = up ? target - c + 1 : c - target;
    const int v0 = up ? p : p - 1;  // first entry to examine
    const int glast = (N - 1) >> kShift;
    const int g0 = v0 >> kShift;    // -1 below entry 0
    const int o0 = v0 & (G - 1);
    const uint32_t first = up ? (kAll << o0) & kAll : kAll >> (G - 1 - o0);
    auto test = [&](int g) -> uint32_t {
        if ((unsigned)g > (unsigned)glast) return 0u;
        const uint4 q = om128[g];
        return wt(q.x) | (wt(q.y) << kb) | (wt(q.z) << (2 * kb)) | (wt(q.w) << (3 * kb));
    };
    for (int it = 0; it * 64 <= glast + 1; ++it) {
        // this lane's two groups, in walking order
        const int ga = up ? g0 + 64 * it + 2 * lane : g0 - 64 * it - 2 * lane;
        const int gb = up ? ga + 1 : ga - 1;
        uint32_t ma = test(ga);
        const uint32_t mb = test(gb);
        if (it == 0 && lane == 0) ma &= first;
        const int cnt = __popc(ma) + __popc(mb);
        const int total = (int)__reduce_add_sync(kFull, (unsigned)cnt);
        if (total >= need) {
            int incl = cnt;
            for (int o = 1; o < 32; o <<= 1) {
                const int t = __shfl_up_sync(kFull, incl, o);
                if (lane >= o) incl += t;
            }
            const uint32_t hit = __ballot_sync(kFull, incl >= need);
            const int j = __ffs(hit) - 1;
            int m = 0;
            if (lane == j) {
                int k = need - (incl - cnt);  // the k-th member of this lane's groups, along the walk
                const int ca = __popc(ma);
                const int g = k <= ca ? ga : gb;
                uint32_t mask = k <= ca ? ma : mb;
                if (k > ca) k -= ca;
                if (up) {
                    for (; k > 1; --k) mask &= mask - 1;
                    m = G * g + __ffs(mask) - 1;
                } else {
                    for (; k > 1; --k) mask ^= 1u << (31 - __clz(mask));
                    m = G * g + 31 - __clz(mask);
                }
            }
            return __shfl_sync(kFull, m, j);
        }
        need -= total;
        if (up ? g0 + 64 * (it + 1) > glast : g0 - 64 * (it + 1) < 0) break;
    }
    return -1;
}

// Members of a window below rank `p` (every lane gets the warp's total). Lane l takes kernel rows
// l, l + 32, ... and reads each row segment of the ordinal image in aligned 8-rank chunks (one
// 128-bit load each), comparing the ranks two per 32-bit word; only a row's first and last chunks
// need a mask. `ctr` is the window centre's ordinal-image position shifted by the kernel's first
// row (ymin) rows, as in window_walk; the image is 16-byte aligned.
__device__ __forceinline__ int window_rows_below(const int* spans, int nrows, const uint16_t* ctr, int SP, int p) {
    const int lane = threadIdx.x & 31;
    const uint32_t up = (uint32_t)p;
    int c = 0;
    for (int i = lane; i < nrows; i += 32) {
        const int sp = spans[i];
        const uint16_t* lo = ctr + i * SP + span_lo(sp);
        const uint16_t* hi = ctr + i * SP + span_hi(sp);
        const uint4* q = reinterpret_cast<const uint4*>((uintptr_t)lo & ~(uintptr_t)15);
        const uint4* qe = reinterpret_cast<const uint4*>((uintptr_t)hi & ~(uintptr_t)15);
        for (; q <= qe; ++q) {
            const uint4 v = *q;
            const uint32_t w[4] = {v.x, v.y, v.z, v.w};
            const uint16_t* e0 = reinterpret_cast<const uint16_t*>(q);
            if (e0 >= lo && e0 + 7 <= hi) {
#pragma unroll
                for (int j = 0; j < 4; ++j) c += (int)((w[j] & 0xffffu) < up) + (int)((w[j] >> 16) < up);
            } else {
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    const uint32_t r = (w[j >> 1] >> (16 * (j & 1))) & 0xffffu;
                    c += (int)(e0 + j >= lo && e0 + j <= hi && r < up);
                }
            }
        }
    }
    return (int)__reduce_add_sync(kFull, (unsigned)c);
}

// Per-thread exact selection (vertical sweep): every lane refines its own window. It scans the
// omnigram from its pivot in aligned 64-byte blocks, builds each block's membership mask, and
// stops at the block that holds the target-th member. A warp repeats the block step until its
// longest scan is done; only a few lanes left after many blocks (jumps at edges and impulses) are
// finished one at a time by warp-wide scans.
// Bound by instruction issue: a block takes 64 dot products, 32 masks and 32 shifts, which share
// the issue slots of two half-rate pipes (u16 r = 48: 6.7 blocks per warp and step, 35 % of the
// kernel's instructions). Against scans of 4 or 8 unaligned groups per step with compares and a
// hand-off after 8 groups, the vertical sweep of a u16 r = 48 tile went from 237k to 169k cycles
// together with the packed slide below; a hand-off as early as that costs five warp-wide scans
// per step.
// Arguments: pivot p, members below it c, target t; returns m (-1: inconsistent) and, in *members,
// the members of m's block. Sentinels fill the omnigram's last block. All loops are bounded by the omnigram length.
// A block step costs about 165 instructions for any number of lanes, a hand-off 60 and 25 per 32
// entries for one. In the small CTAs of small kernels, whose scans are one to three blocks, two
// lanes are handed off after four blocks and up to four after eight (impulses: u16 4096^2 r = 4
// 1181 -> 1097 us, 5th percentile r = 5 360 -> 338 us at 2048^2); with the long scans of large
// kernels that costs 4-5 %, and only one or two lanes left after 16 blocks are.
template <int KS>
__device__ __forceinline__ bool hand_off(int blocks, uint32_t alive) {
    if constexpr (KS == 8) return blocks >= 16 && __popc(alive) <= 2;
    else return blocks >= 4 && __popc(alive) <= (blocks >= 8 ? 4 : 2);
}

template <int SHAPE, int W, int KS, bool kDense>
__device__ __forceinline__ int lane_select(const typename Loc<W>::E* __restrict__ om, int N, int p, int c, int t,
                                           int px, int py, const Member<SHAPE, W>& member, uint32_t* members) {
    constexpr int kBlockShift = W == 0 ? 5 : 4;
    constexpr int kBlock = 1 << kBlockShift;  // entries per block
    constexpr uint32_t kAll = kBlock == 32 ? 0xffffffffu : (1u << kBlock) - 1;
    const uint4* om128 = reinterpret_cast<const uint4*>(om);
    const int blast = (N - 1) >> kBlockShift;
    const bool up = c <= t;
    int need = up ? t - c + 1 : c - t;
    const int v = up ? p : max(p - 1, 0);  // next entry to examine
    int b = v >> kBlockShift;
    // the pivot's block counts on the pivot's side only
    uint32_t first = up ? kAll << (v & (kBlock - 1)) : kAll >> (kBlock - 1 - (v & (kBlock - 1)));
    WordTest<SHAPE, W> wt;
    wt.init(member, px, py);
    // Large disks with the omnigram in shared memory (kDense): a lane that has found its block stays on
    // it and computes the same mask again, so that the loop has no divergent branch (u16 r = 48 sweep
    // 147k -> 140k cycles per tile). Where the idle lanes' loads cost more than the branch, they are
    // masked off (hexagon R = 64 241k against 262k, u16 r = 128 221k against 262k, u16 r = 8 64k
    // against 66k). Counts that do not add up end at the omnigram's first or last block and run into
    // the limit.
    const int dir = up ? 1 : -1;
    uint32_t mask = 0;
    int cnt = 0;
    bool todo = true;
    for (int it = 0;; ++it) {
        if (kDense || todo) {
            *members = block_mask<SHAPE, W>(om128, b, wt);
            mask = *members & first;
            cnt = __popc(mask);
            todo = cnt < need;
            if (todo) {
                need -= cnt;
                b = clampi(b + dir, 0, blast);
                first = kAll;
            }
        }
        const uint32_t alive = __ballot_sync(kFull, todo);
        if (alive == 0 || it > blast || hand_off<KS>(it + 1, alive)) break;
    }
    int m = -1;
    if (!todo) m = kBlock * b + nth_bit(mask, up ? need : cnt - need + 1);
    uint32_t rest = __ballot_sync(kFull, todo);
    while (rest) {
        const int j = __ffs(rest) - 1;
        rest &= rest - 1;
        const int upj = __shfl_sync(kFull, (int)up, j);
        const int bj = __shfl_sync(kFull, b, j), nj = __shfl_sync(kFull, need, j);
        const int pxj = __shfl_sync(kFull, px, j), pyj = __shfl_sync(kFull, py, j);
        const int pj = upj ? kBlock * bj : kBlock * bj + kBlock;  // examined so far: all before (after) it
        const int mj = warp_select<SHAPE, W>(om, N, pj, upj ? 0 : nj, upj ? nj - 1 : 0, pxj, pyj, member);
        if ((int)(threadIdx.x & 31) == j) {
            m = mj;
            if (m >= 0) *members = block_mask<SHAPE, W>(om128, m >> kBlockShift, wt);
        }
    }
    return m;
}

// ---- packed slides ---------------------------------------------------------------------------
// Two windows one column apart read their ranks at any kernel column from the halves of one 32-bit
// word of the ordinal image, if that word is aligned. PairBelow compares both halves with the
// windows' pivots at once: with signed ranks (at most 32766) one add-min-relu instruction gives
// [rank >= p] per half; ranks up to 65535 take two unsigned minima and a subtraction, giving
// [rank < p]. `diff` adds the top entry's indicator minus the bottom entry's, so that a window
// sliding down gains exactly the sum of diffs in members below its pivot (its bottom entries
// enter, its top ones leave). The two halves accumulate in one word: differences may borrow across
// the halves, and unpack_pair undoes it.
template <bool S16>
struct PairBelow {
    uint32_t pv;  // S16: 1 - p per half, otherwise p per half
    __device__ __forceinline__ void init(int p0, int p1) {
        if constexpr (S16) {
            p0 = 1 - p0;
            p1 = 1 - p1;
        }
        pv = __byte_perm((uint32_t)p0, (uint32_t)p1, 0x5410);
    }
    __device__ __forceinline__ int diff(int acc, uint32_t top, uint32_t bot) const {
        if constexpr (S16) {
            return acc + (int)__viaddmin_s16x2_relu(top, pv, 0x00010001u) -
                   (int)__viaddmin_s16x2_relu(bot, pv, 0x00010001u);
        } else {
            return acc + (int)__vminu2(pv - __vminu2(bot, pv), 0x00010001u) -
                   (int)__vminu2(pv - __vminu2(top, pv), 0x00010001u);
        }
    }
};

__device__ __forceinline__ void unpack_pair(int acc, int* lo, int* hi) {
    *lo = (int)(int16_t)(acc & 0xffff);
    *hi = (acc - *lo) >> 16;
}

// Count change of every lane's window for one vertical step, lanes on adjacent columns. Each lane
// takes the kernel columns whose words are aligned for its own window (box columns of its own
// parity) and counts them for its window and the next lane's, so the warp reads and compares every
// (window, column) pair once, two per instruction; each lane then adds the previous lane's high
// half. The warp's first window has no previous lane: its other columns are split over the lanes.
// `ctr` is the byte address of the window's centre in the ordinal image (one row above it for a
// step up). `tab` lists the kernel columns as (top entry, bottom entry + 1) byte offsets, in units
// of two columns of even box columns followed by two of odd ones; `units` such pairs. p is the
// pivot as the ordinal image holds ranks. Returns the difference for a downward step.
// Bound by issue: eight instructions (two loads, two compares, one accumulation, two addresses,
// half a table load) per kernel column and two windows, against 18 for two 16-bit loads and
// compares per window.
template <bool S16, int kUnroll>
__device__ __forceinline__ int slide(const unsigned char* ctr, const int4* tab, int units, int p) {
    const int lane = threadIdx.x & 31;
    const int pn = __shfl_down_sync(kFull, p, 1);
    PairBelow<S16> pair;
    pair.init(p, pn);
    auto word = [](const unsigned char* q, int off) { return *reinterpret_cast<const uint32_t*>(q + off); };
    const int4* mine = tab + (lane & 1);
    int a = 0, a2 = 0;
#pragma unroll kUnroll
    for (int j = 0; j < units; ++j) {
        const int4 o = mine[2 * j];
        a = pair.diff(a, word(ctr, o.x), word(ctr, o.y));
        a2 = pair.diff(a2, word(ctr, o.z), word(ctr, o.w));
    }
    // the first window's odd columns (its own column is even), one or two per lane
    const unsigned char* c0 = ctr - 2 * lane;
    const int pf = __shfl_sync(kFull, p, 0);
    int s = 0;
    for (int i = lane; i < 2 * units; i += 32) {
        const int2 o = reinterpret_cast<const int2*>(tab + 1 + (i >> 1) * 2)[i & 1];
        s += (int)(*reinterpret_cast<const uint16_t*>(c0 + o.y) < pf) -
             (int)(*reinterpret_cast<const uint16_t*>(c0 + o.x) < pf);
    }
    s = __reduce_add_sync(kFull, s);
    int lo, hi;
    unpack_pair(a + a2, &lo, &hi);
    const int prev = __shfl_up_sync(kFull, hi, 1);
    return lo + (lane == 0 ? s : prev);
}

// Kernels of up to kScalarUnits units (12 columns) take slide_scalar: at 4096^2 u16 r = 4 it is 1.06x,
// at u16 416x568 r = 5 1.11x the packed form, whose exchange costs about 80 instructions a step.
constexpr int kScalarUnits = 3;
// The same count change, every lane reading its own window's ranks one by one: for kernels of a few
// columns, where the exchange between the lanes would cost more than it saves.
__device__ __forceinline__ int slide_scalar(const unsigned char* ctr, const int4* tab, int units, int p) {
    auto below = [&](int off) { return (int)(*reinterpret_cast<const uint16_t*>(ctr + off) < p); };
    int d = 0;
#pragma unroll 4
    for (int j = 0; j < 2 * units; ++j) {
        const int4 o = tab[j];
        d += below(o.y) - below(o.x) + below(o.w) - below(o.z);
    }
    return d;
}

// Block-wide exclusive scan of 65536 16-bit counters packed two per word (bin 2k in the low
// half of word k). Offsets stay below 2^16 because the footprint holds at most 65535 pixels.
__device__ void scan_bins16(uint32_t* bins, uint32_t* wtot, const Plan& P, const Grp& G) {
    const int lane = G.lane, warp = G.warp;
    const int chunk = 32768 / P.nwarps;  // words per warp, a multiple of 128
    uint4* b4 = reinterpret_cast<uint4*>(bins + warp * chunk);
    uint32_t acc = 0;
    for (int it = 0; it < chunk / 128; ++it) {
        const uint4 q = b4[it * 32 + lane];
        acc += ((q.x + (q.x >> 16)) & 0xffffu) + ((q.y + (q.y >> 16)) & 0xffffu) +
               ((q.z + (q.z >> 16)) & 0xffffu) + ((q.w + (q.w >> 16)) & 0xffffu);
    }
    acc = __reduce_add_sync(kFull, acc);
    if (lane == 0) wtot[warp] = acc;
    G.sync();
    if (warp == 0) {
        const uint32_t x = lane < P.nwarps ? wtot[lane] : 0;
        uint32_t incl = x;
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t t = __shfl_up_sync(kFull, incl, o);
            if (lane >= o) incl += t;
        }
        wtot[lane] = incl - x;
    }
    G.sync();
    uint32_t run = wtot[warp];
    for (int it = 0; it < chunk / 128; ++it) {
        uint4 q = b4[it * 32 + lane];
        const uint32_t s = ((q.x + (q.x >> 16)) & 0xffffu) + ((q.y + (q.y >> 16)) & 0xffffu) +
                           ((q.z + (q.z >> 16)) & 0xffffu) + ((q.w + (q.w >> 16)) & 0xffffu);
        uint32_t incl = s;
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t t = __shfl_up_sync(kFull, incl, o);
            if (lane >= o) incl += t;
        }
        uint32_t b = run + incl - s;
        uint32_t w[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const uint32_t lo = w[k] & 0xffffu, hi = w[k] >> 16;
            w[k] = b | ((b + lo) << 16);
            b += lo + hi;
        }
        b4[it * 32 + lane] = make_uint4(w[0], w[1], w[2], w[3]);
        run += __shfl_sync(kFull, incl, 31);
    }
    G.sync();
}

// Block-wide exclusive scan of 32768 32-bit counters, offset by `base`; returns their total
// (every thread). Each warp owns a contiguous chunk; each lane 4 counters (one 128-bit word) per
// 128-counter slab.
__device__ uint32_t scan_bins32(uint32_t* bins, uint32_t* wtot, uint32_t base, const Plan& P, const Grp& G) {
    const int lane = G.lane, warp = G.warp;
    const int chunk = 32768 / P.nwarps;  // counters per warp, a multiple of 128
    uint4* b4 = reinterpret_cast<uint4*>(bins + warp * chunk);
    uint32_t acc = 0;
    for (int it = 0; it < chunk / 128; ++it) {
        const uint4 q = b4[it * 32 + lane];
        acc += q.x + q.y + q.z + q.w;
    }
    acc = __reduce_add_sync(kFull, acc);
    if (lane == 0) wtot[warp] = acc;
    G.sync();
    if (warp == 0) {
        const uint32_t x = lane < P.nwarps ? wtot[lane] : 0;
        uint32_t incl = x;
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t t = __shfl_up_sync(kFull, incl, o);
            if (lane >= o) incl += t;
        }
        wtot[lane] = incl - x;
        if (lane == 31) wtot[32] = incl;
    }
    G.sync();
    uint32_t run = base + wtot[warp];
    const uint32_t total = wtot[32];
    for (int it = 0; it < chunk / 128; ++it) {
        uint4 q = b4[it * 32 + lane];
        const uint32_t sum = q.x + q.y + q.z + q.w;
        uint32_t incl = sum;
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t t = __shfl_up_sync(kFull, incl, o);
            if (lane >= o) incl += t;
        }
        uint32_t b = run + incl - sum;
        const uint32_t c0 = q.x, c1 = q.y, c2 = q.z;
        q.x = b;
        q.y = b + c0;
        q.z = q.y + c1;
        q.w = q.z + c2;
        b4[it * 32 + lane] = q;
        run += __shfl_sync(kFull, incl, 31);
    }
    G.sync();
    return total;
}

// The image as the tile pipeline reads it, held in registers.
struct Img {
    const char* in;
    long long pitch;
    int w, h;
    __device__ __forceinline__ explicit Img(const Plan& P)
        : in(static_cast<const char*>(P.in)), pitch(P.pitch), w(P.w), h(P.h) {}
};

template <int DT>
__device__ __forceinline__ typename Traits<DT>::T load_px(const Img& im, int gx, int gy) {
    using V = typename Traits<DT>::T;
    const V* row = reinterpret_cast<const V*>(im.in + (long long)clampi(gy, 0, im.h - 1) * im.pitch);
    return __ldg(row + clampi(gx, 0, im.w - 1));
}

// Where phase 1 reads the footprint from: the box staged in shared memory by the tensor memory
// accelerator (interior tiles), or the image in global memory with clamp-to-edge (every other
// tile). `off` is the staged column of box column 0 (the copy starts on a 16-byte boundary).
// STAGED is fixed per call (the sorts are compiled for both), so the loads of the global-memory
// form stay free of a per-pixel branch.
template <int DT>
struct Footprint {
    using V = typename Traits<DT>::T;
    const unsigned char* stage;  // null: read the image
    int pitch;                   // bytes per staged row
    int off;
    Img im;
    int gx0, gy0;
    template <bool STAGED>
    __device__ __forceinline__ uint32_t key(int u, int v) const {
        if constexpr (STAGED) return Traits<DT>::key(reinterpret_cast<const V*>(stage + v * pitch)[u + off]);
        else return Traits<DT>::key(load_px<DT>(im, gx0 + u, gy0 + v));
    }
};

__device__ __forceinline__ uint32_t smem_addr(const void* p) {
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

// mbarrier of the footprint copies: one arrival (the issuing thread) plus the copy's bytes.
__device__ __forceinline__ void mbar_init(uint64_t* bar) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_addr(bar)) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}

// Copies the box of `rows` x `cols` elements at image column x0 (a multiple of 16 bytes) and row
// y0 into shared memory at dst, completing on `bar` (issued by one thread).
__device__ __forceinline__ void tma_load_box(const void* tmap, unsigned char* dst, uint64_t* bar, int x0, int y0,
                                             uint32_t bytes) {
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_addr(bar)), "r"(bytes)
                 : "memory");
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];"
        ::"r"(smem_addr(dst)), "l"(reinterpret_cast<uint64_t>(tmap)), "r"(x0), "r"(y0), "r"(smem_addr(bar))
        : "memory");
}

// Waits for phase `parity` of `bar` to complete; gives up (false) after a bounded number of tries.
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity) {
    const uint32_t a = smem_addr(bar);
    for (int i = 0; i < (1 << 22); ++i) {
        uint32_t done;
        asm volatile(
            "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
            : "=r"(done)
            : "r"(a), "r"(parity)
            : "memory");
        if (done) return true;
    }
    return false;
}

// State of the footprint copies of one CTA across its tiles.
struct TmaState {
    uint32_t parity;  // phase of the next copy's completion
    int off;          // 1 once a copy timed out: global loads from then on
};

// Counting-sort ordinal transform for 8/16-bit data (Sec. 4.1, Eq. 5): histogram of the
// footprint, exclusive prefix, then every pixel takes the next free ordinal of its value.
// Ties get consecutive ordinals in arrival order, which is all the method needs.
template <int DT, int W, bool STAGED>
__device__ void ordinal_transform_count(const Plan& P, const int* frow, uint32_t* bins, uint32_t* misc,
                                        typename Loc<W>::E* om, const Footprint<DT>& fp, const Grp& G) {
    const int tid = G.tid, lane = G.lane, warp = G.warp;
    const int SH = P.SH, nwarps = P.nwarps, cx0 = P.cx0, cy0 = P.cy0;
    constexpr bool k16 = DT == FIM_U16;
    constexpr int kLoads = 8;
    if constexpr (k16) {
        if (P.sort == kSortCount16x2) {
            // Footprints of more than 65535 pixels: the same construction in two rounds over the
            // key range (top bit 0, then 1), each with 32768 32-bit bins in the same 128 KiB; the
            // second round's offsets start after the first round's pixels.
            uint32_t base = 0;
            for (int h = 0; h < 2; ++h) {
                for (int i = tid * 4; i < 32768; i += P.threads * 4)
                    *reinterpret_cast<uint4*>(bins + i) = make_uint4(0, 0, 0, 0);
                G.sync();
                for (int v = warp; v < SH; v += nwarps) {
                    const int fr = frow[v];
                    const int hi = span_hi(fr);
                    for (int u0 = span_lo(fr) + lane; u0 <= hi; u0 += 32 * kLoads) {
                        uint32_t key[kLoads];
#pragma unroll
                        for (int k = 0; k < kLoads; ++k)
                            key[k] = u0 + 32 * k <= hi ? fp.template key<STAGED>(u0 + 32 * k, v) : 0xffffffffu;
#pragma unroll
                        for (int k = 0; k < kLoads; ++k)
                            if ((key[k] >> 15) == (uint32_t)h) atomicAdd(&bins[key[k] & 0x7fffu], 1u);
                    }
                }
                G.sync();
                base += scan_bins32(bins, misc, base, P, G);
                for (int v = warp; v < SH; v += nwarps) {
                    const int fr = frow[v];
                    const int hi = span_hi(fr);
                    for (int u0 = span_lo(fr) + lane; u0 <= hi; u0 += 32 * kLoads) {
                        uint32_t key[kLoads];
#pragma unroll
                        for (int k = 0; k < kLoads; ++k)
                            key[k] = u0 + 32 * k <= hi ? fp.template key<STAGED>(u0 + 32 * k, v) : 0xffffffffu;
#pragma unroll
                        for (int k = 0; k < kLoads; ++k)
                            if ((key[k] >> 15) == (uint32_t)h)
                                om[atomicAdd(&bins[key[k] & 0x7fffu], 1u)] = Loc<W>::pack(u0 + 32 * k, v, cx0, cy0);
                    }
                }
                G.sync();
            }
            return;
        }
    }
    const int nwords = k16 ? 32768 : 256;
    for (int i = tid * 4; i < nwords; i += P.threads * 4)
        *reinterpret_cast<uint4*>(bins + i) = make_uint4(0, 0, 0, 0);
    G.sync();
    // A warp takes one footprint row at a time; each lane loads up to kLoads pixels of it (all in
    // flight at once) before it issues their shared-memory atomics.
    for (int v = warp; v < SH; v += nwarps) {
        const int fr = frow[v];
        const int hi = span_hi(fr);
        for (int u0 = span_lo(fr) + lane; u0 <= hi; u0 += 32 * kLoads) {
            uint32_t key[kLoads];
#pragma unroll
            for (int k = 0; k < kLoads; ++k)
                key[k] = u0 + 32 * k <= hi ? fp.template key<STAGED>(u0 + 32 * k, v) : 0u;
#pragma unroll
            for (int k = 0; k < kLoads; ++k) {
                if (u0 + 32 * k > hi) break;
                if (k16)
                    atomicAdd(&bins[key[k] >> 1], 1u << ((key[k] & 1u) << 4));
                else
                    atomicAdd(&bins[key[k]], 1u);
            }
        }
    }
    G.sync();
    if (k16) {
        scan_bins16(bins, misc, P, G);
    } else {
        if (warp == 0) {
            uint32_t c[8], s = 0;
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                c[k] = bins[lane * 8 + k];
                s += c[k];
            }
            uint32_t incl = s;
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t t = __shfl_up_sync(kFull, incl, o);
                if (lane >= o) incl += t;
            }
            uint32_t b = incl - s;
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                bins[lane * 8 + k] = b;
                b += c[k];
            }
        }
        G.sync();
    }
    for (int v = warp; v < SH; v += nwarps) {
        const int fr = frow[v];
        const int hi = span_hi(fr);
        for (int u0 = span_lo(fr) + lane; u0 <= hi; u0 += 32 * kLoads) {
            uint32_t key[kLoads];
#pragma unroll
            for (int k = 0; k < kLoads; ++k)
                key[k] = u0 + 32 * k <= hi ? fp.template key<STAGED>(u0 + 32 * k, v) : 0u;
#pragma unroll
            for (int k = 0; k < kLoads; ++k) {
                if (u0 + 32 * k > hi) break;
                uint32_t o;
                if (k16) {
                    const uint32_t sh = (key[k] & 1u) << 4;
                    o = (atomicAdd(&bins[key[k] >> 1], 1u << sh) >> sh) & 0xffffu;
                } else {
                    o = atomicAdd(&bins[key[k]], 1u);
                }
                om[o] = Loc<W>::pack(u0 + 32 * k, v, cx0, cy0);
            }
        }
    }
}

// ---- ordinal transform by equalised codes --------------------------------------------------
// Float keys have no counting sort of their own size, and an LSD radix sort's stable passes cost a
// warp match per 32 pixels (64 cycles of the SM where the digits differ) and a scattered global
// store. In CTAs of 256 threads or more one counting sort places every pixel by a 16-bit code that follows the
// tile's own distribution instead: histograms of a sample of the footprint over the keys' top bits
// deal out codes in proportion, in two levels so that a tile whose values differ in their low
// bits only is resolved as well, and within one bin the code is linear in the key. Codes never
// decrease with the key, so pixels of different codes are in order; pixels of equal code (about
// one other each) stay in any order, and `tie` has a bit per rank that shares its predecessor's
// code. All counts, pivots and scans then work in this fixed total order, and the one place where
// the order among equal codes matters, the value of a solved pixel, is settled there
// (resolve_tie): for one pixel in five a comparison of two or three keys, instead of an exact order
// of all the footprint's. (f32 8192^2 r = 64: the sort 227k -> 83k cycles per tile, the sweep
// 143k -> 163k, the launch 13.2 -> 9.8 ms; the passes are bound by their shared-memory atomics
// and table look-ups.)

// Group of equal codes around rank v: its first rank, and one past its last. Rank 0 has no bit, and
// a zero bit follows the last rank.
__device__ __forceinline__ int tie_start(const uint32_t* tie, int v) {
    int w = v >> 5;
    uint32_t m = ~tie[w] & (0xffffffffu >> (31 - (v & 31)));
    while (m == 0) m = ~tie[--w];
    return 32 * w + 31 - __clz(m);
}
__device__ __forceinline__ int tie_end(const uint32_t* tie, int v) {
    int w = (v + 1) >> 5;
    uint32_t m = ~tie[w] & (0xffffffffu << ((v + 1) & 31));
    while (m == 0) m = ~tie[++w];
    return 32 * w + __ffs(m) - 1;
}

// The rank that holds the value of the window's element of rank m: where m shares its code with
// other members of the window, the one with as many smaller members among them as precede m.
// `mask` holds the members of m's 64-byte block, which a group rarely leaves; groups that do, and
// groups with more than four members in the window, are walked entry by entry.
template <class T, class K>
__device__ __forceinline__ int resolve_tie(const uint16_t* om, const uint32_t* tie, int m, uint32_t mask, const T& wt,
                                           K&& key_of) {
    const uint32_t t = tie[m >> 5], next = tie[(m >> 5) + 1];
    const uint32_t upto = 0xffffffffu >> (31 - (m & 31));  // entries of the block up to m
    const uint32_t zlo = ~t & upto, zhi = ~t & ~upto;
    if (zlo != 0 && (zhi != 0 || (next & 1u) == 0)) {  // the group lies in the block
        // its entries: from the highest zero bit up to m on, below the lowest zero bit after m
        const uint32_t group = (zhi != 0 ? (zhi & (0u - zhi)) - 1u : 0xffffffffu) & ~((1u << (31 - __clz(zlo))) - 1u);
        uint32_t in = mask & group;
        if ((in & (in - 1u)) == 0) return m;
        const int before = __popc(in & (upto >> 1)), base = m & ~31;
        const uint32_t low = in & (0u - in);
        if (((in ^ low) & ((in ^ low) - 1u)) == 0) {  // two members
            const int a = base + 31 - __clz(low), b = base + 31 - __clz(in);
            const uint32_t ka = key_of(om[a]), kb = key_of(om[b]);
            return (before == 0) == (ka <= kb) ? a : b;
        }
        int r[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {  // the members, in rank order; the last one repeats
            r[i] = base + 31 - __clz(in & (0u - in));
            const uint32_t rest = in & (in - 1u);
            in = rest != 0 || i == 3 ? rest : in;
        }
        if (in == 0) {  // at most four
            uint32_t k[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) k[i] = key_of(om[r[i]]);
            int ans = m;
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                if (i > 0 && r[i] == r[i - 1]) continue;
                int less = 0;
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    if (j != i && (j == 0 || r[j] != r[j - 1])) less += j < i ? k[j] <= k[i] : k[j] < k[i];
                if (less == before) ans = r[i];
            }
            return ans;
        }
    }
    const int s = tie_start(tie, m), e = tie_end(tie, m);
    int n = 0, before = 0;
    for (int u = s; u < e; ++u)
        if (wt.lo(om[u]) < 0) {
            ++n;
            before += u < m;
        }
    if (n <= 1) return m;
    // the members' distinct keys in ascending order, until one covers place `before`
    uint32_t last = 0;
    for (bool any = false;; any = true) {
        uint32_t least = 0xffffffffu;
        int at = -1, cnt = 0;
        for (int u = s; u < e; ++u) {
            if (wt.lo(om[u]) >= 0) continue;
            const uint32_t k = key_of(om[u]);
            if (any && k <= last) continue;
            if (at < 0 || k < least) {
                least = k;
                at = u;
                cnt = 0;
            }
            cnt += k == least;
        }
        if (at < 0 || before < cnt) return at < 0 ? m : at;
        before -= cnt;
        last = least;
    }
}

// Deals out places in proportion to n counts (n a multiple of the group's threads): entry i becomes
// its first place | its number of places << 16, one place plus floor(count * scale).
__device__ void deal_places(uint32_t* t, int n, float scale, uint32_t* wtot, const Plan& P, const Grp& G) {
    const int per = n / P.threads;
    uint32_t sum = 0;
    for (int j = 0; j < per; ++j) sum += 1u + (uint32_t)((float)t[G.tid * per + j] * scale);
    uint32_t incl = sum;
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t v = __shfl_up_sync(kFull, incl, o);
        if (G.lane >= o) incl += v;
    }
    if (G.lane == 31) wtot[G.warp] = incl;
    G.sync();
    uint32_t base = incl - sum;
    for (int w = 0; w < G.warp; ++w) base += wtot[w];
    for (int j = 0; j < per; ++j) {
        const uint32_t c = 1u + (uint32_t)((float)t[G.tid * per + j] * scale);
        t[G.tid * per + j] = base | (c << 16);
        base += c;
    }
    G.sync();
}

// Exclusive scan of P.codes 16-bit counters packed two per word, as scan_bins16, setting the tie
// bits of every code with 2 to kMaxTie pixels. Codes of more go to `list` (first rank | pixels << 16),
// *listed of them.
__device__ void scan_codes(uint32_t* bins, uint32_t* tie, uint32_t* list, uint32_t* listed, int cap, uint32_t* wtot,
                           const Plan& P, const Grp& G) {
    const int lane = G.lane, warp = G.warp;
    const int chunk = P.codes / 2 / P.nwarps;  // words per warp, a multiple of 128
    uint4* b4 = reinterpret_cast<uint4*>(bins + warp * chunk);
    uint32_t acc = 0;
    for (int it = 0; it < chunk / 128; ++it) {
        const uint4 q = b4[it * 32 + lane];
        acc += ((q.x + (q.x >> 16)) & 0xffffu) + ((q.y + (q.y >> 16)) & 0xffffu) +
               ((q.z + (q.z >> 16)) & 0xffffu) + ((q.w + (q.w >> 16)) & 0xffffu);
    }
    acc = __reduce_add_sync(kFull, acc);
    if (lane == 0) wtot[warp] = acc;
    G.sync();
    uint32_t run = 0;
    for (int w = 0; w < warp; ++w) run += wtot[w];
    for (int it = 0; it < chunk / 128; ++it) {
        uint4 q = b4[it * 32 + lane];
        const uint32_t s = ((q.x + (q.x >> 16)) & 0xffffu) + ((q.y + (q.y >> 16)) & 0xffffu) +
                           ((q.z + (q.z >> 16)) & 0xffffu) + ((q.w + (q.w >> 16)) & 0xffffu);
        uint32_t incl = s;
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t t = __shfl_up_sync(kFull, incl, o);
            if (lane >= o) incl += t;
        }
        uint32_t b = run + incl - s;
        uint32_t w[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const uint32_t lo = w[k] & 0xffffu, hi = w[k] >> 16;
            w[k] = b | ((b + lo) << 16);
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const uint32_t c = h ? hi : lo;
                if (c > (uint32_t)kMaxTie) {
                    const uint32_t at = atomicAdd(listed, 1u);
                    if (at < (uint32_t)cap) list[at] = b | (c << 16);
                    b += c;
                    continue;
                }
                uint32_t v = b + 1;  // ranks b + 1 .. b + c - 1 share their predecessor's code
                b += c;
                while (v < b) {
                    const uint32_t len = min(b - v, 32u - (v & 31u));
                    atomicOr(&tie[v >> 5], (0xffffffffu >> (32u - len)) << (v & 31u));
                    v += len;
                }
            }
        }
        b4[it * 32 + lane] = make_uint4(w[0], w[1], w[2], w[3]);
        run += __shfl_sync(kFull, incl, 31);
    }
}

// Calls f(column, row, load(column, row)) for every footprint pixel of the rows v0, v0 + dv, ...: one
// row per warp in turn, up to eight pixels of a lane loaded before the first call.
template <class Ld, class Fn>
__device__ __forceinline__ void each_pixel(const Plan& P, const int* frow, const Grp& G, int v0, int dv, Ld&& load,
                                           Fn&& f) {
    for (int v = v0 + G.warp * dv; v < P.SH; v += P.nwarps * dv) {
        const int fr = frow[v], hi = span_hi(fr);
        for (int u0 = span_lo(fr) + G.lane; u0 <= hi; u0 += 256) {
            uint32_t x[8];
#pragma unroll
            for (int k = 0; k < 8; ++k) x[k] = u0 + 32 * k <= hi ? load(u0 + 32 * k, v) : 0u;
#pragma unroll
            for (int k = 0; k < 8; ++k)
                if (u0 + 32 * k <= hi) f(u0 + 32 * k, v, x[k]);
        }
    }
}

// Builds the omnigram and the tie bits; false (to every thread) if the tile's groups of equal code
// hold too many different keys, which then takes the radix sort. `work`: P.codes 16-bit bins,
// then the dealing tables. `code` keeps every box position's code from the count to the scatter.
template <int DT, int W, bool STAGED>
__device__ bool ordinal_transform_codes(const Plan& P, const int* frow, uint32_t* work, uint32_t* tie, uint16_t* code,
                                        uint32_t* misc, typename Loc<W>::E* om, const Footprint<DT>& fp, const Grp& G) {
    const int tid = G.tid, N = P.N, nt = P.threads, nb = 1 << P.code_bits, shift = 32 - P.code_bits;
    uint32_t* bins = work;
    uint32_t* t1 = work + P.codes / 2;
    uint32_t* t2 = t1 + nb;
    constexpr bool kTwo = DT == FIM_F32;              // 16-bit keys need one dealing level
    constexpr int kKeyShift = DT == FIM_U16 ? 16 : 0;  // (the tables take 32-bit keys)
    const int tables = kTwo ? 3 * nb : nb;
    const int nwords = P.codes / 2 + tables, ntie = N / 32 + 2;
    for (int i = 4 * tid; i < nwords; i += 4 * nt) *reinterpret_cast<uint4*>(work + i) = make_uint4(0, 0, 0, 0);
    for (int i = tid; i < ntie; i += nt) tie[i] = 0;
    if (tid == 0) misc[36] = misc[37] = 0;
    G.sync();
    auto key = [&](int u, int v) { return fp.template key<STAGED>(u, v) << kKeyShift; };
    // (scales rounded down: never more places than there are)
    each_pixel(P, frow, G, P.sample_step / 2, P.sample_step, key,
               [&](int, int, uint32_t k) { atomicAdd(&t1[k >> shift], 1u); });
    G.sync();
    deal_places(t1, nb, 0.9999f / (float)P.nsample * (float)(kTwo ? nb : P.codes - nb), misc, P, G);
    if constexpr (kTwo) {
    each_pixel(P, frow, G, 0, 2, key, [&](int, int, uint32_t k) {
        const uint32_t e = t1[k >> shift];
        atomicAdd(&t2[(e & 0xffffu) + __umulhi(k << P.code_bits, e >> 16)], 1u);
    });
    G.sync();
    deal_places(t2, 2 * nb, 0.9999f / (float)P.nsample2 * (float)(P.codes - 2 * nb), misc, P, G);
    }
    auto code_of = [&](uint32_t k) -> uint32_t {
        const uint32_t e = t1[k >> shift];
        if constexpr (!kTwo) return (e & 0xffffu) + __umulhi(k << P.code_bits, e >> 16);
        const unsigned long long p = (unsigned long long)(k << P.code_bits) * (e >> 16);
        const uint32_t e2 = t2[(e & 0xffffu) + (uint32_t)(p >> 32)];
        return (e2 & 0xffffu) + __umulhi((uint32_t)p, e2 >> 16);
    };
    each_pixel(P, frow, G, 0, 1, key, [&](int u, int v, uint32_t k) {
        const uint32_t c = code_of(k);
        code[v * P.S + u] = (uint16_t)c;
        atomicAdd(&bins[c >> 1], 1u << ((c & 1u) << 4));
    });
    G.sync();
    uint32_t* list = t1;  // (the codes are known: the tables are free)
    const int cap = tables;
    scan_codes(bins, tie, list, &misc[36], cap, misc, P, G);
    G.sync();
    each_pixel(P, frow, G, 0, 1, [&](int u, int v) -> uint32_t { return code[v * P.S + u]; },
               [&](int u, int v, uint32_t c) {
                   const uint32_t sh = (c & 1u) << 4;
                   om[(atomicAdd(&bins[c >> 1], 1u << sh) >> sh) & 0xffffu] = Loc<W>::pack(u, v, P.cx0, P.cy0);
               });
    const int n = (int)misc[36];
    if (n == 0) return true;
    if (n > cap) return false;
    // Codes of many pixels. Where all keys are equal (flat areas, impulses, data of few distinct values)
    // the group needs no order; one with different keys leaves the tile to the radix sort. Groups of
    // up to 1024 pixels take a warp each, larger ones the whole tile group.
    G.sync();
    auto key_at = [&](int v) {
        const uint32_t e = om[v];
        return fp.template key<STAGED>(Loc<W>::x(e) + P.cx0, Loc<W>::y(e) + P.cy0);
    };
    auto settle = [&](uint32_t first, uint32_t count, int from, int by) {
        const uint32_t k0 = key_at((int)first);
        bool same = true;
        for (uint32_t i = 1 + from; i < count; i += by) same = same && key_at((int)(first + i)) == k0;
        if (!same) misc[37] = 1;
    };
    for (int i = G.warp; i < n; i += P.nwarps)
        if (list[i] >> 16 <= 1024u) settle(list[i] & 0xffffu, list[i] >> 16, G.lane, 32);
    for (int i = 0; i < n; ++i)
        if (list[i] >> 16 > 1024u) settle(list[i] & 0xffffu, list[i] >> 16, tid, nt);
    G.sync();
    return misc[37] == 0;
}

// The valid lanes whose byte equals this lane's: eight votes (about 32 issue slots), where a warp match
// takes two cycles of the SM per distinct value.
__device__ __forceinline__ uint32_t same_byte(int d, bool valid) {
    uint32_t peers = __ballot_sync(kFull, valid);
#pragma unroll
    for (int b = 0; b < 8; ++b) {
        const bool bit = (d >> b) & 1;
        const uint32_t m = __ballot_sync(kFull, bit);
        peers &= bit ? m : ~m;
    }
    return peers;
}

// LSD radix ordinal transform over bounding-box positions. Float keys in 1024-thread CTAs (C16):
// a 65536-bin counting pass on the low 16 bits (Eq. 5's construction, like 16-bit data) followed
// by two stable 8-bit passes on the high bytes; otherwise 8-bit passes only, four for 32-bit
// float keys and two for 16-bit data. The first pass may order equal digits arbitrarily
// (shared-memory atomics), since the later passes are stable. In a stable pass each warp owns one
// contiguous segment of the current order, and a pixel's new place is its (digit, warp)-major
// exclusive offset plus its position among equal digits earlier in the segment (warp match).
// Histograms are laid out warp-major with a pad word so that the leaders of one warp never share
// a bank. Where the keys live in global scratch (large footprints), each stable pass first copies
// its digit of every box position into a shared byte array (`dig`, coalesced reads of the keys),
// so that the passes look digits up in shared memory instead of gathering keys from L2 one by one.
// The sorted positions end in list B, which is then rewritten in place as the omnigram.
template <int DT, int W, bool C16, bool STAGED, int KS>
__device__ void ordinal_transform_radix(const Plan& P, const int* frow, uint32_t* keys, typename Loc<W>::Pos* bufA,
                                        typename Loc<W>::Pos* bufB, uint32_t* hist, uint32_t* wsum, uint32_t* bins,
                                        uint8_t* dig, const Footprint<DT>& fp, const Grp& G) {
    using Pos = typename Loc<W>::Pos;
    const int tid = G.tid, lane = G.lane, warp = G.warp;
    const int nthreads = P.threads, nwarps = P.nwarps, S = P.S;
    constexpr int HS = kSortBins + 1;
    const int area = S * P.SH;
    uint32_t* hw = hist + warp * HS;
    // Exclusive scan of the per-warp digit counts in (digit, warp) order, in place: each thread
    // takes 8 consecutive counters (256 * nwarps counters over 32 * nwarps threads).
    auto scan_counts = [&]() {
        const int d0 = tid * 8 / nwarps, w0 = tid * 8 - d0 * nwarps;
        uint32_t c[8];
        uint32_t local = 0;
#pragma unroll
        for (int j = 0, d = d0, wq = w0; j < 8; ++j) {
            c[j] = hist[wq * HS + d];
            local += c[j];
            if (++wq == nwarps) wq = 0, ++d;
        }
        uint32_t incl = local;
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t t = __shfl_up_sync(kFull, incl, o);
            if (lane >= o) incl += t;
        }
        if (lane == 31) wsum[warp] = incl;
        G.sync();
        if (warp == 0) {
            const uint32_t x = lane < nwarps ? wsum[lane] : 0;
            uint32_t y = x;
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t t = __shfl_up_sync(kFull, y, o);
                if (lane >= o) y += t;
            }
            wsum[lane] = y - x;
        }
        G.sync();
        uint32_t run = incl - local + wsum[warp];
#pragma unroll
        for (int j = 0, d = d0, wq = w0; j < 8; ++j) {
            hist[wq * HS + d] = run;
            run += c[j];
            if (++wq == nwarps) wq = 0, ++d;
        }
    };
    // box position i lies in the footprint (Fig. 10)
    auto inside = [&](int i) {
        const int v = (int)__umulhi((unsigned)i, P.div_magic);
        const int fr = frow[v];
        const int u = i - v * S;
        return u >= span_lo(fr) && u <= span_hi(fr);
    };
    // Pass 0, fused with the footprint load: every thread takes box positions tid, tid +
    // nthreads, ... (coalesced rows), four loads in flight, and counts the low digit (8 bits in its
    // warp's histogram, or 16 bits in the block's packed bins); equal digits may then land in any
    // order (returned atomics), since the later passes are stable.
    // Footprints of more than 65535 pixels would overflow the packed 16-bit counters: the 16-bit
    // pass then counts in two rounds over the digit range (top bit 0, then 1), each with 32768
    // 32-bit bins in the same 128 KiB (the first round's histogram fused with the load).
    const bool two = C16 && P.N > 65535;
    if constexpr (C16) {
        for (int i = tid * 4; i < 32768; i += nthreads * 4)
            *reinterpret_cast<uint4*>(bins + i) = make_uint4(0, 0, 0, 0);
        G.sync();
    } else {
        for (int d = lane; d < kSortBins; d += 32) hw[d] = 0;
        __syncwarp();
    }
    for (int i0 = tid; i0 < area; i0 += 4 * nthreads) {
        uint32_t key[4];
        bool in[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const int i = i0 + k * nthreads;
            in[k] = i < area && inside(i);
            key[k] = 0;
            if (in[k]) {
                const int v = (int)__umulhi((unsigned)i, P.div_magic);
                key[k] = fp.template key<STAGED>(i - v * S, v);
            }
        }
#pragma unroll
        for (int k = 0; k < 4; ++k)
            if (in[k]) {
                keys[i0 + k * nthreads] = key[k];
                if constexpr (C16) {
                    const uint32_t d = key[k] & 0xffffu;
                    if (!two)
                        atomicAdd(&bins[d >> 1], 1u << ((d & 1u) << 4));
                    else if ((d >> 15) == 0)
                        atomicAdd(&bins[d], 1u);
                } else {
                    atomicAdd(&hw[key[k] & 0xff], 1u);
                }
            }
    }
    G.sync();
    // the first pass's result goes to the list the stable passes start from: with C16 two stable
    // passes follow (B -> A -> B), otherwise an odd number (A -> B -> ... -> B)
    Pos* first = C16 ? bufB : bufA;
    // The keys may live in global scratch: every loop below loads kG of them (all in flight)
    // before it uses the first.
    constexpr int kG = 4;
    if constexpr (C16) {
        if (two) {
            uint32_t base = 0;
            for (int h = 0; h < 2; ++h) {
                if (h == 1) {  // the second round's histogram (the keys, in order, from scratch)
                    for (int i = tid * 4; i < 32768; i += nthreads * 4)
                        *reinterpret_cast<uint4*>(bins + i) = make_uint4(0, 0, 0, 0);
                    G.sync();
                    for (int i0 = tid; i0 < area; i0 += kG * nthreads) {
                        uint32_t key[kG];
                        bool in[kG];
#pragma unroll
                        for (int k = 0; k < kG; ++k) {
                            const int i = i0 + k * nthreads;
                            in[k] = i < area && inside(i);
                            key[k] = in[k] ? keys[i] & 0xffffu : 0u;
                        }
#pragma unroll
                        for (int k = 0; k < kG; ++k)
                            if (in[k] && (key[k] >> 15) == 1u) atomicAdd(&bins[key[k] & 0x7fffu], 1u);
                    }
                    G.sync();
                }
                base += scan_bins32(bins, wsum, base, P, G);
                for (int i0 = tid; i0 < area; i0 += kG * nthreads) {
                    uint32_t key[kG];
                    bool in[kG];
#pragma unroll
                    for (int k = 0; k < kG; ++k) {
                        const int i = i0 + k * nthreads;
                        in[k] = i < area && inside(i);
                        key[k] = in[k] ? keys[i] & 0xffffu : 0u;
                    }
#pragma unroll
                    for (int k = 0; k < kG; ++k)
                        if (in[k] && (key[k] >> 15) == (uint32_t)h)
                            first[atomicAdd(&bins[key[k] & 0x7fffu], 1u)] = (Pos)(i0 + k * nthreads);
                }
                G.sync();
            }
        } else {
            scan_bins16(bins, wsum, P, G);
        }
    } else {
        scan_counts();
        G.sync();
    }
    for (int i0 = tid; i0 < area && !two; i0 += kG * nthreads) {
        uint32_t key[kG];
        bool in[kG];
#pragma unroll
        for (int k = 0; k < kG; ++k) {
            const int i = i0 + k * nthreads;
            in[k] = i < area && inside(i);
            key[k] = in[k] ? keys[i] : 0u;
        }
#pragma unroll
        for (int k = 0; k < kG; ++k)
            if (in[k]) {
                const int i = i0 + k * nthreads;
                if constexpr (C16) {
                    const uint32_t d = key[k] & 0xffffu, sh = (d & 1u) << 4;
                    first[(atomicAdd(&bins[d >> 1], 1u << sh) >> sh) & 0xffffu] = (Pos)i;
                } else {
                    first[atomicAdd(&hw[key[k] & 0xff], 1u)] = (Pos)i;
                }
            }
    }
    G.sync();
    // stable passes over the current order: each warp owns one contiguous segment; a pixel's
    // new place is its (digit, warp)-major exclusive offset plus its position among equal
    // digits earlier in the segment (warp match)
    const Pos* src = first;
    Pos* dst = C16 ? bufA : bufB;
    constexpr int kBits0 = C16 ? 16 : 8;                       // key bits the first pass sorted
    constexpr int kPasses = (DT == FIM_F32 ? 32 - kBits0 : 16 - kBits0) / 8;  // stable 8-bit passes
    static_assert(kPasses % 2 == (C16 ? 0 : 1), "the sorted positions must end in list B");
    const int N = P.N;
    const int seg = ((N + nwarps - 1) / nwarps + 31) & ~31;
    const int s0 = min(N, warp * seg), s1 = min(N, s0 + seg);
    // the stable passes, compiled for digits looked up in `dig` and for digits taken from the keys
    auto stable_pass = [&](auto use_dig, auto last, int pass) {
        constexpr bool kDig = decltype(use_dig)::value, kLast = decltype(last)::value;
        {
            const int shift = kBits0 + 8 * pass;
            if constexpr (kDig) {
                const int nq = (area + 3) >> 2;  // keys of 4 consecutive box positions per load
                const uint4* k4 = reinterpret_cast<const uint4*>(keys);
                uint32_t* d4 = reinterpret_cast<uint32_t*>(dig);
                for (int j = tid; j < nq; j += nthreads) {
                    const uint4 q = k4[j];
                    d4[j] = ((q.x >> shift) & 0xffu) | (((q.y >> shift) & 0xffu) << 8) |
                            (((q.z >> shift) & 0xffu) << 16) | ((q.w >> shift) << 24);
                }
                G.sync();
            }
            auto digit = [&](int pos) -> int {
                if constexpr (kDig) return dig[pos];
                else return (int)(keys[pos] >> shift) & 0xff;
            };
            for (int d = lane; d < kSortBins; d += 32) hw[d] = 0;
            __syncwarp();
            for (int i0 = s0 + lane; i0 < s1; i0 += 32 * kG) {  // counts do not depend on the order
                int dk[kG];
#pragma unroll
                for (int k = 0; k < kG; ++k) {
                    const int i = i0 + 32 * k;
                    dk[k] = i < s1 ? digit(src[i]) : 0;
                }
#pragma unroll
                for (int k = 0; k < kG; ++k)
                    if (i0 + 32 * k < s1) atomicAdd(&hw[dk[k]], 1u);
            }
            G.sync();
            scan_counts();
            G.sync();
            for (int b0 = s0; b0 < s1; b0 += 32 * kG) {
                int pos[kG], d[kG];
#pragma unroll
                for (int k = 0; k < kG; ++k) {
                    const int i = b0 + 32 * k + lane;
                    pos[k] = i < s1 ? (int)src[i] : -1;
                }
#pragma unroll
                for (int k = 0; k < kG; ++k)
                    d[k] = pos[k] >= 0 ? digit(pos[k]) : kSortBins + lane;
                // batches in segment order, so equal digits keep their order
#pragma unroll
                for (int k = 0; k < kG; ++k) {
                    if (b0 + 32 * k >= s1) break;
                    const bool valid = pos[k] >= 0;
                    const uint32_t peers = kLast ? __match_any_sync(kFull, d[k]) : same_byte(d[k], valid);
                    uint32_t base = 0;
                    if (valid) base = hw[d[k]];
                    __syncwarp();
                    if (valid) {
                        const int earlier = __popc(peers & lanemask_lt());
                        dst[base + earlier] = (Pos)pos[k];
                        if (earlier == 0) hw[d[k]] = base + __popc(peers);
                    }
                    __syncwarp();
                }
            }
            G.sync();
            src = dst;
            dst = (dst == bufA) ? bufB : bufA;
        }
    };
    // A float key's top byte takes few values, which a match finds quickly; in the small CTAs the votes'
    // code costs more instruction fetches than they save (f32 4096^2 r = 100 sort 543k -> 486k cycles
    // per tile; u16 r = 8 1033 -> 1165 us with them).
    constexpr int kSpread = KS != 8 ? 0 : (DT == FIM_F32 ? kPasses - 1 : kPasses);
    auto stable_passes = [&](auto use_dig) {
        for (int pass = 0; pass < kSpread; ++pass) stable_pass(use_dig, std::false_type{}, pass);
        if constexpr (kSpread < kPasses)
            for (int pass = kSpread; pass < kPasses; ++pass) stable_pass(use_dig, std::true_type{}, pass);
    };
    if constexpr (DT == FIM_F32) {  // only float plans place digits (one stable pass otherwise)
        if (dig != nullptr)
            stable_passes(std::true_type{});
        else
            stable_passes(std::false_type{});
    } else {
        stable_passes(std::false_type{});
    }
    // the sorted positions are in B; rewrite them in place as entries
    typename Loc<W>::E* om = reinterpret_cast<typename Loc<W>::E*>(bufB);
    for (int v = tid; v < N; v += nthreads) {
        const int pos = (int)bufB[v];
        const int y = (int)__umulhi((unsigned)pos, P.div_magic);
        om[v] = Loc<W>::pack(pos - y * S, y, P.cx0, P.cy0);
    }
}

// ---- learned rank bracket (seed windows) ---------------------------------------------------

__device__ __forceinline__ float bf16_to_f32(uint16_t b) { return __uint_as_float((uint32_t)b << 16); }

// Features of the seed window centred at box position (cu, cv): the tile's normalised value
// quantiles (already in q[0..31]) and the ranks / N of the 3x3 pixels around the centre
// (the centre's own rank where a neighbour lies outside the footprint, 0 where the centre does: a
// kernel may lie off its centre).
__device__ __forceinline__ void seed_features(const uint16_t* ord, int SP, const int* frow, int SH, int N, int cu,
                                              int cv, const float* q, float* fa, float* fb) {
    const int lane = threadIdx.x & 31;
    *fa = q[lane];
    float nb = 0.f;
    if (lane < kNeigh) {
        int u = cu + lane % 3 - 1, v = cv + lane / 3 - 1;
        bool in = v >= 0 && v < SH;
        if (in) {
            const int fr = frow[v];
            in = u >= span_lo(fr) && u <= span_hi(fr);
        }
        if (!in) {
            u = cu;
            v = cv;
            in = v >= 0 && v < SH;
            if (in) {
                const int fr = frow[v];
                in = u >= span_lo(fr) && u <= span_hi(fr);
            }
        }
        nb = in ? (float)ord[v * SP + u] / (float)N : 0.f;
    }
    *fb = nb;
}

// Visits the ranks of every pixel of a window (row i of the kernel at ctr + (ymin + i) * SP,
// ctr being the window centre's ordinal-image position shifted by ymin rows). Lane l takes
// kernel rows l, l+32, ... and walks each from a lane-dependent column, so the 32 pixels
// visited at once lie far apart (their ranks rarely share a histogram bin). Four ranks are
// loaded before they are handed to `f`, so the loads of a group overlap instead of each
// waiting behind the previous group's shared-memory atomics.
template <class Fn>
__device__ __forceinline__ void window_walk(const int* spans, int nrows, const uint16_t* ctr, int SP, Fn&& f) {
    const int lane = threadIdx.x & 31;
    for (int i = lane; i < nrows; i += 32) {
        const int sp = spans[i];
        const int width = span_hi(sp) - span_lo(sp) + 1;
        const uint16_t* row = ctr + i * SP + span_lo(sp);
        int x = (lane * 37) % width;
        int k = 0;
        for (; k + 4 <= width; k += 4) {
            int x1 = x + 1, x2 = x + 2, x3 = x + 3;
            if (x1 >= width) x1 -= width;
            if (x2 >= width) x2 -= width;
            if (x3 >= width) x3 -= width;
            const int r0 = row[x], r1 = row[x1], r2 = row[x2], r3 = row[x3];
            f(r0);
            f(r1);
            f(r2);
            f(r3);
            x = x3 + 1 == width ? 0 : x3 + 1;
        }
        for (; k < width; ++k) {
            f((int)row[x]);
            x = (x + 1 == width) ? 0 : x + 1;
        }
    }
}

// Target rank of output pixel (gx, gy) under a percentile map (Fig. 14), from the rank image
// the host computed before the launch. Pixels beyond the image (the ragged edge of a tile) take
// the nearest pixel's rank; their results are never stored.
__device__ __forceinline__ int map_rank(const Plan& P, int gx, int gy) {
    return __ldg(P.rank_map + (long long)min(gy, P.h - 1) * P.w + min(gx, P.w - 1));
}

// Seed histogram (kSeedBins bins of one warp): the bin holding window-rank `target` when
// `base` window members lie below bin 0. Returns the bin and, in *below, the members below it.
__device__ __forceinline__ int hist_pick(const uint32_t* hw, int base, int target, int* below) {
    const int lane = threadIdx.x & 31;
    constexpr int per = kSeedBins / 32;
    uint32_t local = 0;
    for (int j = 0; j < per; ++j) local += hw[lane * per + j];
    uint32_t incl = local;
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t tt = __shfl_up_sync(kFull, incl, o);
        if (lane >= o) incl += tt;
    }
    const int excl = base + (int)(incl - local);
    const bool mine = excl <= target && target < base + (int)incl;
    const uint32_t who = __ballot_sync(kFull, mine);
    int bin = 0, run = 0;
    if (mine) {
        run = excl;
        int j = 0;
        for (; j < per - 1; ++j) {
            const int c = (int)hw[lane * per + j];
            if (run + c > target) break;
            run += c;
        }
        bin = lane * per + j;
    }
    const int src = who ? __ffs(who) - 1 : 0;
    *below = __shfl_sync(kFull, run, src);
    return __shfl_sync(kFull, bin, src);
}

template <class T>
__device__ __forceinline__ T* place(unsigned char* smem, unsigned char* gslice, int loc) {
    return reinterpret_cast<T*>(loc >= 0 ? smem + loc : gslice + (-(long long)loc - 1));
}

// Fills the omnigram's last 64-byte block with sentinels no window contains.
template <int W>
__device__ __forceinline__ void pad_omnigram(typename Loc<W>::E* om, int N, int tid) {
    constexpr int kBlock = 64 / (int)sizeof(typename Loc<W>::E);
    const int pad = ((N + kBlock - 1) & ~(kBlock - 1)) - N;
    if (tid < pad) om[N + tid] = Loc<W>::kSentinel;
}

// Several radii from one transform: keeps, in order, the omnigram entries that lie in a smaller
// disk's footprint (`qfrow`: per box row, its columns lo | hi << 16; rows outside hold an empty
// span), and gives those pixels their new ranks in the ordinal image. The order of the kept
// entries is the sorted order restricted to the smaller footprint, i.e. that footprint's own
// ordinal transform, obtained in one pass with no sort. Each thread takes 4 consecutive entries
// of a 4 * group-size chunk; a block scan of the per-thread counts gives the new places. Every
// write goes to an index no larger than the entry's own, and all reads of a chunk precede its
// first barrier, so the compaction can run in place. Returns the number kept.
template <int W>
__device__ int compact_omnigram(typename Loc<W>::E* om, int N, const int* qfrow, uint16_t* ord, int SP, int cx0,
                                int cy0, uint32_t* wsum, const Grp& G, int nthreads, int nwarps) {
    using E = typename Loc<W>::E;
    const int tid = G.tid, lane = G.lane, warp = G.warp;
    int base = 0;
    for (int c0 = 0; c0 < N; c0 += 4 * nthreads) {
        E e[4];
        bool keep[4];
        int cnt = 0;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const int i = c0 + 4 * tid + k;
            keep[k] = false;
            e[k] = 0;
            if (i < N) {
                e[k] = om[i];
                const int u = Loc<W>::x(e[k]) + cx0, v = Loc<W>::y(e[k]) + cy0;
                const int fr = qfrow[v];
                keep[k] = u >= span_lo(fr) && u <= span_hi(fr);
            }
            cnt += keep[k];
        }
        int incl = cnt;
        for (int o = 1; o < 32; o <<= 1) {
            const int t = __shfl_up_sync(kFull, incl, o);
            if (lane >= o) incl += t;
        }
        if (lane == 31) wsum[warp] = (uint32_t)incl;
        G.sync();
        if (warp == 0) {
            const uint32_t x = lane < nwarps ? wsum[lane] : 0u;
            uint32_t y = x;
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t t = __shfl_up_sync(kFull, y, o);
                if (lane >= o) y += t;
            }
            wsum[lane] = y - x;         // exclusive per-warp offsets
            if (lane == 31) wsum[32] = y;  // the chunk's total
        }
        G.sync();
        int idx = base + (int)wsum[warp] + incl - cnt;
#pragma unroll
        for (int k = 0; k < 4; ++k)
            if (keep[k]) {
                om[idx] = e[k];
                ord[(Loc<W>::y(e[k]) + cy0) * SP + Loc<W>::x(e[k]) + cx0] = (uint16_t)idx;
                ++idx;
            }
        base += (int)wsum[32];
        G.sync();  // the offsets are read before the next chunk rewrites them
    }
    pad_omnigram<W>(om, base, tid);
    G.sync();
    return base;
}

// KS: the kernel set. 8: 1024-thread CTAs, and smaller ones that sort by codes (deeper unrolled
// slides, scans without a divergent branch, the sort by codes); 4: the other, smaller CTAs, whose
// several phases in flight share the instruction cache (short code); 0: extras and percentile maps
// of those.
// XT: 1 compiles the extras — the learned bracket, training-row output, seed statistics and
// several target ranks per launch — and 2 a target rank per output pixel (a percentile map).
// Each lives in kernels of its own: at the 64-register cap of 1024-thread CTAs their code
// changes how the compiler allocates the plain pipeline's registers, and the reverse.
// TMA: how interior footprints are copied into the staging region: 0 not at all; 1 the
// single-image kernels (mbarrier in the scan scratch, tensor map in the kernel parameter);
// 2 the batch kernels (`bar` and `tmap` given: a CTA-wide mbarrier and the job's tensor map in
// the plan array in global memory, since their plans are read from shared memory).
template <int DT, int SHAPE, int W, int OG, int KS = 0, int XT = 0, int TMA = 1>
__device__ __forceinline__ void process_tile(const Plan& P, int tile, unsigned char* gslice, const Grp& G,
                                             TmaState* tma = nullptr, uint64_t* bar = nullptr,
                                             const void* tmap = nullptr) {
    extern __shared__ __align__(128) unsigned char smem_base[];
    unsigned char* const smem = smem_base + G.shift;  // this group's partition (tables excluded)
    using V = typename Traits<DT>::T;
    using E = typename Loc<W>::E;
    // Plans that sort by codes run on these kernels only: the small CTAs of the others hold several
    // phases in flight at once, and its code would crowd theirs out of the instruction cache (u16
    // 4096^2 r = 16: 1289 -> 1392 us with it compiled in and not used).
    constexpr bool kCodes = DT != FIM_U8 && W == 0 && KS == 8;
    const int tid = G.tid;
    const int lane = G.lane;
    const int warp = G.warp;
    const int nthreads = P.threads;
    const int nwarps = P.nwarps;
    const int SP = P.SP, N = P.N, TX = P.Tx, TY = P.Ty;
    const int tx0 = (tile % P.tiles_x) * TX;
    const int ty0 = (tile / P.tiles_x) * TY;
    const int gx0 = tx0 + P.xmin;  // global coordinates of bounding-box pixel (0, 0)
    const int gy0 = ty0 + P.ymin;
    const int cx0 = P.cx0, cy0 = P.cy0, xmin = P.xmin, ymin = P.ymin, hist_shift = P.hist_shift;
    // The ordinal image and the medians hold ranks minus rank_base, clamped to 16 bits: every
    // pivot lies in the tile's feasible median ranks (Fig. 10), which then compare exactly, so
    // footprints beyond 65535 pixels keep a 16-bit ordinal image and most others a signed one.
    const int rb = P.rank_base, rel_max = P.rel_max;

    const int4* vtab = reinterpret_cast<const int4*>(smem_base + P.off_vtab);
    const int2* htab = reinterpret_cast<const int2*>(smem_base + P.off_htab);
    const int* spans = reinterpret_cast<const int*>(smem_base + P.off_spans);
    const int* frow = reinterpret_cast<const int*>(smem_base + P.off_frow);
    uint32_t* misc = reinterpret_cast<uint32_t*>(smem + P.off_misc);
    // The omnigram's home is fixed per instantiation (OG), so the compiler keeps shared-memory
    // accesses as such; everything else of the solve always lives in shared memory.
    E* om = OG ? reinterpret_cast<E*>(gslice + (-(long long)P.loc_om - 1)) : reinterpret_cast<E*>(smem + P.loc_om);
    uint16_t* ord = reinterpret_cast<uint16_t*>(smem + P.loc_ord);
    uint16_t* med = reinterpret_cast<uint16_t*>(smem + P.loc_med);
    uint32_t* shist = reinterpret_cast<uint32_t*>(smem + P.loc_shist);
    uint32_t* tie = reinterpret_cast<uint32_t*>(smem + P.loc_tie);

    // ---- 1. ordinal transform ------------------------------------------------------------------
    stamp(P, tile, 1, G);
    // The footprint: for an interior tile with a staging region, one thread has the tensor memory
    // accelerator copy the whole box (from the 16-byte boundary at or left of its first column)
    // into shared memory, and every thread waits on the mbarrier (bounded: after a timeout the
    // tile, and the CTA's later tiles, read the image instead).
    Footprint<DT> fp{nullptr, 0, 0, Img(P), gx0, gy0};
    if (TMA != 0 && tma != nullptr && P.use_tma && !tma->off) {
        constexpr int A = 16 / (int)sizeof(V);  // elements per 16 bytes
        const int x0 = gx0 & ~(A - 1);
        if (x0 >= 0 && gy0 >= 0 && x0 + P.stage_bw <= P.w && gy0 + P.SH <= P.h) {
            unsigned char* st = smem + P.loc_stage;
            st += (128u - (smem_addr(st) & 127u)) & 127u;  // the region has 128 bytes of slack
            if constexpr (TMA == 1) {  // the single-image kernel: barrier in the scan scratch
                bar = reinterpret_cast<uint64_t*>(misc + 34);
                tmap = &P.tmap;
            }
            if (tid == 0)
                tma_load_box(tmap, st, bar, x0, gy0, (uint32_t)(P.stage_bw * P.SH * (int)sizeof(V)));
            const bool ok = mbar_wait(bar, tma->parity) || mbar_wait(bar, tma->parity);
            tma->parity ^= 1u;
            if (ok) {
                fp.stage = st;
                fp.pitch = P.stage_bw * (int)sizeof(V);
                fp.off = gx0 - x0;
            } else {
                tma->off = 1;
                set_status(FIM_ERR_TIMEOUT);
            }
        }
    }
    // The sort, compiled for the staged box and for the image (one branch per tile): by codes where the
    // plan has them and the box lies inside the image; otherwise float data takes the radix sort, and
    // 16-bit data in small CTAs, where the counting sort's 65536 bins would keep other CTAs off the SM.
    auto sort = [&](auto staged) {
        constexpr bool ST = decltype(staged)::value;
        if constexpr (kCodes) {
            if (P.codes > 0) {
                // (a box that leaves the image repeats its edge pixels many times: exact order)
                if (gx0 >= 0 && gy0 >= 0 && gx0 + P.S <= P.w && gy0 + P.SH <= P.h) {
                    if (ordinal_transform_codes<DT, W, ST>(P, frow, reinterpret_cast<uint32_t*>(smem + P.loc_codes),
                                                           tie, place<uint16_t>(smem, gslice, P.loc_cbuf), misc, om, fp, G))
                        return;
                    G.sync();
                }
                for (int i = tid; i < N / 32 + 2; i += nthreads) tie[i] = 0;
            }
        }
        if constexpr (DT == FIM_F32) {
            if (P.sort == kSortRadix16)
                ordinal_transform_radix<DT, W, true, ST, KS>(P, frow, place<uint32_t>(smem, gslice, P.loc_keys),
                                                         place<typename Loc<W>::Pos>(smem, gslice, P.loc_a),
                                                         place<typename Loc<W>::Pos>(smem, gslice, P.loc_b),
                                                         reinterpret_cast<uint32_t*>(smem + P.loc_hist), misc,
                                                         reinterpret_cast<uint32_t*>(smem + P.loc_bins),
                                                         P.loc_dig >= 0 ? smem + P.loc_dig : nullptr, fp, G);
            else
                ordinal_transform_radix<DT, W, false, ST, KS>(P, frow, place<uint32_t>(smem, gslice, P.loc_keys),
                                                          place<typename Loc<W>::Pos>(smem, gslice, P.loc_a),
                                                          place<typename Loc<W>::Pos>(smem, gslice, P.loc_b),
                                                          reinterpret_cast<uint32_t*>(smem + P.loc_hist), misc,
                                                          nullptr, P.loc_dig >= 0 ? smem + P.loc_dig : nullptr, fp,
                                                          G);
        } else if (DT == FIM_U16 && (KS == 4 || P.sort == kSortRadix)) {  // (fewer than 1024 threads: radix)
            ordinal_transform_radix<DT, W, false, ST, KS>(P, frow, place<uint32_t>(smem, gslice, P.loc_keys),
                                                      place<typename Loc<W>::Pos>(smem, gslice, P.loc_a),
                                                      place<typename Loc<W>::Pos>(smem, gslice, P.loc_b),
                                                      reinterpret_cast<uint32_t*>(smem + P.loc_hist), misc, nullptr,
                                                      P.loc_dig >= 0 ? smem + P.loc_dig : nullptr, fp, G);
        } else {
            ordinal_transform_count<DT, W, ST>(P, frow, reinterpret_cast<uint32_t*>(smem + P.loc_bins), misc, om, fp,
                                               G);
        }
    };
    if constexpr (TMA != 0) {
        if (fp.stage != nullptr)
            sort(std::true_type{});
        else
            sort(std::false_type{});
    } else {
        sort(std::false_type{});
    }
    G.sync();

    // ---- 2. ordinal image I (Eq. 4) ------------------------------------------------------------
    stamp(P, tile, 2, G);
    if constexpr (OG) {  // omnigram in global scratch: four entries per thread in flight
        for (int v0 = tid; v0 < N; v0 += 4 * nthreads) {
            uint32_t e[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) e[k] = v0 + k * nthreads < N ? (uint32_t)om[v0 + k * nthreads] : 0u;
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const int v = v0 + k * nthreads;
                if (v < N)
                    ord[(Loc<W>::y(e[k]) + cy0) * SP + Loc<W>::x(e[k]) + cx0] = (uint16_t)clampi(v - rb, 0, rel_max);
            }
        }
    } else {
        for (int v = tid; v < N; v += nthreads) {
            const uint32_t e = om[v];
            ord[(Loc<W>::y(e) + cy0) * SP + Loc<W>::x(e) + cx0] = (uint16_t)clampi(v - rb, 0, rel_max);
        }
    }
    pad_omnigram<W>(om, N, tid);
    G.sync();

    Member<SHAPE, W> member;
    if constexpr (SHAPE == kShapeDisk) {
        member.r2 = P.r2;
    } else {
        member.test = reinterpret_cast<const uint32_t*>(smem_base + P.off_test);
        member.xmin = P.xmin;
        member.ymin = P.ymin;
        member.nrows = P.nrows;
    }
    // Extras kernels may take several target ranks (percentiles) of one window size: the
    // ordinal transform and the ordinal image above are built once and serve them all.
    const int nr = XT == 1 ? P.nranks : 1;
    // With a percentile map every output pixel has its own target rank. A slide's pivot is the
    // previous window's result, which has exactly that window's target below it, so the count
    // at the pivot after the slide is the previous target plus the change.
    const bool mapped = XT == 2 && P.rank_map != nullptr;
    int Nq = N;  // omnigram length for this target (several radii: the current disk's footprint)
    for (int q = 0; q < nr; ++q) {
        const int target = q == 0 ? P.rank : P.ranks[q];
        // the kernel of this target: the plan's own, or (several radii) the q-th disk's tables
        const int4* qvtab = vtab;
        const int2* qhtab = htab;
        const int* qspans = spans;
        int qn = P.n, qymin = ymin, qnrows = P.nrows, qunits = P.vunits;
        Member<SHAPE, W> qmember = member;
        if constexpr (XT == 1) {
            if (P.multi) {
                qvtab = reinterpret_cast<const int4*>(smem_base + P.q_vtab[q]);
                qhtab = reinterpret_cast<const int2*>(smem_base + P.q_htab[q]);
                qspans = reinterpret_cast<const int*>(smem_base + P.q_spans[q]);
                qn = P.q_n[q];
                qymin = P.q_ymin[q];
                qnrows = P.q_nrows[q];
                qunits = P.q_vunits[q];
                if constexpr (SHAPE == kShapeDisk) {
                    qmember.r2 = P.q_r2[q];
                } else {
                    qmember.ymin = qymin;
                    qmember.nrows = qnrows;
                }
                // targets come largest disk first: narrow the omnigram to this disk's footprint
                if (P.q_N[q] < Nq) {
                    const int kept = compact_omnigram<W>(om, Nq, reinterpret_cast<const int*>(smem_base + P.q_frow[q]),
                                                         ord, SP, cx0, cy0, misc, G, nthreads, nwarps);
                    if (kept != P.q_N[q]) set_status(FIM_ERR_INTERNAL);
                    Nq = P.q_N[q];
                }
            }
        }
        const int qhist_shift = XT == 1 && P.multi ? P.q_hshift[q] : hist_shift;
        const int BH = TY / P.RB;      // band height
        const int GW = TX / P.G;       // seed spacing within a seed row
        // feasible median ranks of any window of this tile (Fig. 10): [lof, hif]
        const int lof = target, hif = Nq - qn + target;

        // ---- 3. seeds: coarse histogram of I over the window, then ballot refine ----------------
        // (or, with a learned bracket, two exact counts at predicted ranks, then ballot refine)
        stamp(P, tile, 3, G);
        const bool learned = XT == 1 && P.model != nullptr;
        const bool sampling = XT == 1 && P.samples != nullptr;
        const bool counting = XT == 1 && P.stats != nullptr;
        float* quant = reinterpret_cast<float*>(misc);  // the sort's scan scratch is free from here on
        if (learned || sampling) {
            if (warp == 0) {  // normalised value quantiles of the footprint: C at N (j + 1/2) / 32
                const int q = min(Nq - 1, (int)(((long long)Nq * (2 * lane + 1)) / (2 * kQuantiles)));
                const uint32_t e = om[q];
                const float v = (float)load_px<DT>(Img(P), gx0 + Loc<W>::x(e) + cx0, gy0 + Loc<W>::y(e) + cy0);
                const float mid = __shfl_sync(kFull, v, kQuantiles / 2);
                const float spread = __shfl_sync(kFull, v, 7 * kQuantiles / 8) - __shfl_sync(kFull, v, kQuantiles / 8);
                const float z = (v - mid) / (spread > 0.f ? spread : 1.f);
                quant[lane] = fminf(fmaxf(z, -8.f), 8.f);
            }
            G.sync();
        }
        const int nseeds = P.RB * P.G;
        static_assert(kHidden <= kSeedBins, "the quantiles' layer-1 pre-activations fit one seed histogram");
        if (learned) {
            // Learned bracket (extension): the layer-1 contribution of the tile's quantiles is
            // computed once, block-wide; then each warp takes one seed at a time and, with no
            // further block barrier, evaluates the bracket MLP for it (lanes hold hidden units
            // lane and lane + 32, activations move by shuffles), counts the window's ranks below
            // the predicted median, and walks Omega 512 entries a step from there to the exact
            // median. It replaces the plain seeds' histogram or long walk.
            const uint16_t* wts =
                P.off_model >= 0 ? reinterpret_cast<const uint16_t*>(smem_base + P.off_model) : P.model;
            float* hbase = reinterpret_cast<float*>(shist);  // layer-1 pre-activation of the quantiles
            for (int j = tid; j < kHidden; j += nthreads) {
                float h = bf16_to_f32(wts[kOffB1 + j]);
                for (int i = 0; i < kQuantiles; ++i) h = fmaf(quant[i], bf16_to_f32(wts[kOffW1 + i * kHidden + j]), h);
                hbase[j] = h;
            }
            G.sync();
            for (int sd = warp; sd < nseeds; sd += nwarps) {
                const int band = sd / P.G, g = sd % P.G;
                const int s = g * GW + GW / 2, t = band * BH + BH / 2;
                const int cu = s - xmin, cv = t - ymin;
                float fa, fb;
                seed_features(ord, SP, frow, P.SH, Nq, cu, cv, quant, &fa, &fb);
                float a0 = hbase[lane], a1 = hbase[lane + 32];
#pragma unroll
                for (int i = 0; i < kNeigh; ++i) {
                    const float x = __shfl_sync(kFull, fb, i);
                    a0 = fmaf(x, bf16_to_f32(wts[kOffW1 + (kQuantiles + i) * kHidden + lane]), a0);
                    a1 = fmaf(x, bf16_to_f32(wts[kOffW1 + (kQuantiles + i) * kHidden + lane + 32]), a1);
                }
                a0 = fmaxf(a0, 0.f);
                a1 = fmaxf(a1, 0.f);
                float b0 = bf16_to_f32(wts[kOffB2 + lane]), b1 = bf16_to_f32(wts[kOffB2 + lane + 32]);
#pragma unroll 8
                for (int k = 0; k < kHidden; ++k) {
                    const float x = __shfl_sync(kFull, k < 32 ? a0 : a1, k & 31);
                    b0 = fmaf(x, bf16_to_f32(wts[kOffW2 + k * kHidden + lane]), b0);
                    b1 = fmaf(x, bf16_to_f32(wts[kOffW2 + k * kHidden + lane + 32]), b1);
                }
                b0 = fmaxf(b0, 0.f);
                b1 = fmaxf(b1, 0.f);
                float o0 = bf16_to_f32(wts[kOffW3 + lane * 2]) * b0 + bf16_to_f32(wts[kOffW3 + (lane + 32) * 2]) * b1;
                float o1 = bf16_to_f32(wts[kOffW3 + lane * 2 + 1]) * b0 + bf16_to_f32(wts[kOffW3 + (lane + 32) * 2 + 1]) * b1;
                for (int o = 16; o > 0; o >>= 1) {
                    o0 += __shfl_xor_sync(kFull, o0, o);
                    o1 += __shfl_xor_sync(kFull, o1, o);
                }
                o0 += bf16_to_f32(wts[kOffB3]);
                o1 += bf16_to_f32(wts[kOffB3 + 1]);
                const float sig = __expf(fminf(fmaxf(o1, -8.f), 2.f)) * P.bracket_z;
                const float span = (float)(hif - lof);
                const int lo = clampi(__float2int_rn(lof + (o0 - sig) * span), 0, Nq - 1);
                const int hi = clampi(__float2int_rn(lof + (o0 + sig) * span), lo, Nq - 1);
                // (pivots stay in the feasible ranks, where the ordinal image's ranks compare exactly)
                const int pivot = clampi(clampi(__float2int_rn(lof + o0 * span), lo, hi), lof, hif);
                // The count at the predicted median is exact, so the walk from it finds the exact
                // median wherever it lies: on a miss it simply walks past the bracket, over the
                // full range if need be. The bracket ends only classify the outcome.
                const int below = window_rows_below(qspans, qnrows, ord + (cv + qymin) * SP + cu, SP, pivot - rb);
                const int m = wide_select<SHAPE, W>(om, Nq, pivot, below, target, cu - cx0, cv - cy0, qmember);
                if (m < 0) set_status(FIM_ERR_INTERNAL);
                if (lane == 0) med[band * TX + s] = (uint16_t)(max(m, 0) - rb);
                if (counting && lane == 0) {
                    const int kind = m < lo ? 2 : (m > hi ? 3 : 1);
                    atomicAdd(P.stats + 0, 1ull);
                    atomicAdd(P.stats + kind, 1ull);
                    atomicAdd(P.stats + 4, (unsigned long long)abs(max(m, 0) - pivot));
                }
            }
        } else {
            for (int sd = warp; sd < nseeds; sd += nwarps) {
                const int band = sd / P.G, g = sd % P.G;
                const int s = g * GW + GW / 2, t = band * BH + BH / 2;  // tile-local output pixel
                const int cu = s - xmin, cv = t - ymin;                 // window centre in the box
                float fa = 0.f, fb = 0.f;
                if (sampling) seed_features(ord, SP, frow, P.SH, Nq, cu, cv, quant, &fa, &fb);
                const int ts = mapped ? map_rank(P, tx0 + s, ty0 + t) : target;
                int pivot = 0, below = 0, m;
                if (P.seed_mode == kSeedHistogram) {
                    // a coarse histogram of the window's ranks (one per concurrently solved seed),
                    // scanned to the bin of the target, then a ballot scan of Omega from that bin
                    uint32_t* hw = shist + (nwarps >= nseeds ? sd : warp) * kSeedBins;
                    for (int j = lane; j < kSeedBins; j += 32) hw[j] = 0;
                    __syncwarp();
                    window_walk(qspans, qnrows, ord + (cv + qymin) * SP + cu, SP,
                                [&](int r) { atomicAdd(&hw[r >> qhist_shift], 1u); });
                    __syncwarp();
                    pivot = hist_pick(hw, 0, ts, &below) << qhist_shift;
                    // bin 0 also counts the members below the image's lowest rank
                    if (pivot > 0) pivot += rb;
                    m = warp_select<SHAPE, W>(om, Nq, pivot, below, ts, cu - cx0, cv - cy0, qmember);
                } else {
                    if (P.seed_mode == kSeedWalk) {
                        // walk Omega from whichever end is known exactly: nothing lies below
                        // rank 0, and all n members lie below rank N
                        if (2 * ts >= qn) {
                            pivot = Nq;
                            below = qn;
                        }
                    } else {
                        // count the window below the middle of the tile's feasible ranks, walk from there
                        pivot = (lof + hif) >> 1;
                        below = window_rows_below(qspans, qnrows, ord + (cv + qymin) * SP + cu, SP, pivot - rb);
                    }
                    m = wide_select<SHAPE, W>(om, Nq, pivot, below, ts, cu - cx0, cv - cy0, qmember);
                }
                if (m < 0) set_status(FIM_ERR_INTERNAL);
                if (lane == 0) med[band * TX + s] = (uint16_t)(max(m, 0) - rb);
                if (sampling) {  // training row: features and the exact median's place in [lof, hif]
                    unsigned int row = 0;
                    if (lane == 0) row = atomicAdd(P.sample_count, 1u);
                    row = __shfl_sync(kFull, row, 0);
                    if ((int)row < P.sample_cap) {
                        float* dst = P.samples + (size_t)row * (kFeatures + 1);
                        dst[lane] = fa;
                        if (lane < kNeigh) dst[kQuantiles + lane] = fb;
                        if (lane == 0) dst[kFeatures] = hif > lof ? (float)(max(m, 0) - lof) / (float)(hif - lof) : 0.5f;
                    }
                }
                if (counting && lane == 0) {
                    atomicAdd(P.stats + 0, 1ull);
                    atomicAdd(P.stats + 4, (unsigned long long)abs(max(m, 0) - pivot));
                }
                __syncwarp();
            }
        }
        G.sync();

        // ---- 4. seed rows: horizontal slides, lanes split the kernel rows ----------------------
        stamp(P, tile, 4, G);
        for (int job = warp; job < 2 * P.RB * P.G; job += nwarps) {
            const int sd = job >> 1, right = job & 1;
            const int band = sd / P.G, g = sd % P.G;
            int s = g * GW + GW / 2;
            const int t = band * BH + BH / 2;
            const int steps = right ? (GW - GW / 2 - 1) : (GW / 2);
            int cu = s - xmin;
            const int cv = t - ymin;
            int p = med[band * TX + s] + rb;
            constexpr int kRowsPerLane = (kMaxExtent + 31) / 32;
            int eo[kRowsPerLane], lo[kRowsPerLane];  // this lane's rows: entering / leaving offsets
    #pragma unroll
            for (int q = 0; q < kRowsPerLane; ++q) {
                const int i = lane + 32 * q;
                // rows beyond the kernel compare a pixel of the window with itself: no change (not the
                // centre, which lies outside the footprint, and may lie outside shared memory, where
                // the kernel is off centre)
                eo[q] = lo[q] = qhtab[0].x;
                if (i < qnrows) {
                    const int2 o = qhtab[i];
                    eo[q] = right ? o.y : o.x - 1;
                    lo[q] = right ? o.x : o.y - 1;
                }
            }
            for (int k = 0; k < steps; ++k) {
                const uint16_t* ctr = ord + cv * SP + cu;
                const int pr = p - rb;  // the pivot among the ordinal image's ranks
                int d = 0;
    #pragma unroll
                for (int q = 0; q < kRowsPerLane; ++q)
                    if (32 * q < qnrows) d += (int)(ctr[eo[q]] < pr) - (int)(ctr[lo[q]] < pr);
                d = __reduce_add_sync(kFull, d);
                // targets of the pivot's window and of the next one (re-read: no extra live state)
                const int tp = mapped ? map_rank(P, tx0 + s, ty0 + t) : target;
                cu += right ? 1 : -1;
                s += right ? 1 : -1;
                const int tn = mapped ? map_rank(P, tx0 + s, ty0 + t) : target;
                const int m = warp_select<SHAPE, W>(om, Nq, p, tp + d, tn, cu - cx0, cv - cy0, qmember);
                if (m < 0) set_status(FIM_ERR_INTERNAL);
                p = max(m, 0);
                if (lane == 0) med[band * TX + s] = (uint16_t)(p - rb);
            }
        }
        G.sync();

        // ---- 5. vertical sweeps: thread per window column, per-thread refinement ----------------
        // ---- 6. output, fused: out = C[m], the input value at Omega[m] --------------------------
        // Each sweep thread writes the pixels it solves (the downward threads also the seed row's
        // pixel they start from). The gather of a pixel's value is issued right after its solve
        // and its store waits for the next step, so the L2 latency of the scattered gathers hides
        // behind the next slide instead of queueing at the end of the tile.
        stamp(P, tile, 5, G);
        if (warp < P.vthreads / 32) {
            const int groups = TX / 32;
            const int cg = warp % groups;
            const int rest = warp / groups;
            const int band = rest % P.RB;
            const int down = rest / P.RB;  // 0: up, 1: down
            const int s = cg * 32 + lane;
            int t = band * BH + BH / 2;
            const int steps = down ? (BH - BH / 2 - 1) : (BH / 2);
            const int cu = s - xmin;
            int cv = t - ymin;
            int p = med[band * TX + s] + rb;
            const Img im(P);
            char* const out = static_cast<char*>(q == 0 ? P.out : P.outs[q]);
            const int gx = tx0 + s;
            V pval = V(0);       // value gathered for the last solved pixel, not yet stored
            V* pdst = nullptr;   // where it goes (null: outside the image, or nothing pending)
            auto gather = [&](int m, int tt, uint32_t members) {
                if constexpr (kCodes) {
                    if (P.codes > 0) {  // (cv is the window's row)
                        WordTest<SHAPE, W> wt;
                        wt.init(qmember, cu - cx0, cv - cy0);
                        // (only boxes inside the image have ties: no clamps)
                        const char* mid = im.in + (long long)(gy0 + cy0) * im.pitch + (long long)(gx0 + cx0) * (int)sizeof(V);
                        m = resolve_tie(om, tie, m, members, wt, [&](uint32_t e) {
                            return Traits<DT>::key(__ldg(
                                reinterpret_cast<const V*>(mid + (long long)Loc<W>::y(e) * im.pitch) + Loc<W>::x(e)));
                        });
                    }
                }
                const uint32_t e = om[m];
                pval = load_px<DT>(im, gx0 + Loc<W>::x(e) + cx0, gy0 + Loc<W>::y(e) + cy0);
                const int gy = ty0 + tt;
                pdst = (gx < im.w && gy < im.h) ? reinterpret_cast<V*>(out + (long long)gy * im.pitch) + gx : nullptr;
            };
            if (down) {  // the seed row's pixel
                uint32_t members = 0;
                if constexpr (kCodes) {
                    WordTest<SHAPE, W> wt;
                    wt.init(qmember, cu - cx0, cv - cy0);
                    if (P.codes > 0) members = block_mask<SHAPE, W>(reinterpret_cast<const uint4*>(om), p >> 5, wt);
                }
                gather(p, t, members);
            }
            for (int k = 0; k < steps; ++k) {
                const unsigned char* ctr = reinterpret_cast<const unsigned char*>(ord + (down ? cv : cv - 1) * SP + cu);
                // slide unrolled deeper in the kernels of the 1024-thread tiles (KS = 8)
                const int d = KS != 8 && qunits <= kScalarUnits ? slide_scalar(ctr, qvtab, qunits, p - rb)
                              : P.s16 ? slide<true, KS == 8 ? 4 : 2>(ctr, qvtab, qunits, p - rb)
                                      : slide<false, 2>(ctr, qvtab, qunits, p - rb);
                const int tp = mapped ? map_rank(P, tx0 + s, ty0 + t) : target;
                cv += down ? 1 : -1;
                t += down ? 1 : -1;
                const int tn = mapped ? map_rank(P, tx0 + s, ty0 + t) : target;
                uint32_t members = 0;
                const int m = lane_select<SHAPE, W, KS, SHAPE == kShapeDisk && OG == 0 && KS == 8>(om, Nq, p, tp + (down ? d : -d), tn, cu - cx0, cv - cy0, qmember,
                                                    &members);
                if (m < 0) set_status(FIM_ERR_INTERNAL);
                p = max(m, 0);
                if (pdst) *pdst = pval;  // the previous pixel's value has arrived by now
                gather(p, t, members);
            }
            if (pdst) *pdst = pval;
        }
        stamp(P, tile, 6, G);  // the first group thread's own sweep is done (output is fused into it)
        G.sync();
        stamp(P, tile, 7, G);
    }
}

__device__ __forceinline__ void load_tables(const Plan& P) {
    extern __shared__ __align__(128) unsigned char smem[];
    const int tid = threadIdx.x, nt = blockDim.x;
    int2* vtab = reinterpret_cast<int2*>(smem + P.off_vtab);
    const int nvtab = 4 * P.vunits;
    int2* htab = reinterpret_cast<int2*>(smem + P.off_htab);
    int* spans = reinterpret_cast<int*>(smem + P.off_spans);
    int* frow = reinterpret_cast<int*>(smem + P.off_frow);
    for (int i = tid; i < nvtab; i += nt) vtab[i] = make_int2(P.vtab[2 * i], P.vtab[2 * i + 1]);
    for (int i = tid; i < P.nrows; i += nt) {
        htab[i] = make_int2(P.htab[2 * i], P.htab[2 * i + 1]);
        spans[i] = P.spans[i];
    }
    for (int i = tid; i < P.SH; i += nt) frow[i] = P.frow[i];
    if (P.off_test >= 0) {  // the span test's words, kSpanCopies of each row and of the empty one
        uint32_t* test = reinterpret_cast<uint32_t*>(smem + P.off_test);
        for (int i = tid; i < (P.nrows + 1) * kSpanCopies; i += nt) {
            const int r = i / kSpanCopies;
            uint32_t t = 0x4000u << 16;
            if (r < P.nrows)
                t = (uint32_t)(0x8000 - (span_lo(P.spans[r]) - P.xmin + 256)) << 16 |
                    (uint32_t)(0x7fff - (span_hi(P.spans[r]) - P.xmin + 256));
            test[i] = t;
        }
    }
    if (P.xtab != nullptr) {
        int* xt = reinterpret_cast<int*>(smem + P.off_xtab);
        for (int i = tid; i < P.xtab_words; i += nt) xt[i] = P.xtab[i];
    }
    if (P.off_model >= 0 && P.model != nullptr) {  // kMlpParams is even: copy 32-bit pairs
        const uint32_t* src = reinterpret_cast<const uint32_t*>(P.model);
        uint32_t* dst = reinterpret_cast<uint32_t*>(smem + P.off_model);
        for (int i = tid; i < kMlpParams / 2; i += nt) dst[i] = src[i];
    }
}

}  // namespace
}  // namespace fim
