// Pieces shared by the attention kernels (one CTA per SM, and one CTA pair per two SMs): launch parameters, the walk over
// the key tiles an item visits, the per-tile keep bitmaps of the Focus mask (paper Appendix D, first equation), the order
// in which items are handed out.
#pragma once

#include <cuda_fp16.h>

#include "common.cuh"
#include "sm100_ptx.cuh"

namespace focus {

using namespace ptx;

constexpr float LOG2E = 1.4426950408889634f;
constexpr float LN2 = 0.6931471805599453f;
constexpr float RESCALE_THRESHOLD = 8.0f;   // log2 units: the stale maximum may lag by a factor of 256
// Of every 8 consecutive probabilities, this many take their exponential from a polynomial on the
// FMA/ALU pipes instead of the special-function unit, which would otherwise be as busy as the tensor pipe.
constexpr int EX2_POLY_PER_8 = 0;
// Registers per thread after the warps have split into roles (setmaxnreg): the load/MMA warpgroup
// gives most of its share to the softmax warpgroups.
constexpr int REGS_CONTROL = 88;
constexpr int REGS_SOFTMAX_2WG = 208;        // 128*88 + 256*208 = 64512 = the 384 * 168 of the launch

__device__ __forceinline__ float max3(float a, float b, float c) {
    float d;
    asm("max.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
    return d;
}
template <int N> __device__ __forceinline__ void reg_dec() { asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(N)); }
template <int N> __device__ __forceinline__ void reg_inc() { asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(N)); }

// 2^x for a pair of arguments in [-inf, 8] without the special-function unit: split x = n + f with
// n = round(x) (magic-number addition), evaluate a cubic for 2^f on [-0.5, 0.5] (relative error
// 7.5e-5, far below the bf16 rounding of the probabilities) and add n to the exponent field.
// Arguments below -126 (masked pairs arrive as -inf) give 2^-126, which vanishes in every sum.
__device__ __forceinline__ float2 ex2_poly2(float2 x) {
    constexpr float MAGIC = 12582912.f;      // 1.5 * 2^23
    x.x = fmaxf(x.x, -126.f);
    x.y = fmaxf(x.y, -126.f);
    const float2 t = __fadd2_rn(x, make_float2(MAGIC, MAGIC));
    const float2 n = __fadd2_rn(t, make_float2(-MAGIC, -MAGIC));
    const float2 f = __ffma2_rn(n, make_float2(-1.f, -1.f), x);
    float2 p = __ffma2_rn(make_float2(0.0551716648f, 0.0551716648f), f, make_float2(0.2426111251f, 0.2426111251f));
    p = __ffma2_rn(p, f, make_float2(0.6932609677f, 0.6932609677f));
    p = __ffma2_rn(p, f, make_float2(0.9999280572f, 0.9999280572f));
    float2 r;
    r.x = __int_as_float(__float_as_int(p.x) + (__float_as_int(t.x) << 23));
    r.y = __int_as_float(__float_as_int(p.y) + (__float_as_int(t.y) << 23));
    return r;
}

// Division of 0 <= n < 2^31 by d >= 1 as a multiplication: q = n (2^(31 + l) / d + 1) / 2^(31 + l) with 2^l >= d (Granlund and
// Montgomery, Division by Invariant Integers using Multiplication, 1994).  (The compiler's own, for a divisor it does not know, is
// some 20 instructions.)
struct Divisor {
    uint32_t d, m;
    int s;
    Divisor() = default;
    explicit Divisor(int by) : d((uint32_t)by), m(0), s(0) {
        int l = 0;
        while ((1ll << l) < by) ++l;
        if (l > 0) { m = (uint32_t)((1ull << (31 + l)) / d + 1); s = l - 1; }
    }
    __host__ __device__ int div(int n) const {
        if (d == 1) return n;
#ifdef __CUDA_ARCH__
        return (int)(__umulhi((uint32_t)n, m) >> s);
#else
        return (int)((uint64_t)(uint32_t)n * m >> 32 >> s);
#endif
    }
};

// Place in a ring of N slots guarded by a full and an empty mbarrier each: the slot, and the parity of its use.  Whoever empties the ring
// waits for `phase`, whoever fills it for `phase ^ 1` (which a fresh barrier passes).  Nothing counts up: a count of 32 bits comes round
// after 2^32 key tiles of one CTA, where a ring of 3 or 5 slots would jump.
template <int N> struct RingAt {
    uint32_t slot = 0, phase = 0;
    __host__ __device__ void next() {
        if (++slot == N) { slot = 0; phase ^= 1; }
    }
};

// The clock of the bounded waits: nanoseconds in units of 1024, 32 bits of them.  They come round after 73 minutes; the low word of the
// nanoseconds does after 4.3 s, so that a wait of 4 s whose block was not on the SM from its end until then began anew.
__host__ __device__ inline uint32_t wait_ticks(unsigned long long ns) { return (uint32_t)(ns >> 10); }
__host__ __device__ inline uint32_t wait_limit(unsigned long long ns) { return wait_ticks(ns) + 2; }       // (a wait's ends are rounded: never early)
__host__ __device__ inline bool wait_over(uint32_t since, uint32_t now, uint32_t limit) { return now - since > limit; }

// codes of the waits of the item queue: for the CTA's next item, for room to ask for one
constexpr int WAIT_NEXT_ITEM = 50, WAIT_NEXT_ROOM = 51;
// status word 2 of a wait that gave up: the query block at work, or the number in the CTA of the item waited for (50) or asking (51)
__host__ __device__ inline int stalled_work(int where, int query_block, uint32_t ord) {
    return where == WAIT_NEXT_ITEM || where == WAIT_NEXT_ROOM ? (int)ord : query_block;
}

struct AttnParams {
    int B, Hq, Hkv, G, n, K;
    int w;                   // window, at most n: positions and differences of positions stay within 32 bits
    int nqb;                 // items per head: 256-row query blocks (128-row tiles when D = 256)
    int nqt, nkt, nkw;
    Divisor by_heads, by_group, by_G, by_Hkv, by_Hq;      // by batch * Hq, nqb * G, G, Hkv, Hq
    float scale, softcap;
    const uint32_t* mq;
    const uint32_t* gbits;
    const uint32_t* live;
    __nv_bfloat16* o;
    int64_t o_sb, o_sh, o_sn;
    bool o_wide;             // its base and strides allow 32-byte stores
    float* lse;
    int32_t* status;
    long long nitems;
    int by_length;           // token order: items longest first over all heads (else KV head by KV head)
    // class-sorted layout: Q/K/V are the sorted copies, tiles are tiles of the sorted order
    int nqp, nkp, nqblk;
    int ipb;                 // items per block of 256 sorted queries (1, or 2 when an item is one query tile)
    const int32_t* perm_q;
    const int32_t* perm_k;
    const uint32_t* cls_k;
    const int32_t* ncls_k;
    const int32_t* qrange;
    const int32_t* order;
    const unsigned long long* counters;
    // training-time soft gate (Sec. 2 "Gated attention"): assignments [B, n, gate_ld] fp32, lambda / 2
    const float* gate_g;
    int gate_ld;
    float gate_hl;
    // window pass of the split layout: only the tiles that reach into the window, only pairs WITHOUT a shared group
    // class-sorted pass of the split layout: only pairs WITH a shared group (the window pass covers the others)
    int share_only;
    // group-major keys: bitmaps of the list entries per group, [B*Hkv][nkp/128][K][4] (nullptr in the other layouts)
    const uint32_t* gbits_s;
    int local_only;
    const float* join;       // partial O (fp32, rows as in o32; its logsumexps in `lse`) to join with this pass's, or nullptr
    float* o32;              // partial passes: O in fp32, rows [B*Hq][n][D], instead of bf16 to `o`
    unsigned long long wait_limit_ns;   // bound of every wait inside the kernel
    long long stall_at;      // diagnostic: index of a K/V ring stage the producer leaves unfilled (-1 = none)
};

// What decides which tiles are visited and which pairs kept: every causal pair; masks of tokens in their own order (live far
// tiles and the window, or the window alone: `local_only`); the class-sorted copies.  A template parameter of the kernel: the
// softmax warps hold 128 scores a thread, and the state of a walk they do not take would go to local memory, every tile.
enum : int { WALK_DENSE = 0, WALK_TOKEN = 1, WALK_SORTED = 2 };

// Enumerates the key tiles a 256-row query block visits, in increasing order.  In dense mode every role of the CTA runs the
// walk for itself; in the other modes the TMA thread runs it and hands the tiles on (TileInfo).
template <int WALK> struct TileWalk;

// One visited tile as the TMA thread hands it to the MMA and softmax warps, through a ring in shared memory: which tile (-1:
// the item has no more), and what its mask is made from, copied by the TMA unit while earlier tiles are computed: token
// order, the tile's bitmaps per group (K x 128 bits); class-sorted, the 128 positions and the mask value of the class.
// With every softmax warp walking for itself and reading this from L2 when a tile came up, the mask took 1070 cycles of a
// tile's 3900 in token order and 750 in the sorted one, in series with the tile's scores.
struct __align__(16) TileInfo {
    int kb;
    uint32_t cls;
    uint32_t pad[2];
    uint32_t data[128];
};

template <> struct TileWalk<WALK_DENSE> {
    int b, b_last;
    static constexpr int jk = 0;
    // a0 = first 128-row query tile of the item, nq = number of query tiles of the item (1 or 2)
    __device__ __forceinline__ void init(const AttnParams& p, int, int a0, int nq) {
        b = 0;
        b_last = (min(p.n, (a0 + nq) * 128) - 1) >> 7;
    }
    // next key tile, or -1
    __device__ __forceinline__ int next() { return b <= b_last ? b++ : -1; }
};

template <> struct TileWalk<WALK_TOKEN> {
    const uint32_t* l0;
    int nl, nkw;                // live rows (query tiles) to OR, and their stride in words
    int f0, b_last, b, wd;      // wd = current word of the live bitmap, past its end when the far tiles are through
    uint32_t bits;
    static constexpr int jk = 0;
    __device__ __forceinline__ void init(const AttnParams& p, int hq, int a0, int nq) {
        b_last = (min(p.n, (a0 + nq) * 128) - 1) >> 7;
        const int d = a0 * 128 - p.w;
        f0 = d > 0 ? d >> 7 : 0;                          // tiles before f0 are far for every query tile of the item
        nkw = p.nkw;
        l0 = p.live + ((size_t)hq * p.nqt + a0) * nkw;
        nl = min(nq, p.nqt - a0);
        wd = p.local_only ? nkw : -1;
        bits = 0;
        b = f0;
    }
    __device__ __forceinline__ int next() {
#pragma unroll 1
        while (wd * 32 < f0) {
            if (bits) {
                const int c = __ffs(bits) - 1;
                bits &= bits - 1;
                return wd * 32 + c;
            }
            ++wd;
            if (wd * 32 >= f0) break;
            uint32_t x = 0;
#pragma unroll 1
            for (int r = 0; r < nl; ++r) x |= dep_load(l0 + (size_t)r * nkw + wd);
            const int rem = f0 - wd * 32;
            bits = rem < 32 ? x & ((1u << rem) - 1u) : x;
        }
        return b <= b_last ? b++ : -1;
    }
};

template <> struct TileWalk<WALK_SORTED> {
    const int32_t* qr;          // the ranges of sorted key tiles, key class by key class
    int nck, jk, b, rend;       // jk = class of the tile that next() returned
    __device__ __forceinline__ void init(const AttnParams& p, int hq, int a0, int) {
        const int bb = p.by_Hq.div(hq), hk = bb * p.Hkv + p.by_G.div(hq - bb * p.Hq);
        qr = p.qrange + ((size_t)hq * p.nqblk + (a0 >> 1)) * FOCUS_MAX_CLASSES * 2;
        nck = dep_load(p.ncls_k + hk);
        jk = -1;
        b = rend = 0;
    }
    __device__ __forceinline__ int next() {
#pragma unroll 1
        while (b >= rend) {
            if (++jk >= nck) return -1;
            const int2 r = dep_load(reinterpret_cast<const int2*>(qr) + jk);
            b = r.x;
            rend = r.y;
        }
        return b++;
    }
};

// Per-row 128-bit keep bitmap of one (query tile, key tile) pair; `masked` when it has to be applied at all.
struct TileMask {
    uint32_t kw[4];
    bool masked;
};

__device__ __forceinline__ uint32_t low_bits(int n) { return n >= 32 ? 0xffffffffu : (n <= 0 ? 0u : ((1u << n) - 1u)); }

// every causal pair
__device__ __forceinline__ void build_tile_mask_dense(TileMask& tm, int a, int kb, int i) {
    tm.masked = kb >= a;
    if (tm.masked) {
#pragma unroll
        for (int q = 0; q < 4; ++q) tm.kw[q] = low_bits(i - kb * 128 + 1 - 32 * q);       // columns < that are causal
    }
}

// `gbits`: the tile's bitmaps per group (shared memory)
__device__ __forceinline__ void build_tile_mask(TileMask& tm, const AttnParams& p, int a, int kb, int i, uint32_t mi, int f_x,
                                                const uint32_t* gbits) {
    const int c0 = kb * 128;
    const bool need_causal = kb >= a;
    const bool need_window = p.local_only || (kb >= f_x && a * 128 + 127 - c0 > p.w);
    const bool need_group = need_window || kb < f_x;
    tm.masked = need_causal || need_group;
    if (tm.masked) {
        uint32_t sh[4] = {0, 0, 0, 0};
        if (need_group) {
#pragma unroll 1
            for (uint32_t rem = mi; rem; rem &= rem - 1) {
                const uint4 t = *reinterpret_cast<const uint4*>(gbits + (__ffs(rem) - 1) * 4);
                sh[0] |= t.x; sh[1] |= t.y; sh[2] |= t.z; sh[3] |= t.w;
            }
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            uint32_t keep = 0xffffffffu;
            if (need_group) {
                keep = sh[q];
                if (need_window) {
                    const uint32_t win = ~low_bits(i - p.w - c0 - 32 * q);      // columns from there on are inside the window
                    keep = p.local_only ? (win & ~keep) : (keep | win);     // window pass: in the window and not sharing
                }
            }
            if (need_causal) keep &= low_bits(i - c0 + 1 - 32 * q);
            tm.kw[q] = keep;
        }
        // a tile that every row of the warp keeps whole needs no mask after all (rows past the end keep nothing: not asked)
        tm.masked = __any_sync(0xffffffffu, i < p.n && (tm.kw[0] & tm.kw[1] & tm.kw[2] & tm.kw[3]) != 0xffffffffu);
    }
}

// Item `id` of the list.  The grid has one block per item; blocks start in the order of the list and a running CTA takes
// over the next one that has not started (cluster launch control), so the list is worked off like a queue and what counts
// is that the expensive items come first.  Class-sorted: as build_tiles ordered them, KV head by KV head, most key tiles
// first.  Token order: longest query blocks first, over all heads at once (`by_length`) while K and V of all heads stay in
// L2, else KV head by KV head, so that the CTAs running at the same time stream the K/V of one head through L2.
struct Item { int A, bb, h, hq; };
template <int WALK>
__device__ __forceinline__ void item_at(const AttnParams& p, int id, Item& t) {
    if (WALK == WALK_SORTED) {
        const int2 e = dep_load(reinterpret_cast<const int2*>(p.order) + (id >> (p.ipb - 1)));      // (ipb is 1 or 2)
        t.hq = e.x;
        t.A = e.y * p.ipb + (id & (p.ipb - 1));
    } else if (p.by_length) {
        const int q = p.by_heads.div(id);
        t.A = p.nqb - 1 - q;
        t.hq = id - q * p.B * p.Hq;
    } else {
        const int grp = p.by_group.div(id);               // batch * Hkv + KV head
        const int rem = id - grp * p.nqb * p.G, q = p.by_G.div(rem), b = p.by_Hkv.div(grp);
        t.A = p.nqb - 1 - q;
        t.hq = b * p.Hq + (grp - b * p.Hkv) * p.G + rem - q * p.G;
    }
    t.bb = p.by_Hq.div(t.hq);
    t.h = t.hq - t.bb * p.Hq;
}

// number of entries of the ascending 128-entry array `a` that are <= v (fixed-depth search)
__device__ __forceinline__ int count_le_128(const int32_t* __restrict__ a, int v) {
    int lo = 0;
#pragma unroll
    for (int step = 64; step >= 1; step >>= 1)
        if (a[lo + step - 1] <= v) lo += step;
    return lo + (lo == 127 && a[127] <= v ? 1 : 0);
}

// Tile mask in the class-sorted layout.  The keys of a tile belong to one class and their original
// positions `kpos` ascend, so a row keeps a contiguous range of columns: those at or before its own
// position and, unless the classes share a group, not further back than the window.  The decisions
// "no mask needed" / "nothing attended" are taken per warp from the warp's smallest and largest row
// position.
// `window_ok` = false (class-sorted pass of the split layout): a row that shares no group with the tile's class keeps
// nothing of it, whatever the distance.
__device__ __forceinline__ void build_tile_mask_sorted(TileMask& tm, int w, const int32_t* __restrict__ kpos, bool share,
                                                       int pos, int wmin, int wmax, bool window_ok) {
    const int k_first = kpos[0], k_last = kpos[127];
    const bool none = wmax < 0 || k_first > wmax || (!share && !window_ok);
    const bool need_causal = k_last > wmin;
    const bool need_window = !share && wmax - k_first > w;          // (wmax >= -1, k_first >= 0)
    tm.masked = __any_sync(0xffffffffu, need_causal || need_window || none);        // (rows of one warp may differ: padding)
    tm.kw[0] = tm.kw[1] = tm.kw[2] = tm.kw[3] = 0xffffffffu;
    if (tm.masked) {
        const int hi = none ? 0 : (need_causal ? (pos < 0 ? 0 : count_le_128(kpos, pos)) : 128);          // columns < hi are causal
        const int edge = pos - w - 1;
        const int lo = (need_window && pos >= 0 && edge >= 0) ? count_le_128(kpos, edge) : 0;   // columns >= lo are in the window
#pragma unroll
        for (int q = 0; q < 4; ++q) tm.kw[q] = low_bits(hi - 32 * q) & ~low_bits(lo - 32 * q);
    }
}

// Group-major keys: the tile belongs to the list of group g.  A key that shares a LOWER group with the row is attended
// under that lower group's list, so here it is masked out: `lower` = the row's groups below g, `gb` = the tile's
// per-group bitmaps.  Every sharing pair is then computed exactly once.
__device__ __forceinline__ void exclude_lower_groups(TileMask& tm, const uint32_t* gb, uint32_t lower, int K) {
    uint32_t ex[4] = {0u, 0u, 0u, 0u};
#pragma unroll 1
    for (uint32_t rem = lower; rem; rem &= rem - 1) {
        const int a = __ffs(rem) - 1;
        if (a < K) {
            const uint4 t = dep_load(reinterpret_cast<const uint4*>(gb + a * 4));
            ex[0] |= t.x; ex[1] |= t.y; ex[2] |= t.z; ex[3] |= t.w;
        }
    }
    tm.kw[0] &= ~ex[0]; tm.kw[1] &= ~ex[1]; tm.kw[2] &= ~ex[2]; tm.kw[3] &= ~ex[3];
    tm.masked = __any_sync(0xffffffffu, tm.masked || (ex[0] | ex[1] | ex[2] | ex[3]) != 0u);
}

}  // namespace focus
