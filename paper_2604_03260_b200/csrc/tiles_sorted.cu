// Class-sorted layout of focus_build_tiles (paper Sec. 2, item "Group": sort tokens by group with a
// stable sort, which keeps causal order inside a group).
//
// A token's class is its membership-mask value.  Per head the tokens are stably sorted by class
// (classes ascending by mask value, original positions ascending inside a class); every class
// segment is padded to a whole number of tiles, so that a tile of the sorted order holds one class.
// Then a (query tile, key tile) pair is all-share or none-share, and the attended pairs of a query
// block are: for every key class that shares a group with the block's class, the keys of that class
// up to the block's last position; for every other key class, only the keys inside the window.
// These ranges are written per block of 256 sorted queries, together with an order of the blocks
// (most key tiles first inside each KV head group) for the persistent attention kernel.
#include "common.cuh"

#include <limits.h>

namespace focus {

constexpr int MAXC = FOCUS_MAX_CLASSES;
constexpr unsigned long long HASH_EMPTY = 0ull;

__device__ __forceinline__ unsigned int hash_slot(uint32_t v) { return (v * 2654435761u) >> 24; }   // 0..255

// Query and key heads go through the same steps, in the same launches: row r of a grid is head r of the query side, then
// of the key side.
struct SortSide {
    const uint32_t* m;
    unsigned long long* table;
    uint32_t* cls;
    int32_t *ncls, *hist, *cnt, *seg, *perm;
    int heads, npad, pad, fill;          // pad = slots a class segment is rounded up to; fill = what perm holds in the padding
};
struct SortSides { SortSide s[2]; };
__device__ __forceinline__ const SortSide& side_of(const SortSides& sides, int row, int& head) {
    const bool second = row >= sides.s[0].heads;
    head = second ? row - sides.s[0].heads : row;
    return sides.s[second ? 1 : 0];
}

// ---------------------------------------------------------------------------------------------
// 1. distinct mask values per head: block-local hash set, merged into a global one per head
// ---------------------------------------------------------------------------------------------
__global__ void __launch_bounds__(256)
collect_classes_kernel(const SortSides sides, int n, int nchunk) {
    __shared__ unsigned long long loc[SORT_HASH];
    int head;
    const SortSide& sd = side_of(sides, blockIdx.x / nchunk, head);
    const uint32_t* __restrict__ m = sd.m;
    for (int s = threadIdx.x; s < SORT_HASH; s += blockDim.x) loc[s] = HASH_EMPTY;
    __syncthreads();
    const int t0 = (blockIdx.x % nchunk) * SORT_CHUNK;
    for (int t = t0 + threadIdx.x; t < min(n, t0 + SORT_CHUNK); t += blockDim.x) {
        const uint32_t v = m[(size_t)head * n + t];
        const unsigned long long key = (1ull << 32) | v;
        unsigned int s = hash_slot(v);
        for (int probe = 0; probe < SORT_HASH; ++probe) {
            const unsigned long long old = atomicCAS(&loc[s], HASH_EMPTY, key);
            if (old == HASH_EMPTY || old == key) break;
            s = (s + 1) & (SORT_HASH - 1);
        }
    }
    __syncthreads();
    unsigned long long* glob = sd.table + (size_t)head * SORT_HASH;
    for (int i = threadIdx.x; i < SORT_HASH; i += blockDim.x) {
        const unsigned long long key = loc[i];
        if (key == HASH_EMPTY) continue;
        unsigned int s = hash_slot((uint32_t)key);
        for (int probe = 0; probe < SORT_HASH; ++probe) {
            const unsigned long long old = atomicCAS(&glob[s], HASH_EMPTY, key);
            if (old == HASH_EMPTY || old == key) break;
            s = (s + 1) & (SORT_HASH - 1);
        }
    }
}

// one block per head: compact the hash set, sort ascending, flag more than MAXC values
__global__ void __launch_bounds__(SORT_HASH)
finalize_classes_kernel(const SortSides sides, unsigned long long* counters) {
    __shared__ uint32_t vals[SORT_HASH];
    __shared__ int cnt;
    int head;
    const SortSide& sd = side_of(sides, blockIdx.x, head);
    uint32_t* __restrict__ cls = sd.cls;
    if (threadIdx.x == 0) cnt = 0;
    __syncthreads();
    const unsigned long long key = sd.table[(size_t)head * SORT_HASH + threadIdx.x];
    if (key != HASH_EMPTY) vals[atomicAdd(&cnt, 1)] = (uint32_t)key;
    __syncthreads();
    const int c = cnt;
    if (threadIdx.x < c) {
        const uint32_t v = vals[threadIdx.x];
        int rank = 0;
        for (int j = 0; j < c; ++j) rank += vals[j] < v;
        if (rank < MAXC) cls[(size_t)head * MAXC + rank] = v;
    }
    if ((int)threadIdx.x >= c && threadIdx.x < MAXC) cls[(size_t)head * MAXC + threadIdx.x] = 0u;
    if (threadIdx.x == 0) {
        sd.ncls[head] = min(c, MAXC);
        if (c > MAXC) atomicAdd(&counters[4], 1ull);
    }
}

// index of value v in the ascending table (values not in the table, possible only after an
// overflow, fall into the last class below them)
__device__ __forceinline__ int class_index(const uint32_t* tab, int c, uint32_t v) {
    int lo = 0, hi = c - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (tab[mid] <= v) lo = mid; else hi = mid - 1;
    }
    return lo;
}

// ---------------------------------------------------------------------------------------------
// 2. counting sort: per-chunk histograms, scan over chunks, stable scatter
// ---------------------------------------------------------------------------------------------
__global__ void __launch_bounds__(SORT_CHUNK)
chunk_hist_kernel(const SortSides sides, int n, int nchunk) {
    __shared__ uint32_t tab[MAXC];
    __shared__ int h[MAXC];
    int head;
    const SortSide& sd = side_of(sides, blockIdx.x / nchunk, head);
    const int chunk = blockIdx.x % nchunk;
    if (threadIdx.x < MAXC) { tab[threadIdx.x] = sd.cls[(size_t)head * MAXC + threadIdx.x]; h[threadIdx.x] = 0; }
    __syncthreads();
    const int c = sd.ncls[head];
    const int t = chunk * SORT_CHUNK + threadIdx.x;
    const int ci = t < n ? class_index(tab, c, sd.m[(size_t)head * n + t]) : -1;
    const unsigned int same = __match_any_sync(0xffffffffu, ci);
    if (ci >= 0 && (threadIdx.x & 31) == __ffs(same) - 1) atomicAdd(&h[ci], __popc(same));        // one per warp and class
    __syncthreads();
    if (threadIdx.x < MAXC) sd.hist[((size_t)head * nchunk + chunk) * MAXC + threadIdx.x] = h[threadIdx.x];
}

// one block of MAXC threads per head (thread = class): running offsets over the chunks, class
// totals and padded segment starts
__global__ void __launch_bounds__(MAXC)
scan_chunks_kernel(const SortSides sides, int nchunk, unsigned long long* counters) {
    __shared__ int tot[MAXC];
    int head;
    const SortSide& sd = side_of(sides, blockIdx.x, head);
    const int c = threadIdx.x;
    int run = 0;
    constexpr int AHEAD = 16;       // loads under way at a time
    for (int k0 = 0; k0 < nchunk; k0 += AHEAD) {
        int32_t* p = sd.hist + ((size_t)head * nchunk + k0) * MAXC + c;
        int v[AHEAD];
#pragma unroll
        for (int k = 0; k < AHEAD; ++k) v[k] = k0 + k < nchunk ? p[(size_t)k * MAXC] : 0;
#pragma unroll
        for (int k = 0; k < AHEAD; ++k) {
            if (k0 + k < nchunk) p[(size_t)k * MAXC] = run;           // tokens of class c in earlier chunks
            run += v[k];
        }
    }
    tot[c] = run;
    sd.cnt[(size_t)head * MAXC + c] = run;
    __syncthreads();
    if (c == 0) {
        const int nc = sd.ncls[head];
        int s = 0;
        for (int j = 0; j <= MAXC; ++j) {
            sd.seg[(size_t)head * (MAXC + 1) + j] = s;
            if (j < nc) s += (tot[j] + sd.pad - 1) / sd.pad * sd.pad;
        }
        if (s > sd.npad) atomicAdd(&counters[4], 1ull);      // more entries than the sorted arrays hold (group-major lists of
                                                          // masks with more than topk bits): the attention kernel refuses
    }
}

__global__ void fill_kernel(int32_t* __restrict__ p, size_t count, int32_t value) {
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < count; i += (size_t)gridDim.x * blockDim.x)
        p[i] = value;
}

// stable scatter: slot = segment start + tokens of the class in earlier chunks + earlier warps of
// this chunk + earlier lanes of this warp.  Every block also fills its share of the padding slots.
__global__ void __launch_bounds__(SORT_CHUNK)
scatter_kernel(const SortSides sides, int n, int nchunk) {
    __shared__ uint32_t tab[MAXC];
    __shared__ int wcnt[SORT_CHUNK / 32][MAXC];
    __shared__ int seg[MAXC + 1], end[MAXC];
    int head;
    const SortSide& sd = side_of(sides, blockIdx.x / nchunk, head);
    const int chunk = blockIdx.x % nchunk, npad = sd.npad;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x < MAXC) tab[threadIdx.x] = sd.cls[(size_t)head * MAXC + threadIdx.x];
    if (threadIdx.x <= MAXC) {
        seg[threadIdx.x] = sd.seg[(size_t)head * (MAXC + 1) + threadIdx.x];
        if (threadIdx.x < MAXC) end[threadIdx.x] = seg[threadIdx.x] + sd.cnt[(size_t)head * MAXC + threadIdx.x];
    }
    for (int i = threadIdx.x; i < (SORT_CHUNK / 32) * MAXC; i += blockDim.x) (&wcnt[0][0])[i] = 0;
    __syncthreads();
    const int c = sd.ncls[head];
    const int t = chunk * SORT_CHUNK + threadIdx.x;
    const bool in = t < n;
    const int ci = in ? class_index(tab, c, sd.m[(size_t)head * n + t]) : -1;
    const unsigned int same = __match_any_sync(0xffffffffu, ci);
    const int rank = __popc(same & ((1u << lane) - 1u));
    if (in && rank == 0) wcnt[warp][ci] = __popc(same);
    __syncthreads();
    if (threadIdx.x < MAXC) {               // exclusive scan over the warps, per class
        int run = 0;
        for (int w = 0; w < SORT_CHUNK / 32; ++w) {
            const int v = wcnt[w][threadIdx.x];
            wcnt[w][threadIdx.x] = run;
            run += v;
        }
    }
    __syncthreads();
    int32_t* __restrict__ perm = sd.perm + (size_t)head * npad;
    if (in) {
        const int slot = seg[ci] + sd.hist[((size_t)head * nchunk + chunk) * MAXC + ci] + wcnt[warp][ci] + rank;
        if (slot < npad) perm[slot] = t;
    }
    // the padding: slots past the tokens of their class, and past the last class
    const int share = (npad + nchunk - 1) / nchunk;
    for (int slot = chunk * share + threadIdx.x; slot < min(npad, (chunk + 1) * share); slot += SORT_CHUNK) {
        int lo = 0, hi = c - 1;             // last class that starts at or before the slot
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (seg[mid] <= slot) lo = mid; else hi = mid - 1;
        }
        if (slot >= end[lo]) perm[slot] = sd.fill;
    }
}

// ---------------------------------------------------------------------------------------------
// 2b. group-major keys: K lists per KV head, list g = the keys that are members of group g, in token order.
// "Class" j of the key side is group j, so that the range and attention code reads the lists like class segments.
// ---------------------------------------------------------------------------------------------
__global__ void group_classes_kernel(int heads, int K, uint32_t* __restrict__ cls, int32_t* __restrict__ ncls) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < heads * MAXC) cls[i] = (i % MAXC) < K ? 1u << (i % MAXC) : 0u;
    if (i < heads) ncls[i] = K;
}

__global__ void __launch_bounds__(SORT_CHUNK)
group_hist_kernel(const uint32_t* __restrict__ m, int n, int K, int nchunk, int32_t* __restrict__ hist) {
    __shared__ int h[MAXC];
    const int head = blockIdx.y, chunk = blockIdx.x;
    if (threadIdx.x < MAXC) h[threadIdx.x] = 0;
    __syncthreads();
    const int t = chunk * SORT_CHUNK + threadIdx.x;
    const uint32_t v = t < n ? m[(size_t)head * n + t] : 0u;
    for (int g = 0; g < K; ++g) {
        const unsigned int b = __ballot_sync(0xffffffffu, (v >> g) & 1u);
        if ((threadIdx.x & 31) == 0 && b) atomicAdd(&h[g], __popc(b));
    }
    __syncthreads();
    if (threadIdx.x < MAXC) hist[((size_t)head * nchunk + chunk) * MAXC + threadIdx.x] = h[threadIdx.x];
}

// stable scatter into the lists: a key goes to the list of every group it belongs to
__global__ void __launch_bounds__(SORT_CHUNK)
group_scatter_kernel(const uint32_t* __restrict__ m, int n, int K, int nchunk, const int32_t* __restrict__ base,
                     const int32_t* __restrict__ seg, int npad, int32_t* __restrict__ perm) {
    __shared__ int wcnt[SORT_CHUNK / 32][32];
    const int head = blockIdx.y, chunk = blockIdx.x;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int t = chunk * SORT_CHUNK + threadIdx.x;
    const uint32_t v = t < n ? m[(size_t)head * n + t] : 0u;
    int rank[32];
#pragma unroll
    for (int g = 0; g < 32; ++g) {
        const unsigned int b = g < K ? __ballot_sync(0xffffffffu, (v >> g) & 1u) : 0u;
        rank[g] = __popc(b & ((1u << lane) - 1u));
        if (lane == 0) wcnt[warp][g] = __popc(b);
    }
    __syncthreads();
    if (threadIdx.x < 32) {                 // exclusive scan over the warps, per group
        int run = 0;
        for (int w = 0; w < SORT_CHUNK / 32; ++w) {
            const int c = wcnt[w][threadIdx.x];
            wcnt[w][threadIdx.x] = run;
            run += c;
        }
    }
    __syncthreads();
#pragma unroll
    for (int g = 0; g < 32; ++g) {
        if (g < K && ((v >> g) & 1u)) {
            const int slot = seg[(size_t)head * (MAXC + 1) + g] + base[((size_t)head * nchunk + chunk) * MAXC + g] +
                             wcnt[warp][g] + rank[g];
            if (slot < npad) perm[(size_t)head * npad + slot] = t;
        }
    }
}

// block of 128 threads per (tile of the lists, KV head): per group the bitmap of entries that are members of it
__global__ void __launch_bounds__(128)
gbits_sorted_kernel(const uint32_t* __restrict__ m, int n, int K, const int32_t* __restrict__ perm, int npad,
                    uint32_t* __restrict__ gbits_s) {
    const int tile = blockIdx.x, head = blockIdx.y;
    const int pos = perm[(size_t)head * npad + (size_t)tile * 128 + threadIdx.x];
    const uint32_t v = (pos >= 0 && pos < n) ? m[(size_t)head * n + pos] : 0u;
    uint32_t* gb = gbits_s + ((size_t)head * (npad / 128) + tile) * K * 4;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    for (int g = 0; g < K; ++g) {
        const uint32_t word = __ballot_sync(0xffffffffu, (v >> g) & 1u);
        if (lane == 0) gb[g * 4 + warp] = word;
    }
}

// ---------------------------------------------------------------------------------------------
// 3. key-tile ranges per query block, block costs, block order
// ---------------------------------------------------------------------------------------------
// number of entries of the ascending array a[0..len) that are <= v
__device__ __forceinline__ int count_le(const int32_t* __restrict__ a, int len, long long v) {
    int lo = 0, hi = len;
    while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if ((long long)a[mid] <= v) lo = mid + 1; else hi = mid;
    }
    return lo;
}

// thread = (query head, query block, key class)
__global__ void __launch_bounds__(256)
qrange_kernel(int HQ, int Hq, int Hkv, int G_heads, int w, int nqp, int nkp, const int32_t* __restrict__ ncls_q,
              const int32_t* __restrict__ ncls_k, const uint32_t* __restrict__ cls_q, const uint32_t* __restrict__ cls_k,
              const int32_t* __restrict__ cnt_q, const int32_t* __restrict__ cnt_k, const int32_t* __restrict__ seg_q,
              const int32_t* __restrict__ seg_k, const int32_t* __restrict__ perm_q, const int32_t* __restrict__ perm_k,
              int32_t* __restrict__ qrange, int32_t* __restrict__ cost, unsigned long long* counters, int sharing_only) {
    // a block of 256 threads holds the classes of four query blocks: their costs are summed here (an atomic per thread on
    // the one counter of all tiles made this launch 50 us long at 32 heads x 32768 tokens, 81 us at 131072)
    __shared__ int sum_s[8];
    const int nqblk = nqp / 256;
    const long long gid = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const bool in = gid < (long long)HQ * nqblk * MAXC;
    const int jk = (int)(gid % MAXC);
    const int blk = (int)((gid / MAXC) % nqblk);
    const int hq = in ? (int)(gid / ((long long)MAXC * nqblk)) : 0;
    const int hk = (hq / Hq) * Hkv + (hq % Hq) / G_heads;
    int first = 0, last = 0;
    const int32_t* sq = seg_q + (size_t)hq * (MAXC + 1);
    const int ncq = ncls_q[hq], nck = ncls_k[hk];
    const int start = blk * 256;
    if (in && jk < nck && start < sq[ncq]) {
        int jq = 0;
        while (jq + 1 < ncq && sq[jq + 1] <= start) ++jq;          // class of this query block
        const int valid_end = sq[jq] + cnt_q[(size_t)hq * MAXC + jq];    // one past the last real row of the class
        const int32_t* pq = perm_q + (size_t)hq * nqp;
        const long long pmin = pq[start], pmax = pq[min(start + 256, valid_end) - 1];
        const int ks0 = seg_k[(size_t)hk * (MAXC + 1) + jk], kc = cnt_k[(size_t)hk * MAXC + jk];
        const int32_t* pk = perm_k + (size_t)hk * nkp + ks0;
        const bool share = (cls_q[(size_t)hq * MAXC + jq] & cls_k[(size_t)hk * MAXC + jk]) != 0u;
        const int hi = count_le(pk, kc, pmax);                             // keys at or before the block's last position
        const int lo = share ? 0 : count_le(pk, kc, pmin - w - 1);          // keys before the window of the first row
        // with a separate window pass only the classes that share a group with the block's class are listed
        if (hi > lo && (share || !sharing_only)) {
            first = (ks0 + lo) / 128;
            last = (ks0 + hi + 127) / 128;
        }
    }
    if (in) reinterpret_cast<int2*>(qrange)[gid] = make_int2(first, last);
    const int tiles = __reduce_add_sync(0xffffffffu, last - first);
    if ((threadIdx.x & 31) == 0) sum_s[threadIdx.x >> 5] = tiles;
    __syncthreads();
    static_assert(MAXC == 64, "two warps per query block");
    if (in && jk == 0) cost[(size_t)hq * nqblk + blk] = sum_s[threadIdx.x >> 5] + sum_s[(threadIdx.x >> 5) + 1];
    if (threadIdx.x == 0) {
        int all = 0;
        for (int w = 0; w < 8; ++w) all += sum_s[w];
        if (all) atomicAdd(&counters[3], (unsigned long long)all);
    }
}

// one block per KV head group: counting sort of its (query head, query block) pairs by cost, descending
constexpr int ORDER_BUCKETS = 2048;
__global__ void __launch_bounds__(1024)
order_kernel(int Hq, int Hkv, int G_heads, int nqblk, int max_cost, const int32_t* __restrict__ cost,
             int32_t* __restrict__ order) {
    __shared__ int bucket[ORDER_BUCKETS];
    __shared__ int carry;
    const int grp = blockIdx.x;                          // batch * Hkv + KV head
    const int hq0 = (grp / Hkv) * Hq + (grp % Hkv) * G_heads;
    const int items = G_heads * nqblk;
    for (int i = threadIdx.x; i < ORDER_BUCKETS; i += blockDim.x) bucket[i] = 0;
    if (threadIdx.x == 0) carry = 0;
    __syncthreads();
    auto bucket_of = [&](int c) {                        // bucket 0 holds the most expensive blocks
        long long q = (long long)c * (ORDER_BUCKETS - 1) / (max_cost > 0 ? max_cost : 1);
        if (q > ORDER_BUCKETS - 1) q = ORDER_BUCKETS - 1;
        return ORDER_BUCKETS - 1 - (int)q;
    };
    for (int i = threadIdx.x; i < items; i += blockDim.x) {
        const int g = i / nqblk, blk = i % nqblk;
        atomicAdd(&bucket[bucket_of(cost[(size_t)(hq0 + g) * nqblk + blk])], 1);
    }
    __syncthreads();
    // exclusive scan of the buckets, 1024 at a time
    for (int b0 = 0; b0 < ORDER_BUCKETS; b0 += 1024) {
        const int idx = b0 + threadIdx.x;
        const int v = bucket[idx];
        int x = v;
        // inclusive scan inside the warp, then across warps through shared memory
        for (int off = 1; off < 32; off <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, x, off);
            if ((threadIdx.x & 31) >= off) x += y;
        }
        __shared__ int wsum[32];
        if ((threadIdx.x & 31) == 31) wsum[threadIdx.x >> 5] = x;
        __syncthreads();
        if (threadIdx.x < 32) {
            int s = wsum[threadIdx.x];
            for (int off = 1; off < 32; off <<= 1) {
                const int y = __shfl_up_sync(0xffffffffu, s, off);
                if (threadIdx.x >= off) s += y;
            }
            wsum[threadIdx.x] = s;
        }
        __syncthreads();
        const int before = carry + (threadIdx.x >= 32 ? wsum[(threadIdx.x >> 5) - 1] : 0) + x - v;
        __syncthreads();
        bucket[idx] = before;
        if (threadIdx.x == 1023) carry = before + v;
        __syncthreads();
    }
    int32_t* out = order + (size_t)grp * items * 2;
    for (int i = threadIdx.x; i < items; i += blockDim.x) {
        const int g = i / nqblk, blk = i % nqblk;
        const int pos = atomicAdd(&bucket[bucket_of(cost[(size_t)(hq0 + g) * nqblk + blk])], 1);
        out[2 * pos] = hq0 + g;
        out[2 * pos + 1] = blk;
    }
}

// ---------------------------------------------------------------------------------------------
// 4. gather of Q / K / V rows into the sorted order (run by focus_attn_fwd), one launch
// ---------------------------------------------------------------------------------------------
// Four rows per thread, all their loads under way at once (one row per thread: 4.5 TB/s read and written at 32 x 131072 x 128).
constexpr int GATHER_ROWS = 4;
struct GatherSide {
    const __nv_bfloat16* src;
    int64_t sb, sh, sn;
    const int32_t* perm;
    const int32_t* seg;
    __nv_bfloat16* dst;
    int H, npad, blocks;             // heads per sequence, slots per head, thread blocks per head
};
struct GatherSides { GatherSide s[3]; int first[3]; };       // first[k] = first block of side k

template <int D>
__global__ void __launch_bounds__(256)
gather_rows_kernel(const GatherSides sides, int n) {
    constexpr int VEC = D / 8, RPB = 256 / VEC;          // 16-byte pieces per row, rows a block covers at a time
    const int k = (int)blockIdx.x >= sides.first[2] ? 2 : (int)blockIdx.x >= sides.first[1] ? 1 : 0;
    const GatherSide& g = sides.s[k];
    const int head = (blockIdx.x - sides.first[k]) / g.blocks, blk = (blockIdx.x - sides.first[k]) % g.blocks;
    const int used = g.seg[(size_t)head * (MAXC + 1) + MAXC];
    const int slot0 = blk * RPB * GATHER_ROWS + threadIdx.x / VEC, v = threadIdx.x % VEC;
    if (slot0 >= used) return;
    const __nv_bfloat16* src = g.src + (size_t)(head / g.H) * g.sb + (size_t)(head % g.H) * g.sh + v * 8;
    int pos[GATHER_ROWS];
    uint4 val[GATHER_ROWS];
#pragma unroll
    for (int r = 0; r < GATHER_ROWS; ++r) {
        const int slot = slot0 + r * RPB;
        pos[r] = slot < used ? g.perm[(size_t)head * g.npad + slot] : -1;
    }
#pragma unroll
    for (int r = 0; r < GATHER_ROWS; ++r) {
        val[r] = make_uint4(0u, 0u, 0u, 0u);             // padding rows are zero
        if (pos[r] >= 0 && pos[r] < n) val[r] = *reinterpret_cast<const uint4*>(src + (size_t)pos[r] * g.sn);
    }
#pragma unroll
    for (int r = 0; r < GATHER_ROWS; ++r) {
        const int slot = slot0 + r * RPB;
        if (slot < used) *reinterpret_cast<uint4*>(g.dst + ((size_t)head * g.npad + slot) * D + v * 8) = val[r];
    }
}

int launch_gather_sorted(const focus_shape* s, const focus_tensor& q, const focus_tensor& k, const focus_tensor& v, const focus_tiles_layout& L,
                         char* ws, cudaStream_t st) {
    const int per_block = 256 / (s->D / 8) * GATHER_ROWS;
    GatherSides sides;
    long long blocks = 0;
    for (int i = 0; i < 3; ++i) {
        const focus_tensor& t = i == 0 ? q : i == 1 ? k : v;
        const int npad = i == 0 ? L.nqp : L.nkp, H = i == 0 ? s->Hq : s->Hkv;
        sides.s[i] = {reinterpret_cast<const __nv_bfloat16*>(t.ptr), t.stride_b, t.stride_h, t.stride_n,
                      reinterpret_cast<const int32_t*>(ws + (i == 0 ? L.perm_q : L.perm_k)), reinterpret_cast<const int32_t*>(ws + (i == 0 ? L.seg_q : L.seg_k)),
                      reinterpret_cast<__nv_bfloat16*>(ws + (i == 0 ? L.qs : i == 1 ? L.ks : L.vs)), H, npad, cdiv(npad, per_block)};
        sides.first[i] = (int)blocks;
        blocks += (long long)s->batch * H * sides.s[i].blocks;
    }
    if (blocks > 0x7fffffffll) return fail(FOCUS_ERR_CUDA, "gather: too many rows for one launch");
    switch (s->D) {
        case 64: gather_rows_kernel<64><<<(unsigned)blocks, 256, 0, st>>>(sides, s->n); break;
        case 128: gather_rows_kernel<128><<<(unsigned)blocks, 256, 0, st>>>(sides, s->n); break;
        case 256: gather_rows_kernel<256><<<(unsigned)blocks, 256, 0, st>>>(sides, s->n); break;
        default: return fail(FOCUS_ERR_UNSUPPORTED, "D (%d) must be 64, 128 or 256", s->D);
    }
    return check_cuda(cudaGetLastError(), "gather kernel");
}

// ---------------------------------------------------------------------------------------------
int launch_build_tiles_sorted(const focus_shape* s, const uint32_t* mq, const uint32_t* mk,
                              const focus_tiles_layout& L, char* ws, cudaStream_t st) {
    const int HQ = s->batch * s->Hq, HK = s->batch * s->Hkv;
    const int nchunk = cdiv(s->n, SORT_CHUNK);
    const int nqblk = L.nqp / 256;
    // scratch: hash sets | chunk histograms | block costs
    char* scr = ws + L.scratch;
    auto* table = reinterpret_cast<unsigned long long*>(scr);
    const size_t table_bytes = align_up((size_t)(HQ + HK) * SORT_HASH * 8, 256);
    auto* hist = reinterpret_cast<int32_t*>(scr + table_bytes);
    const size_t hist_bytes = align_up((size_t)(HQ + HK) * nchunk * MAXC * 4, 256);
    auto* cost = reinterpret_cast<int32_t*>(scr + table_bytes + hist_bytes);
    auto* counters = reinterpret_cast<unsigned long long*>(ws + L.counters);
    int rc;
    if ((rc = check_cuda(cudaMemsetAsync(table, 0, table_bytes, st), "cudaMemsetAsync(class tables)"))) return rc;
    SortSides sides;
    for (int k = 0; k < 2; ++k)
        sides.s[k] = {k ? mk : mq, table + (k ? (size_t)HQ * SORT_HASH : 0), reinterpret_cast<uint32_t*>(ws + (k ? L.cls_k : L.cls_q)),
                      reinterpret_cast<int32_t*>(ws + (k ? L.ncls_k : L.ncls_q)), hist + (k ? (size_t)HQ * nchunk * MAXC : 0),
                      reinterpret_cast<int32_t*>(ws + (k ? L.cnt_k : L.cnt_q)), reinterpret_cast<int32_t*>(ws + (k ? L.seg_k : L.seg_q)),
                      reinterpret_cast<int32_t*>(ws + (k ? L.perm_k : L.perm_q)), k ? HK : HQ, k ? L.nkp : L.nqp, k ? 128 : 256, k ? INT_MAX : -1};
    // group-major keys have lists of their own: only the query side is sorted by class
    const bool lists = L.layout == FOCUS_LAYOUT_GROUP_MAJOR;
    const int rows = lists ? HQ : HQ + HK;
    if ((long long)rows * nchunk > 0x7fffffffll) return fail(FOCUS_ERR_CUDA, "build_tiles: too many chunks of %d tokens for one launch", SORT_CHUNK);
    const unsigned grid = (unsigned)rows * (unsigned)nchunk;
    collect_classes_kernel<<<grid, 256, 0, st>>>(sides, s->n, nchunk);
    finalize_classes_kernel<<<rows, SORT_HASH, 0, st>>>(sides, counters);
    chunk_hist_kernel<<<grid, SORT_CHUNK, 0, st>>>(sides, s->n, nchunk);
    scan_chunks_kernel<<<rows, MAXC, 0, st>>>(sides, nchunk, counters);
    scatter_kernel<<<grid, SORT_CHUNK, 0, st>>>(sides, s->n, nchunk);
    if (lists) {
        SortSides keys;
        keys.s[0] = keys.s[1] = sides.s[1];
        const SortSide& k = keys.s[0];
        group_classes_kernel<<<cdiv(HK * MAXC, 256), 256, 0, st>>>(HK, s->K, k.cls, k.ncls);
        group_hist_kernel<<<dim3(nchunk, HK), SORT_CHUNK, 0, st>>>(mk, s->n, s->K, nchunk, k.hist);
        scan_chunks_kernel<<<HK, MAXC, 0, st>>>(keys, nchunk, counters);
        fill_kernel<<<1184, 256, 0, st>>>(k.perm, (size_t)HK * k.npad, INT_MAX);
        group_scatter_kernel<<<dim3(nchunk, HK), SORT_CHUNK, 0, st>>>(mk, s->n, s->K, nchunk, k.hist, k.seg, k.npad, k.perm);
        gbits_sorted_kernel<<<dim3(k.npad / 128, HK), 128, 0, st>>>(mk, s->n, s->K, k.perm, k.npad, reinterpret_cast<uint32_t*>(ws + L.gbits_s));
    }
    const long long nthreads = (long long)HQ * nqblk * MAXC;
    qrange_kernel<<<(unsigned)((nthreads + 255) / 256), 256, 0, st>>>(
        HQ, s->Hq, s->Hkv, s->Hq / s->Hkv, s->window, L.nqp, L.nkp, reinterpret_cast<const int32_t*>(ws + L.ncls_q),
        reinterpret_cast<const int32_t*>(ws + L.ncls_k), reinterpret_cast<const uint32_t*>(ws + L.cls_q),
        reinterpret_cast<const uint32_t*>(ws + L.cls_k), reinterpret_cast<const int32_t*>(ws + L.cnt_q),
        reinterpret_cast<const int32_t*>(ws + L.cnt_k), reinterpret_cast<const int32_t*>(ws + L.seg_q),
        reinterpret_cast<const int32_t*>(ws + L.seg_k), reinterpret_cast<const int32_t*>(ws + L.perm_q),
        reinterpret_cast<const int32_t*>(ws + L.perm_k), reinterpret_cast<int32_t*>(ws + L.qrange), cost, counters,
        layout_has_window_pass(L.layout) ? 1 : 0);
    order_kernel<<<HK, 1024, 0, st>>>(s->Hq, s->Hkv, s->Hq / s->Hkv, nqblk, L.nkp / 128, cost,
                                      reinterpret_cast<int32_t*>(ws + L.order));
    return check_cuda(cudaGetLastError(), "build_tiles (class-sorted) kernels");
}

__global__ void __launch_bounds__(256) fill_f32_kernel(float* __restrict__ x, size_t count, float v) {
    const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < count) x[i] = v;
}

int launch_fill_f32(float* x, size_t count, float v, cudaStream_t st) {
    fill_f32_kernel<<<(unsigned)((count + 255) / 256), 256, 0, st>>>(x, count, v);
    return check_cuda(cudaGetLastError(), "fill kernel launch");
}

}  // namespace focus
