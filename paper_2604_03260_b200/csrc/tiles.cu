// focus_build_tiles / focus_count_kept: integer-only passes over the membership masks.
//   summaries   OR/AND of the masks of each 128-token tile, per-group column bitmaps of key tiles
//   live set    far tile pairs whose OR summaries intersect (everything else far is skipped)
//   kept count  exact number of attended pairs per query head
#include "common.cuh"

namespace focus {

constexpr int TM = FOCUS_TILE_M;
constexpr int TN = FOCUS_TILE_N;

// One block of 128 threads per (head, tile): the heads of the query masks, then those of the key masks (+ gbits).  The first
// block clears the counters of the passes that follow.
__global__ void __launch_bounds__(128)
summarise_kernel(const uint32_t* mq, const uint32_t* mk, int HQ, int n, int nt, int K, uint32_t* orq,
                 uint32_t* andq, uint32_t* ork, uint32_t* andk, uint32_t* gbits,
                 unsigned long long* counters) {
    const int tile = blockIdx.x % nt, row = blockIdx.x / nt;
    const bool key = row >= HQ;
    const int head = key ? row - HQ : row;
    const int tok = tile * 128 + threadIdx.x;
    const bool in = tok < n;
    dep_wait();
    dep_trigger();
    if (blockIdx.x == 0 && threadIdx.x < 8) counters[threadIdx.x] = 0ull;
    const uint32_t v = in ? (key ? mk : mq)[(size_t)head * n + tok] : 0u;
    const uint32_t o = __reduce_or_sync(0xffffffffu, v), a = __reduce_and_sync(0xffffffffu, in ? v : 0xffffffffu);
    __shared__ uint32_t so[4], sa[4];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (lane == 0) { so[warp] = o; sa[warp] = a; }
    if (key) {
        uint32_t* gb = gbits + ((size_t)head * nt + tile) * K * 4;
        for (int g = 0; g < K; ++g) {
            const uint32_t word = __ballot_sync(0xffffffffu, (v >> g) & 1u);
            if (lane == 0) gb[g * 4 + warp] = word;
        }
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        (key ? ork : orq)[(size_t)head * nt + tile] = so[0] | so[1] | so[2] | so[3];
        (key ? andk : andq)[(size_t)head * nt + tile] = sa[0] & sa[1] & sa[2] & sa[3];
    }
}

// Live far-tile bitmap.  Key tile b is far for query tile a when every pair has i - j > w, i.e. b < (128 a - w) / 128;
// a far tile is live when the query tile's OR summary meets the key tile's, full when the AND summaries meet.  A warp makes
// a word of the bitmap at a time, its lanes the 32 key tiles; the words past the far tiles are zero.
// One block per (head, query tile).  The blocks past those of the HQ query heads, as many per KV head, write, per
// group g, which key tiles hold a member of g and which consist of members of g only, as bitmaps over the key tiles, also a
// word per warp; nothing in this launch waits for them.  (One thread per word in a launch of its own, before the live
// bitmap, took 6 to 25 us for its 32 dependent loads.)
__global__ void __launch_bounds__(128)
live_kernel(const uint32_t* orq, const uint32_t* andq, const uint32_t* ork,
            const uint32_t* andk, int G_heads, int Hq, int Hkv, int HQ, int w, int K, int nqt, int nkt, int nkw,
            uint32_t* kany, uint32_t* kall, uint32_t* live, int32_t* live_cnt,
            unsigned long long* counters) {
    __shared__ unsigned int s[2];
    if (threadIdx.x < 2) s[threadIdx.x] = 0;
    __syncthreads();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    dep_wait();
    dep_trigger();
    const int a = blockIdx.x % nqt, hq = blockIdx.x / nqt;
    if (hq >= HQ) {
        const int hk = hq - HQ;
        for (int wd = a * 4 + warp; wd < nkw; wd += nqt * 4) {
            const int b = wd * 32 + lane;
            const uint32_t o = b < nkt ? ork[(size_t)hk * nkt + b] : 0u, all = b < nkt ? andk[(size_t)hk * nkt + b] : 0u;
            for (int g = 0; g < K; ++g) {
                const uint32_t any_w = __ballot_sync(0xffffffffu, (o >> g) & 1u), all_w = __ballot_sync(0xffffffffu, (all >> g) & 1u);
                if (lane == 0) {
                    kany[((size_t)hk * K + g) * nkw + wd] = any_w;
                    kall[((size_t)hk * K + g) * nkw + wd] = all_w;
                }
            }
        }
        return;
    }
    const int b_idx = hq / Hq, h = hq % Hq;
    const int hk = b_idx * Hkv + h / G_heads;
    const uint32_t groups = K < 32 ? (1u << K) - 1u : 0xffffffffu;
    const uint32_t oq = orq[(size_t)hq * nqt + a] & groups, aq = andq[(size_t)hq * nqt + a] & groups;
    const long long d = (long long)a * TM - w;
    const int nfar_tiles = d > 0 ? (int)(d / TN) : 0;                 // far tiles are the first nfar_tiles key tiles
    unsigned int nlive = 0, nfull = 0;
    uint32_t* row = live + ((size_t)hq * nqt + a) * nkw;
    for (int wd = warp; wd < nkw; wd += 4) {
        const int b = wd * 32 + lane;
        const bool far = b < nfar_tiles;                              // (far tiles are all below nkt)
        const uint32_t lv = __ballot_sync(0xffffffffu, far && (oq & ork[(size_t)hk * nkt + b]) != 0u);
        const uint32_t fl = __ballot_sync(0xffffffffu, far && (aq & andk[(size_t)hk * nkt + b]) != 0u);
        if (lane == 0) row[wd] = lv;
        nlive += __popc(lv);
        nfull += __popc(fl);
    }
    if (lane == 0 && nlive) atomicAdd(&s[0], nlive);
    if (lane == 0 && nfull) atomicAdd(&s[1], nfull);
    __syncthreads();
    if (threadIdx.x == 0) {
        live_cnt[(size_t)hq * nqt + a] = (int32_t)s[0];
        if (nfar_tiles) atomicAdd(&counters[0], (unsigned long long)nfar_tiles);
        if (s[0]) atomicAdd(&counters[1], (unsigned long long)s[0]);
        if (s[1]) atomicAdd(&counters[2], (unsigned long long)s[1]);
    }
}

// Exact attended-pair count.  One block per (128-row query tile, head); thread = row.
// Row i keeps min(i, w) + 1 local keys plus every key j < i - w whose group bitmap bit is set in
// the OR of the bitmaps of the row's own groups.
__global__ void __launch_bounds__(128)
count_kept_kernel(const uint32_t* __restrict__ mq, const uint32_t* __restrict__ gbits, int G_heads, int Hq, int Hkv,
                  int n, int w, int K, int nkt, unsigned long long* __restrict__ out) {
    const int a = blockIdx.x, hq = blockIdx.y;
    const int b_idx = hq / Hq, h = hq % Hq;
    const int hk = b_idx * Hkv + h / G_heads;
    const int i = a * 128 + threadIdx.x;
    unsigned long long cnt = 0;
    if (i < n) {
        const uint32_t mi = mq[(size_t)hq * n + i];
        cnt = (unsigned long long)min(i, w) + 1ull;
        const long long nfar = (long long)i - w;            // keys 0 .. nfar-1 are beyond the window
        if (nfar > 0) {
            const int last_tile = (int)((nfar - 1) / TN);
            for (int b = 0; b <= last_tile; ++b) {
                const uint32_t* gb = gbits + ((size_t)hk * nkt + b) * K * 4;
                uint32_t wd[4] = {0, 0, 0, 0};
                uint32_t rem = mi;
                while (rem) {
                    const int g = __ffs(rem) - 1;
                    rem &= rem - 1;
                    if (g < K) {
                        const uint4 t = *reinterpret_cast<const uint4*>(gb + g * 4);
                        wd[0] |= t.x; wd[1] |= t.y; wd[2] |= t.z; wd[3] |= t.w;
                    }
                }
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const long long lim = nfar - ((long long)b * TN + q * 32);   // keys of this word below lim are far
                    uint32_t valid = lim >= 32 ? 0xffffffffu : (lim <= 0 ? 0u : ((1u << (int)lim) - 1u));
                    cnt += __popc(wd[q] & valid);
                }
            }
        }
    }
    // block reduce
    for (int off = 16; off >= 1; off >>= 1) cnt += __shfl_xor_sync(0xffffffffu, cnt, off);
    __shared__ unsigned long long s[4];
    if ((threadIdx.x & 31) == 0) s[threadIdx.x >> 5] = cnt;
    __syncthreads();
    if (threadIdx.x == 0) atomicAdd(&out[hq], s[0] + s[1] + s[2] + s[3]);
}

int launch_build_tiles_sorted(const focus_shape* s, const uint32_t* mq, const uint32_t* mk,
                              const focus_tiles_layout& L, char* ws, cudaStream_t st);

int launch_build_tiles(const focus_shape* s, const uint32_t* mq, const uint32_t* mk, int layout,
                       const focus_tiles_layout& L, char* ws, cudaStream_t st) {
    const int HQ = s->batch * s->Hq, HK = s->batch * s->Hkv;
    if (HQ > 65535) return fail(FOCUS_ERR_CUDA, "build_tiles: batch*Hq (%d) must not exceed 65535", HQ);
    const long long blocks = (long long)(HQ + HK) * L.nqt;
    if (blocks > 0x7fffffffll) return fail(FOCUS_ERR_CUDA, "build_tiles: %lld tiles of 128 tokens exceed 2^31 - 1", blocks);
    auto u32 = [&](size_t off) { return reinterpret_cast<uint32_t*>(ws + off); };
    auto* counters = reinterpret_cast<unsigned long long*>(ws + L.counters);
    int rc = check_cuda(launch_dependent(summarise_kernel, dim3((unsigned)blocks), dim3(128), 0, st, mq, mk, HQ, s->n, L.nqt, s->K, u32(L.orq),
                                         u32(L.andq), u32(L.ork), u32(L.andk), u32(L.gbits), counters), "summarise kernel launch");
    if (rc) return rc;
    rc = check_cuda(launch_dependent(live_kernel, dim3((unsigned)blocks), dim3(128), 0, st, u32(L.orq), u32(L.andq), u32(L.ork), u32(L.andk),
                                     s->Hq / s->Hkv, s->Hq, s->Hkv, HQ, s->window, s->K, L.nqt, L.nkt, L.nkw, u32(L.kany), u32(L.kall),
                                     u32(L.live), reinterpret_cast<int32_t*>(ws + L.live_cnt), counters), "live tiles kernel launch");
    if (rc) return rc;
    if (layout_is_sorted(layout))
        return launch_build_tiles_sorted(s, mq, mk, L, ws, st);
    return FOCUS_OK;
}

int launch_count_kept(const focus_shape* s, const uint32_t* mq, const focus_tiles_layout& L, const char* ws,
                      unsigned long long* out, cudaStream_t st) {
    const int HQ = s->batch * s->Hq;
    int rc = check_cuda(cudaMemsetAsync(out, 0, (size_t)HQ * sizeof(unsigned long long), st), "cudaMemsetAsync(counts)");
    if (rc) return rc;
    count_kept_kernel<<<dim3(L.nqt, HQ), 128, 0, st>>>(mq, reinterpret_cast<const uint32_t*>(ws + L.gbits),
                                                       s->Hq / s->Hkv, s->Hq, s->Hkv, s->n, s->window, s->K, L.nkt, out);
    return check_cuda(cudaGetLastError(), "count_kept kernel");
}

}  // namespace focus
