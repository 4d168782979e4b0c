// focus_build_tiles / focus_count_kept: integer-only passes over the membership masks.
//   summaries   OR/AND of the masks of each 128-token tile, per-group column bitmaps of key tiles
//   live set    far tile pairs whose OR summaries intersect (everything else far is skipped)
//   kept count  exact number of attended pairs per query head
#include "common.cuh"

namespace focus {

constexpr int TM = FOCUS_TILE_M;
constexpr int TN = FOCUS_TILE_N;
// Words of a query tile's live bitmap (32 key tiles of 128 tokens each) up to which it is made from the tiles' summaries at once;
// beyond, from the groups' words.  Whole call, at once / from the groups' words, 32 + 8 heads, top-2 of 4: 32768 tokens 16.3 and
// 17.6 us, 65536 32 and 32, 131072 80 and 59, 1048576 2706 and 443; the more groups the more loads a word takes: top-4 of 32,
// 65536 34 and 63, 131072 83 and 122, 262144 238 and 184.
constexpr int live_words(int K) { return K <= 8 ? 16 : 32; }

// A warp per (head, tile), so that no block barrier stands between the loads and the summaries and a block covers four tiles (a
// block per tile: 339 us for 40 heads x 1048576 tokens, 87 so).  The heads of the query masks, then those of the
// key masks (+ gbits).  The first warp clears the counters of the passes that follow.
__global__ void __launch_bounds__(128)
summarise_kernel(const uint32_t* mq, const uint32_t* mk, int HQ, int rows, int n, int nt, int K, uint32_t* orq,
                 uint32_t* andq, uint32_t* ork, uint32_t* andk, uint32_t* gbits,
                 unsigned long long* counters) {
    const int lane = threadIdx.x & 31;
    const long long id = (long long)blockIdx.x * 4 + (threadIdx.x >> 5);
    const int row = (int)(id / nt), tile = (int)(id % nt);
    const bool key = row >= HQ;
    const int head = key ? row - HQ : row;
    dep_wait();
    dep_trigger();
    if (row >= rows) return;
    if (id == 0 && lane < 8) counters[lane] = 0ull;
    const uint32_t* m = (key ? mk : mq) + (size_t)head * n;
    uint32_t v[4], o = 0u, a = 0xffffffffu;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const int tok = tile * 128 + q * 32 + lane;
        const bool in = tok < n;
        v[q] = in ? m[tok] : 0u;
        o |= v[q];
        a &= in ? v[q] : 0xffffffffu;
    }
    o = __reduce_or_sync(0xffffffffu, o);
    a = __reduce_and_sync(0xffffffffu, a);
    if (lane == 0) {
        (key ? ork : orq)[(size_t)head * nt + tile] = o;
        (key ? andk : andq)[(size_t)head * nt + tile] = a;
    }
    if (key) {
        uint4* gb = reinterpret_cast<uint4*>(gbits) + ((size_t)head * nt + tile) * K;
        for (int g = 0; g < K; ++g) {
            const uint4 w = make_uint4(__ballot_sync(0xffffffffu, (v[0] >> g) & 1u), __ballot_sync(0xffffffffu, (v[1] >> g) & 1u),
                                       __ballot_sync(0xffffffffu, (v[2] >> g) & 1u), __ballot_sync(0xffffffffu, (v[3] >> g) & 1u));
            if (lane == 0) gb[g] = w;
        }
    }
}

// One word of the bitmaps, per group g, of the key tiles that hold a member of g and of those that consist of members of g only.
// A warp; its lanes are the 32 key tiles.
__device__ __forceinline__ void group_words(const uint32_t* ork, const uint32_t* andk, int hk, int wd, int K, int nkt, int nkw, uint32_t* kany,
                                            uint32_t* kall) {
    const int lane = threadIdx.x & 31, b = wd * 32 + lane;
    const uint32_t o = b < nkt ? ork[(size_t)hk * nkt + b] : 0u, all = b < nkt ? andk[(size_t)hk * nkt + b] : 0u;
    for (int g = 0; g < K; ++g) {
        const uint32_t any_w = __ballot_sync(0xffffffffu, (o >> g) & 1u), all_w = __ballot_sync(0xffffffffu, (all >> g) & 1u);
        if (lane == 0) {
            kany[((size_t)hk * K + g) * nkw + wd] = any_w;
            kall[((size_t)hk * K + g) * nkw + wd] = all_w;
        }
    }
}

__global__ void __launch_bounds__(128)
group_tiles_kernel(const uint32_t* ork, const uint32_t* andk, int HK, int K, int nkt, int nkw, uint32_t* kany, uint32_t* kall) {
    const int id = blockIdx.x * 4 + (threadIdx.x >> 5);
    dep_wait();
    dep_trigger();
    if (id < HK * nkw) group_words(ork, andk, id / nkw, id % nkw, K, nkt, nkw, kany, kall);
}

// Live far-tile bitmap.  Key tile b is far for query tile a when every pair has i - j > w, i.e. b < (128 a - w) / 128;
// a far tile is live when the query tile's OR summary meets the key tile's, full when the AND summaries meet.  One block per
// (head, query tile).
// BY_GROUP: a thread per word, the OR over the groups of the query tile of the words group_tiles_kernel has left; 32 key tiles
// for a few loads, which is what counts when the bitmap is long.
// Otherwise a warp makes a word at a time, its lanes the 32 key tiles; the blocks past those of the HQ query heads, as many per KV
// head, write the groups' words meanwhile, so that a launch is saved.
template <bool BY_GROUP>
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
    if (!BY_GROUP && hq >= HQ) {
        for (int wd = a * 4 + warp; wd < nkw; wd += nqt * 4) group_words(ork, andk, hq - HQ, wd, K, nkt, nkw, kany, kall);
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
    if constexpr (BY_GROUP) {
        const uint32_t* any = kany + (size_t)hk * K * nkw;
        const uint32_t* all = kall + (size_t)hk * K * nkw;
        for (int wd = threadIdx.x; wd < nkw; wd += 128) {
            const int rem = nfar_tiles - wd * 32;
            uint32_t lv = 0, fl = 0;
            if (rem > 0) {
                for (uint32_t m = oq; m; m &= m - 1) lv |= any[(size_t)(__ffs(m) - 1) * nkw + wd];
                for (uint32_t m = aq; m; m &= m - 1) fl |= all[(size_t)(__ffs(m) - 1) * nkw + wd];
                const uint32_t far_mask = rem >= 32 ? 0xffffffffu : (1u << rem) - 1u;
                lv &= far_mask;
                fl &= far_mask;
            }
            row[wd] = lv;
            nlive += __popc(lv);
            nfull += __popc(fl);
        }
        nlive = __reduce_add_sync(0xffffffffu, nlive);
        nfull = __reduce_add_sync(0xffffffffu, nfull);
    } else {
        for (int wd = warp; wd < nkw; wd += 4) {
            const int b = wd * 32 + lane;
            const bool far = b < nfar_tiles;                          // (far tiles are all below nkt)
            const uint32_t lv = __ballot_sync(0xffffffffu, far && (oq & ork[(size_t)hk * nkt + b]) != 0u);
            const uint32_t fl = __ballot_sync(0xffffffffu, far && (aq & andk[(size_t)hk * nkt + b]) != 0u);
            if (lane == 0) row[wd] = lv;
            nlive += __popc(lv);
            nfull += __popc(fl);
        }
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
    int rc = check_cuda(launch_dependent(summarise_kernel, dim3((unsigned)((blocks + 3) / 4)), dim3(128), 0, st, mq, mk, HQ, HQ + HK, s->n, L.nqt, s->K,
                                         u32(L.orq), u32(L.andq), u32(L.ork), u32(L.andk), u32(L.gbits), counters), "summarise kernel launch");
    if (rc) return rc;
    const bool by_group = L.nkw > live_words(s->K);
    if (by_group) {
        const long long words = (long long)HK * L.nkw;
        if ((rc = check_cuda(launch_dependent(group_tiles_kernel, dim3((unsigned)((words + 3) / 4)), dim3(128), 0, st, u32(L.ork), u32(L.andk), HK, s->K,
                                              L.nkt, L.nkw, u32(L.kany), u32(L.kall)), "group tiles kernel launch"))) return rc;
    }
    rc = check_cuda(launch_dependent(by_group ? live_kernel<true> : live_kernel<false>, dim3((unsigned)(by_group ? (long long)HQ * L.nqt : blocks)),
                                     dim3(128), 0, st, u32(L.orq), u32(L.andq), u32(L.ork), u32(L.andk), s->Hq / s->Hkv, s->Hq, s->Hkv, HQ, s->window,
                                     s->K, L.nqt, L.nkt, L.nkw, u32(L.kany), u32(L.kall), u32(L.live),
                                     reinterpret_cast<int32_t*>(ws + L.live_cnt), counters), "live tiles kernel launch");
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
