// focus_attn_fwd for sm_100a: persistent, warp-specialised attention forward over the attended
// pairs of the Focus mask (paper Sec. 2 and Appendix D, first equation).
//
// One CTA per SM works through (head, 256-query block) items.  Per item, two 128-row query tiles
// share every key/value tile that is fetched:
//   warp 0        TMA producer: Q tiles once per item, then K and V tiles of every visited key tile
//                 into a ring of shared-memory stages (128-byte swizzle)
//   warp 1        MMA issuer: S_x = Q_x K^T and O_x += P_x V with tcgen05.mma, accumulators in TMEM
//                 (the whole warp runs the loop, one elected lane issues)
//   warps 4-7     softmax for query tile 0: tcgen05.ld S, mask, online max/sum, P (bf16) back to TMEM
//   warps 8-11    softmax for query tile 1
// After the split into roles the control warpgroup hands registers to the softmax warpgroups
// (setmaxnreg).  The two softmax groups alternate on the tensor pipe: while one computes exponentials
// the MMAs of the other run.  The running maximum is raised lazily (only when it grows by more than
// 2^8), and then the owner of the row rescales its O row in TMEM itself.
//
// Head dimension 256 does not leave room in TMEM for two query tiles (O alone is 256 columns), so
// there an item is a single 128-row query tile, S is double-buffered over consecutive key tiles
// and the two softmax warpgroups share every row, a thread to each half of the key tile's columns.
//
// Training-time soft gate, two query tiles: the factor of a distant pair is a function of g_i . g_j, and those products are
// an MMA as well.  For a pair of tiles that holds distant pairs G_x = g_q g_k^T goes to the place of S_x first, the softmax
// warps take it into registers and work out the 128 factors while S_x = Q_x K^T is computed over it; warps 2 and 3 write
// the operands (assignments split into bf16 terms).  Per key tile that leaves the softmax warps a tanh, a fused
// multiply-add and half a packed multiplication per pair, in place of K / 2 packed multiply-adds on 2 K / 4 shared-memory
// reads: 8192 tokens, K = 8, 32/8 heads: 1290 -> 862 us (742 with the shorter code below); 32768: 20.7 -> 13.5 ms.  At D = 256
// tensor memory and the ring leave one query tile, whose softmax warps evaluate the products themselves.
//
// Code size: 46 to 82 KB a kernel, from 65 to 118 (0.59 to 0.82 of what each was).  The roles run side by side and each streams
// through its own code once per tile: waits and their reports inlined at full length, loops the compiler unrolled by itself and
// divisions by launch parameters were instructions to issue and registers to hold, and lay between what is executed per tile.  Loops
// with short trip counts therefore say `unroll 1`, except the issue of a tile's MMAs, whose descriptors must be there when the tensor
// pipe is (rolled up: 1228 -> 1714 cycles from P to the next S).  Together with the epilogue in pieces of 16 columns and the lower
// halves of descriptors: 12 heads x 16384 tokens at D = 64 in dense mode: 614 -> 547 us; 65536 tokens at D = 256 class-sorted: 13.1 ->
// 12.0 ms; 32 heads x 8192 in token order: 551 -> 530 us, gated: 794 -> 707.  By the counters (8192 tokens, token order and gated, the
// hand-over of P in two parts included): 7 and 6 % fewer instructions, which waited for memory and tensor memory 0.95 -> 0.77 and
// 3.5 -> 2.9 cycles each; the wait for instructions was never large (0.32 -> 0.26 and 0.42 -> 0.40).
//
// Which key tiles are visited, and in which order of items:
//   dense mode      every tile up to the diagonal
//   original layout far tiles (every pair beyond the window) only when the live bitmap says the OR
//                   of the query-tile masks meets the OR of the key-tile masks; near tiles always
//   class-sorted    Q, K, V are the copies gathered into the class-sorted order; per key class the
//                   range of sorted key tiles listed for the query block; a row's kept columns of a
//                   tile are a contiguous range found from the tile's ascending positions; O and lse
//                   go straight to the rows' original positions
// In the last two the TMA thread alone walks; the other roles get the tiles, with what their masks are made from, through a
// ring in shared memory (TileInfo).
// The items are a queue, expensive ones first: the grid has one block per item, and a CTA that is through with its item
// takes over the next block that has not started (cluster launch control; the TMA thread asks, every role reads the
// answer from shared memory).  Dealing the items out beforehand, a fixed number per CTA, left the fullest CTA 18 % (one
// sequence of 8192), 27 % (three of 3001) and 4.5 % (131072) above the average.
#include "attn_common.cuh"
#include "tma_host.cuh"

namespace focus {

// GATE: 0 = no soft gate, else the number of 8-float chunks of a token's soft assignment (1, 2 or 4: K <= 8, 16, 32)
template <int D, int GATE = 0>
struct AttnCfg {
    static constexpr int NQ = (D == 256) ? 1 : 2;            // 128-row query tiles per item
    static constexpr int SUBT = D / 64;
    static constexpr uint32_t SUB_BYTES = 128 * 64 * 2;
    static constexpr uint32_t TILE_BYTES = SUB_BYTES * SUBT;
    // The K/V ring.  Up to D = 128 a stage holds a whole 128-key tile of K or of V.  At D = 256 only two such stages
    // would fit next to Q, so a tile travels as two half stages cut along the contraction dimension of its MMA (the
    // full-width MMA shapes stay): a K half is all 128 keys x 128 of the 256 head dimensions, a V half is 64 keys x
    // all 256 dimensions.  Five half stages fit, and a half goes back to the producer as soon as its own MMAs are done.
    static constexpr int PARTS = (D == 256) ? 2 : 1;         // ring stages per tile
    static constexpr uint32_t STAGE_BYTES = TILE_BYTES / PARTS;
    static constexpr int NSTAGE = (D == 256) ? (GATE ? 4 : 5)
                                             : ((D == 128) ? (GATE == 4 ? 2 : GATE == 2 ? 3 : GATE == 1 ? 4 : 5) : (GATE == 4 ? 6 : 8));
    // Soft gate, one query tile: per softmax warpgroup two buffers of 128 key assignments, 8 GATE floats each.
    static constexpr uint32_t GATE_ROW_BYTES = 32 * (GATE ? GATE : 1);
    static constexpr uint32_t GATE_BUF_BYTES = 128 * GATE_ROW_BYTES;
    static_assert(!(D == 256 && GATE == 4), "no room for the K/V ring beside 64 KB of gate buffers at D = 256");
    // Soft gate, two query tiles: the inner products of the assignments are an MMA of their own, G = g_q g_k^T.  Every
    // assignment is split into three bf16 terms (24 mantissa bits) and six of the nine products of terms are taken, those
    // above 2^-24.  An operand holds its terms side by side in column blocks of 8, 128 rows x 16 bytes each, no swizzle
    // (so that a 16-deep MMA can pair any two blocks); with 8 values per assignment the key side repeats its first term
    // as the fourth block, see gate_step.
    static constexpr bool GATE_MMA = GATE != 0 && NQ == 2;
    static constexpr int GATE_CH = GATE ? GATE : 1;                              // column blocks per term
    static constexpr uint32_t GBLK_BYTES = 128 * 16;
    static constexpr uint32_t GQ_BYTES = 3 * GATE_CH * GBLK_BYTES;               // one query tile
    static constexpr uint32_t GK_BYTES = (GATE == 1 ? 4 : 3 * GATE_CH) * GBLK_BYTES;     // one key tile, two buffers
    static constexpr uint32_t GATE_SMEM = GATE == 0 ? 0 : (NQ == 2 ? 2 * GQ_BYTES + 2 * GK_BYTES : 4 * GATE_BUF_BYTES);
    static constexpr int NINFO = (D == 256) ? 3 : 4;         // tiles handed on ahead (what fits beside the K/V ring)
    // shared memory: Q | K/V ring | gate operands | tile ring | row exchange | barriers
    static constexpr uint32_t OFF_GATE = NQ * TILE_BYTES + NSTAGE * STAGE_BYTES;
    static constexpr uint32_t OFF_INFO = OFF_GATE + GATE_SMEM;
    static constexpr uint32_t OFF_XVAL = OFF_INFO + (GATE ? 0 : NINFO * (uint32_t)sizeof(TileInfo));
    static constexpr uint32_t OFF_CTL = OFF_XVAL + (NQ == 1 ? 2 * 2 * 128 * 2 : 0);
    // Ring order of the tiles.  With one query tile the S of the next key tile is issued before the current P V, so
    // K(next) travels ahead of V(current); with two query tiles V(current) is consumed and released first.
    static constexpr bool K_AHEAD = NQ == 1;
    // Two query tiles, no gate: P is handed over in two parts, 96 columns and 32, so that most of P V runs while the last exponentials
    // are taken and what lies between the last of them and the next S is a quarter of P V and that S.  From P to the next S
    // 1250 -> 1000 cycles; 32 heads x 16384 tokens, dense: 1706 -> 1632 us, x 8192 in token order 530 -> 513, x 32768 class-sorted
    // 6.41 -> 6.24 ms; in halves 1654, 520 and 6.29.  With the gate nothing is gained (707 -> 706 us at 8192 tokens, 268 -> 275 at
    // D = 64): what is waited for there is G.
    static constexpr bool SPLIT_P = NQ == 2 && GATE == 0;
    static constexpr int P_FIRST = 96;
    static constexpr uint32_t COL_S0 = 0, COL_S1 = 128, COL_O0 = 256, COL_O1 = 256 + D;
    // With a single query tile two threads share a row: each of the two softmax warpgroups owns one 64-column
    // half of every key tile (its S columns, its P columns, its part of the row sum) and one half of the O row.
    static constexpr int NSPLIT = NQ == 1 ? 2 : 1;
    static constexpr int NC = 128 / NSPLIT;                  // S columns per softmax thread
    static constexpr int THREADS = 128 + 128 * NQ * NSPLIT;
    static constexpr int READERS = THREADS / 32 - 3 + (GATE_MMA ? 2 : 0);     // warps that read the queue: MMA, softmax, gate operands
    static constexpr int TILE_READERS = THREADS / 32 - 3;     // warps that read the tile ring: MMA, softmax
};

struct SharedCtl {
    uint64_t q_full, q_empty;
    uint64_t s_full[2], p_full[2], o_full[2];
    uint64_t p_rest[2];               // the second part of P (SPLIT_P)
    uint64_t pv_done;
    uint64_t xchg[4];                 // split rows, per 32-row quadrant: both column halves have published a per-row value
    uint64_t gbar[2];                 // soft gate, one query tile, per softmax warpgroup: the key assignments are in shared memory
    uint64_t kv_full[8], kv_empty[8];
    uint64_t info_full[4], info_empty[4];         // tile ring: handed on, read by TILE_READERS warps
    uint64_t next_full[2], next_empty[2];         // the answers below: arrived, read by the MMA warp and every softmax warp
    uint32_t limit;                   // how long a wait may last before the role gives up (wait_limit)
    uint32_t tmem_base;
    int abort_flag;
    uint32_t asked;                   // how many answers the TMA thread has asked for
    uint4 next[2];                    // which item comes next, by the parity of its ordinal
};

// soft gate, two query tiles (behind SharedCtl)
struct GateCtl {
    uint64_t gq_full, gq_empty, gk_full[2], gk_empty[2];      // operands of G written / read
    uint64_t g_full[2], g_taken[2];   // G of a query tile is in tensor memory / in the softmax warps' registers
};

// Bounded wait that also gives up when another role of the CTA has given up.  `gave_up` becomes `where`; the role reports it at its
// end (give_up), every lane that gave up, for the lanes of a warp may not all have.  Few instructions, for there are some thirty
// places (the note on code size above); the try in front of the loop is worth its own (D = 256, 16384 tokens dense: 1580 us without
// it, 1537 so).
__device__ __forceinline__ bool ctl_wait(uint64_t* bar, uint32_t parity, SharedCtl& ctl, int& gave_up, int where) {
    if (mbar_try_wait(smem_u32(bar), parity)) return true;          // (a try lasts until the phase completes, or about a millisecond)
    uint32_t t0 = 0;
#pragma unroll 1
    for (;;) {
        if (mbar_try_wait(smem_u32(bar), parity)) return true;
        const uint32_t now = wait_ticks(globaltimer_ns()) | 1u;
        if (t0 == 0) t0 = now;
        if (*(volatile int*)&ctl.abort_flag || wait_over(t0, now, ctl.limit)) break;
    }
    gave_up = where;
    return false;
}

__device__ __forceinline__ void give_up(const AttnParams& p, SharedCtl* ctl, int where, int query_block, uint32_t ord) {
    *(volatile int*)&ctl->abort_flag = 1;
    if (p.status && atomicCAS(p.status, 0, 1) == 0) {
        p.status[1] = where;
        p.status[2] = stalled_work(where, query_block, ord);
        p.status[3] = (int)blockIdx.x;
    }
}

// soft gate: does the pair of query tile a and key tile kb hold a distant pair
__device__ __forceinline__ bool gate_tile(const AttnParams& p, int a, int kb) {
    return kb <= a && a * 128 < p.n && a * 128 + 127 - p.w > kb * 128;
}

// One assignment row (8 CH floats, times `scale`) as three bf16 terms into row r of an operand of G: term t, columns 8 c .. at
// block t CH + c; with `again` the first term once more behind the third (CH = 1).
template <int CH>
__device__ __forceinline__ void put_gate_row(unsigned char* op, int r, const float* row, int ld, bool in, float scale, bool again) {
#pragma unroll
    for (int c = 0; c < CH; ++c) {
        float v[8];
#pragma unroll
        for (int f = 0; f < 2; ++f) {
            const bool have = in && 8 * c + 4 * f < ld;
            const float4 x = have ? dep_load(reinterpret_cast<const float4*>(row) + 2 * c + f) : make_float4(0.f, 0.f, 0.f, 0.f);
            v[4 * f] = x.x * scale; v[4 * f + 1] = x.y * scale; v[4 * f + 2] = x.z * scale; v[4 * f + 3] = x.w * scale;
        }
#pragma unroll
        for (int t = 0; t < 3; ++t) {
            uint32_t w[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                w[e] = pack_bf16x2(v[2 * e], v[2 * e + 1]);
                v[2 * e] -= __uint_as_float(w[e] << 16);
                v[2 * e + 1] -= __uint_as_float(w[e] & 0xffff0000u);
            }
            const uint4 x = make_uint4(w[0], w[1], w[2], w[3]);
            *reinterpret_cast<uint4*>(op + (t * CH + c) * 2048 + r * 16) = x;
            if (again && t == 0) *reinterpret_cast<uint4*>(op + (3 * CH + c) * 2048 + r * 16) = x;
        }
    }
}

// Step s of the MMA chain of G, the small products first: byte offset of the first column block of 8 and distance to the
// second, of each side.  CH = 1: a step takes two products at once (terms h, m, l; the key side h, m, l, h):
// (h l + l h), (h m + m h), (h h + m m).  CH > 1: one product of terms, 16 columns of it.
template <int CH> struct GateSteps {
    static constexpr int N = CH == 1 ? 3 : 6 * (CH / 2);
    struct Step { uint32_t a, a_lbo, b, b_lbo; };
    static __device__ __forceinline__ constexpr Step at(int s) {
        constexpr uint32_t B = 2048;
        if (CH == 1) return s == 0 ? Step{0, 2 * B, 2 * B, B} : s == 1 ? Step{0, B, B, 2 * B} : Step{0, B, 0, B};
        constexpr int H = CH > 1 ? CH / 2 : 1;              // steps per product
        const int pr = s / H, c = 2 * (s % H);
        const uint32_t ta = pr == 1 ? 2 : (pr == 2 || pr == 4) ? 1 : 0, tb = pr == 0 ? 2 : (pr == 2 || pr == 3) ? 1 : 0;
        return Step{(ta * CH + c) * B, B, (tb * CH + c) * B, B};
    }
};

// The CTA's item number `ord` (0, 1, ...): the block it was launched as, then what the answers say; false after the last.
// Called by every thread of a role's warp (`reader`: the warp reports that it has read), or by the TMA thread.
template <int WALK>
__device__ __forceinline__ bool next_item(const AttnParams& p, SharedCtl& ctl, uint32_t ord, bool reader, Item& t, int& gave_up) {
    uint32_t block = blockIdx.x;
    if (ord > 0) {
        const uint32_t slot = (ord - 1) & 1, use = (ord - 1) >> 1;
        if (!ctl_wait(&ctl.next_full[slot], use & 1, ctl, gave_up, WAIT_NEXT_ITEM)) return false;
        const bool more = clc_answer(smem_u32(&ctl.next[slot]), block);
        if (reader) {
            fence_proxy_async_smem();                   // the answer is read before the next one is written there
            __syncwarp();
            if ((threadIdx.x & 31) == 0) mbar_arrive(smem_u32(&ctl.next_empty[slot]));
        }
        if (!more) return false;
    }
    item_at<WALK>(p, (int)block, t);
    return true;
}

template <int D, bool SOFTCAP, int GATE, int WALK>
__global__ void __launch_bounds__(AttnCfg<D, GATE>::THREADS, 1)
focus_attn_kernel(const __grid_constant__ CUtensorMap tm_q, const __grid_constant__ CUtensorMap tm_k,
                  const __grid_constant__ CUtensorMap tm_v, const __grid_constant__ AttnParams p) {
    using C = AttnCfg<D, GATE>;
    constexpr int NQ = C::NQ;
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    SharedCtl& ctl = *reinterpret_cast<SharedCtl*>(smem_raw + C::OFF_CTL);
    GateCtl& gctl = *reinterpret_cast<GateCtl*>(smem_raw + C::OFF_CTL + sizeof(SharedCtl));
    // split rows: [parity][column half][row] row maxima, at the end row sums
    // (bf16: a rounded row maximum serves as well as the exact one as long as both threads use the same value)
    __nv_bfloat16* const xval_s = reinterpret_cast<__nv_bfloat16*>(smem_raw + C::OFF_XVAL);
    auto xval = [&](int par, int hf, int row) -> __nv_bfloat16& { return xval_s[(par * 2 + hf) * 128 + row]; };
    TileInfo* const info = reinterpret_cast<TileInfo*>(smem_raw + C::OFF_INFO);
    const uint32_t base = smem_u32(smem_raw);
    const uint32_t sq = base;                                 // NQ query tiles
    const uint32_t skv = base + NQ * C::TILE_BYTES;            // ring of K / V tiles
    unsigned char* const gate_sm = smem_raw + C::OFF_GATE;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

    if (WALK == WALK_SORTED) dep_wait();
    if (WALK == WALK_SORTED && dep_load(p.counters + 4) != 0ull) {      // more mask values than the sorted layout holds: refuse
        if (threadIdx.x == 0 && p.status && atomicCAS(p.status, 0, 2) == 0) {
            p.status[1] = 1; p.status[2] = 0; p.status[3] = (int)blockIdx.x;
        }
        return;
    }
    if (base & 1023u) {                                   // the operands' swizzle is a function of the address
        if (threadIdx.x == 0 && p.status && atomicCAS(p.status, 0, 1) == 0) {
            p.status[1] = 2; p.status[2] = 0; p.status[3] = (int)blockIdx.x;
        }
        return;
    }
    if (threadIdx.x == 0) {
        mbar_init(smem_u32(&ctl.q_full), 1);
        mbar_init(smem_u32(&ctl.q_empty), 1);
        mbar_init(smem_u32(&ctl.pv_done), 1);
        if constexpr (C::GATE_MMA) {
            mbar_init(smem_u32(&gctl.gq_full), 2);
            mbar_init(smem_u32(&gctl.gq_empty), 1);
        }
        for (int qd = 0; qd < 4; ++qd) mbar_init(smem_u32(&ctl.xchg[qd]), 2);
        for (int g = 0; g < 2; ++g) mbar_init(smem_u32(&ctl.gbar[g]), 4);
        for (int x = 0; x < 2; ++x) {
            mbar_init(smem_u32(&ctl.s_full[x]), 1);
            mbar_init(smem_u32(&ctl.p_full[x]), 128 * C::NSPLIT);
            mbar_init(smem_u32(&ctl.p_rest[x]), 128);
            mbar_init(smem_u32(&ctl.o_full[x]), 1);
        }
        for (int s = 0; s < C::NSTAGE; ++s) {
            mbar_init(smem_u32(&ctl.kv_full[s]), 1);
            mbar_init(smem_u32(&ctl.kv_empty[s]), 1);
        }
        for (int x = 0; x < C::NINFO; ++x) {
            mbar_init(smem_u32(&ctl.info_full[x]), 1);
            mbar_init(smem_u32(&ctl.info_empty[x]), C::TILE_READERS);
        }
        for (int x = 0; x < 2; ++x) {
            mbar_init(smem_u32(&ctl.next_full[x]), 1);
            mbar_init(smem_u32(&ctl.next_empty[x]), C::READERS);
            if constexpr (C::GATE_MMA) {
                mbar_init(smem_u32(&gctl.gk_full[x]), 2);
                mbar_init(smem_u32(&gctl.gk_empty[x]), 1);
                mbar_init(smem_u32(&gctl.g_full[x]), 1);
                mbar_init(smem_u32(&gctl.g_taken[x]), 4);
            }
        }
        ctl.abort_flag = 0;
        ctl.asked = 0;
        ctl.limit = wait_limit(p.wait_limit_ns);
        fence_mbar_init();
    }
    if (warp == 1) {
        tmem_alloc(smem_u32(&ctl.tmem_base), 512);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = ctl.tmem_base;
    if (WALK != WALK_SORTED) dep_wait();
    dep_trigger();

    if (warp < 4) reg_dec<REGS_CONTROL>();
    if (warp == 0) {
        // ------------------------------------------------------------------ TMA producer
        if (lane == 0) {
            prefetch_tmap(&tm_q); prefetch_tmap(&tm_k); prefetch_tmap(&tm_v);
            RingAt<C::NSTAGE> kv;
            RingAt<C::NINFO> handed;        // tiles handed on
            long long until_stall = p.stall_at;
            int it = 0;                     // items processed (items without key tiles are skipped by every role)
            int bad = 0;                    // where a wait gave up
            // ask for the item after number `ord`, when all of that one's loads are on their way
            auto ask_next = [&](uint32_t ord) {
                const uint32_t slot = ord & 1, use = ord >> 1;
                if (use > 0 && !ctl_wait(&ctl.next_empty[slot], (use - 1) & 1, ctl, bad, WAIT_NEXT_ROOM)) return;
                mbar_arrive_expect_tx(smem_u32(&ctl.next_full[slot]), 16);
                clc_try_cancel(smem_u32(&ctl.next[slot]), smem_u32(&ctl.next_full[slot]));
                ctl.asked = ord + 1;
            };
            Item t = {};
            uint32_t ord = 0;
            for (; !bad && next_item<WALK>(p, ctl, ord, false, t, bad); ++ord) {
                const int A = t.A, hq = t.hq, b = t.bb, h = t.h, hk = p.by_G.div(h);
                TileWalk<WALK> walk;
                walk.init(p, hq, A * NQ, NQ);
                int cls_at = -1;
                uint32_t cls = 0;
                // the next tile of the walk, handed on to the other roles
                auto next_tile = [&]() -> int {
                    const int kb = walk.next();
                    if constexpr (WALK != WALK_DENSE) {
                        const uint32_t slot = handed.slot;
                        if (!ctl_wait(&ctl.info_empty[slot], handed.phase ^ 1, ctl, bad, 12)) return -1;
                        handed.next();
                        const uint32_t bar = smem_u32(&ctl.info_full[slot]);
                        info[slot].kb = kb;
                        if (kb < 0) {
                            mbar_arrive(bar);
                        } else {
                            const int khead = b * p.Hkv + hk;
                            const void* src;
                            uint32_t bytes;
                            if constexpr (WALK == WALK_SORTED) {
                                if (walk.jk != cls_at) cls = dep_load(p.cls_k + (size_t)khead * FOCUS_MAX_CLASSES + (cls_at = walk.jk));
                                info[slot].cls = cls;
                                info[slot].pad[0] = (uint32_t)walk.jk;
                                src = p.perm_k + (size_t)khead * p.nkp + (size_t)kb * 128;
                                bytes = 512;
                            } else {
                                src = p.gbits + ((size_t)khead * p.nkt + kb) * p.K * 4;
                                bytes = (uint32_t)p.K * 16;
                            }
                            mbar_arrive_expect_tx(bar, bytes);
                            bulk_load(smem_u32(info[slot].data), src, bytes, bar);
                        }
                    }
                    return kb;
                };
                int kb = next_tile();
                if (bad) break;
                if (kb < 0) {
                    ask_next(ord);
                    if (bad) break;
                    continue;
                }
                if (it > 0 && !ctl_wait(&ctl.q_empty, (it - 1) & 1, ctl, bad, 10)) break;
                mbar_arrive_expect_tx(smem_u32(&ctl.q_full), NQ * C::TILE_BYTES);
                // in the sorted layout the copies are indexed [head of the batch][sorted slot]
                const int qh = WALK == WALK_SORTED ? hq : h, qb = WALK == WALK_SORTED ? 0 : b;
                const int kh = WALK == WALK_SORTED ? b * p.Hkv + hk : hk;
#pragma unroll 1
                for (int c = 0; c < NQ * C::SUBT; ++c)
                    tma_load_4d(sq + c * C::SUB_BYTES, &tm_q, smem_u32(&ctl.q_full), (c % C::SUBT) * 64, (A * NQ + c / C::SUBT) * 128, qh, qb);
                // one K or V tile into the next stage(s) of the ring: K tiles as all keys x D / PARTS dimensions, V tiles as
                // 128 / PARTS keys x all dimensions, in boxes of 64 columns
                auto load_tile = [&](bool is_v, int tile) {
                    const CUtensorMap* const tm = is_v ? &tm_v : &tm_k;
                    const int boxes = is_v ? C::SUBT : C::SUBT / C::PARTS;
                    const uint32_t box_bytes = is_v ? C::SUB_BYTES / C::PARTS : C::SUB_BYTES;
#pragma unroll 1
                    for (int part = 0; part < C::PARTS; ++part, kv.next()) {
                        if (until_stall-- == 0) continue;                  // diagnostic: this stage is never filled
                        if (!ctl_wait(&ctl.kv_empty[kv.slot], kv.phase ^ 1, ctl, bad, 11)) return;
                        const uint32_t bar = smem_u32(&ctl.kv_full[kv.slot]);
                        const int row = tile * 128 + (is_v ? part * (128 / C::PARTS) : 0), col = is_v ? 0 : part * boxes * 64;
                        mbar_arrive_expect_tx(bar, C::STAGE_BYTES);
#pragma unroll
                        for (int c = 0; c < boxes; ++c)
                            tma_load_4d(skv + kv.slot * C::STAGE_BYTES + c * box_bytes, tm, bar, col + c * 64, row, kh, qb);
                    }
                };
                // Step j: the K of tile j and the V of tile j - 1, in the order in which the MMA warp takes them: with two query tiles
                // V(current) is consumed and released before K(next); with one the S of the next tile is issued before the current P V
                int kb_v = -1;
                for (;;) {
#pragma unroll
                    for (int second = 0; second < 2; ++second) {
                        if (bad) break;
                        const bool is_v = C::K_AHEAD == (second != 0);
                        const int tile = is_v ? kb_v : kb;
                        if (tile >= 0) load_tile(is_v, tile);
                    }
                    if (bad || kb < 0) break;
                    kb_v = kb;
                    kb = next_tile();
                }
                if (!bad) ask_next(ord);
                if (bad) break;
                ++it;
            }
            if (bad) give_up(p, &ctl, bad, t.A, ord);
        }
        __syncwarp();
    } else if (warp == 1) {
        // ------------------------------------------------------------------ MMA issuer
        // The whole warp runs the loop (so that addresses and descriptors stay warp-uniform); one elected
        // lane issues the MMAs and commits.
        {
            constexpr uint32_t IDESC_S = idesc_bf16(128, 128, 0, 0);
            constexpr uint32_t IDESC_O = idesc_bf16(128, D, 0, 1);
            RingAt<C::NSTAGE> kv;
            uint32_t np = 0;                // two query tiles: key tiles whose P has been consumed
            RingAt<C::NINFO> taken;         // tiles taken from the ring
            uint32_t gs = 0, gp = 0;        // one query tile: S tiles issued / P tiles consumed (buffer = count & 1)
            uint32_t ngt[2] = {0, 0};       // soft gate: G tiles per query tile
            RingAt<2> gkey;                 // ... key operands taken
            int it = 0;
            int bad = 0;                    // where a wait gave up
            // lower halves of the operand descriptors (the upper ones are the same throughout)
            const uint32_t qdesc0 = (uint32_t)smem_desc_sw128(sq, 16, 1024);
            const uint32_t kdesc0 = (uint32_t)smem_desc_sw128(skv, 16, 1024);             // K tiles: K-major
            const uint32_t vdesc0 = (uint32_t)smem_desc_sw128(skv, C::SUB_BYTES / C::PARTS, 1024);     // V tiles: MN-major, 64-column chunks
            // S_x (+)= `steps` 16-deep steps of Q_x K^T from the first on, K from `kd` on
            auto s_steps = [&](uint32_t d, uint32_t qd, uint32_t kd, int steps, bool more) {
#pragma unroll
                for (int ks = 0; ks < steps; ++ks) {
                    const uint32_t off = (ks >> 2) * (C::SUB_BYTES >> 4) + (ks & 3) * 2;
                    umma_ss_lo(d, qd + off, kd + off, IDESC_S, more || ks > 0);
                }
            };
            // O (+)= 16-key steps of P V
            auto o_steps = [&](uint32_t d, uint32_t a, uint32_t vd, int steps, bool more) {
#pragma unroll
                for (int ks = 0; ks < steps; ++ks) umma_ts_lo(d, a + ks * 8, vd + ks * 128, IDESC_O, more || ks > 0);
            };
            // soft gate: G_x = g_q g_k^T into the place of S_x, if the pair of tiles holds a distant pair; returns when the softmax
            // warps have it in registers
            auto issue_gate = [&](int x, int a0, int kb) -> bool {
                if constexpr (C::GATE_MMA) {
                    const bool g0 = gate_tile(p, a0, kb), g1 = gate_tile(p, a0 + 1, kb);
                    if (!(x ? g1 : g0)) return true;       // (a gated tile 0 without a gated tile 1 gives the key operand back itself)
                    const uint32_t buf = gkey.slot;
                    if (!ctl_wait(&gctl.gk_full[buf], gkey.phase, ctl, bad, 53)) return false;
                    tc_fence_after();
                    if (elect_one()) {
                        using Steps = GateSteps<C::GATE_CH>;
                        const uint32_t qa = sq + C::OFF_GATE + x * C::GQ_BYTES, ka = sq + C::OFF_GATE + 2 * C::GQ_BYTES + buf * C::GK_BYTES;
#pragma unroll
                        for (int st = 0; st < Steps::N; ++st)
                            umma_ss(tmem + (x ? C::COL_S1 : C::COL_S0), smem_desc_plain(qa + Steps::at(st).a, Steps::at(st).a_lbo, 128),
                                    smem_desc_plain(ka + Steps::at(st).b, Steps::at(st).b_lbo, 128), IDESC_S, st > 0);
                        umma_commit(smem_u32(&gctl.g_full[x]));
                        if (x == 1 || !g1) umma_commit(smem_u32(&gctl.gk_empty[buf]));
                    }
                    __syncwarp();
                    if (x == 1 || !g1) gkey.next();
                    const uint32_t par = (x ? ngt[1]++ : ngt[0]++) & 1;
                    if (!ctl_wait(&gctl.g_taken[x], par, ctl, bad, 54)) return false;
                    tc_fence_after();
                }
                return true;
            };
            auto commit = [&](uint64_t* bar) {
                if (elect_one()) umma_commit(smem_u32(bar));
            };
            // wait for the next tile of the ring
            auto wait_kv = [&](int& slot, int where) -> bool {
                slot = (int)kv.slot;
                if (!ctl_wait(&ctl.kv_full[slot], kv.phase, ctl, bad, where)) return false;
                kv.next();
                return true;
            };
            // One query tile: S[buf] = Q K^T and O (+)= P[buf] V stage by stage -- wait for the stage, issue the MMAs that
            // read it, hand it back.  The stages are taken in the ring's order: K(next) before V(current).
            auto s_tile = [&](int buf) -> bool {
                constexpr int KS = D / 16 / C::PARTS;            // k-steps per stage
#pragma unroll
                for (int part = 0; part < C::PARTS; ++part) {
                    int slot;
                    if (!wait_kv(slot, 21)) return false;
                    tc_fence_after();
                    if (elect_one()) {
                        s_steps(tmem + (buf ? C::COL_S1 : C::COL_S0), qdesc0 + part * (KS / 4) * (C::SUB_BYTES >> 4), kdesc0 + slot * (C::STAGE_BYTES >> 4), KS, part > 0);
                        umma_commit(smem_u32(&ctl.kv_empty[slot]));
                        if (part == C::PARTS - 1) umma_commit(smem_u32(&ctl.s_full[buf]));
                    }
                }
                return true;
            };
            auto o_tile = [&](int buf, bool first) -> bool {
#pragma unroll
                for (int part = 0; part < C::PARTS; ++part) {
                    int slot;
                    if (!wait_kv(slot, 22)) return false;
                    tc_fence_after();
                    if (elect_one()) {
                        // split rows: the P of column half h sits at columns 64 h .. 64 h + 31
                        o_steps(tmem + C::COL_O0, tmem + (buf ? C::COL_S1 : C::COL_S0) + part * 64, vdesc0 + slot * (C::STAGE_BYTES >> 4), 8 / C::PARTS, !first || part > 0);
                        umma_commit(smem_u32(&ctl.kv_empty[slot]));
                    }
                }
                return true;
            };
            Item t = {};
            uint32_t ord = 0;
            for (; !bad && next_item<WALK>(p, ctl, ord, true, t, bad); ++ord) {
                const int A = t.A, hq = t.hq;
                TileWalk<WALK> walk;
                if constexpr (WALK == WALK_DENSE) walk.init(p, hq, A * NQ, NQ);
                auto next_tile = [&]() -> int {
                    if constexpr (WALK == WALK_DENSE) {
                        return walk.next();
                    } else {
                        const uint32_t slot = taken.slot;
                        if (!ctl_wait(&ctl.info_full[slot], taken.phase, ctl, bad, 27)) return -1;
                        const int kb = info[slot].kb;
                        __syncwarp();
                        if (lane == 0) mbar_arrive(smem_u32(&ctl.info_empty[slot]));
                        taken.next();
                        return kb;
                    }
                };
                // Steps of the item: step j issues the P V of tile j - 1 and the S of tile j, so the first has no P V and the last no S.
                // Two query tiles: P V_0, S_0, P V_1, S_1, so that one tile's softmax runs during the other's MMAs.  One query tile: S of
                // the next tile goes to the other buffer before the P V.
                bool have_p = false, first = true;
                for (;;) {
                    const int kb = next_tile();
                    if (bad) break;
                    if (kb < 0 && !have_p) break;          // an item without key tiles
                    if (!have_p) {
                        if (!ctl_wait(&ctl.q_full, it & 1, ctl, bad, 20)) break;
                        if constexpr (C::GATE_MMA) {
                            if (!ctl_wait(&gctl.gq_full, it & 1, ctl, bad, 29)) break;
                        }
                    }
                    if constexpr (NQ == 2) {
                        // the ring carries V(current) ahead of K(next) (see the producer)
                        int vslot = 0, kslot = 0;
                        if (have_p && !wait_kv(vslot, 22)) break;
                        if (kb >= 0) {
                            if (!wait_kv(kslot, 23)) break;
                        } else {                           // every S (and G) of this item has been issued
                            commit(&ctl.q_empty);
                            if constexpr (C::GATE_MMA) commit(&gctl.gq_empty);
                        }
#pragma unroll
                        for (int x = 0; x < 2; ++x) {
                            if (have_p && !ctl_wait(&ctl.p_full[x], np & 1, ctl, bad, 24 + x)) break;
                            tc_fence_after();
                            const uint32_t t_s = tmem + (x ? C::COL_S1 : C::COL_S0);
                            const uint32_t t_o = tmem + (x ? C::COL_O1 : C::COL_O0), vd = vdesc0 + vslot * (C::STAGE_BYTES >> 4);
                            constexpr int STEPS1 = C::SPLIT_P ? C::P_FIRST / 16 : 0;      // of the 8 steps of P V
                            if constexpr (C::SPLIT_P) {
                                if (have_p) {
                                    if (elect_one()) o_steps(t_o, t_s, vd, STEPS1, !first);
                                    __syncwarp();
                                    if (!ctl_wait(&ctl.p_rest[x], np & 1, ctl, bad, 44 + x)) break;
                                    tc_fence_after();
                                }
                            }
                            if (have_p && elect_one()) {
                                o_steps(t_o, t_s + STEPS1 * 8, vd + STEPS1 * 128, 8 - STEPS1, !first || C::SPLIT_P);
                                if (x == 1) umma_commit(smem_u32(&ctl.kv_empty[vslot]));
                                if (kb < 0) umma_commit(smem_u32(&ctl.o_full[x]));
                            }
                            __syncwarp();
                            if (kb < 0) continue;
                            if (!issue_gate(x, A * NQ, kb)) break;
                            if (elect_one()) {
                                s_steps(t_s, qdesc0 + x * (C::TILE_BYTES >> 4), kdesc0 + kslot * (C::STAGE_BYTES >> 4), D / 16, false);
                                umma_commit(smem_u32(&ctl.s_full[x]));
                                if (x == 1) umma_commit(smem_u32(&ctl.kv_empty[kslot]));
                            }
                            __syncwarp();
                        }
                        if (bad) break;
                        if (have_p) { ++np; first = false; }
                    } else {
                        if (kb >= 0) {
                            if (!s_tile(gs & 1)) break;
                            ++gs;
                        } else {
                            commit(&ctl.q_empty);
                        }
                        if (have_p) {
                            const int buf = gp & 1;
                            if (!ctl_wait(&ctl.p_full[buf], (gp >> 1) & 1, ctl, bad, 26)) break;
                            ++gp;
                            tc_fence_after();
                            if (!o_tile(buf, first)) break;
                            commit(&ctl.pv_done);
                            if (kb < 0) commit(&ctl.o_full[0]);
                            first = false;
                        }
                    }
                    if (kb < 0) { ++it; break; }
                    have_p = true;
                }
            }
            if (bad) give_up(p, &ctl, bad, t.A, ord);
        }
        __syncwarp();
    } else if (C::GATE_MMA && warp < 4) {
        // ------------------------------------------------------------------ soft gate: operands of G
        const int t64 = threadIdx.x - 64;
        unsigned char* const gq = smem_raw + C::OFF_GATE;
        unsigned char* const gk = gq + 2 * C::GQ_BYTES;
        RingAt<2> gkey;
        int it = 0;
        int bad = 0;                        // where a wait gave up
        Item t = {};
        uint32_t ord = 0;
        for (; !bad && next_item<WALK>(p, ctl, ord, true, t, bad); ++ord) {
            const int a0 = t.A * NQ;
            TileWalk<WALK_DENSE> walk;
            walk.init(p, t.hq, a0, NQ);
            int kb = walk.next();
            if (kb < 0) continue;
            const float* gseq = p.gate_g + (size_t)t.bb * p.n * p.gate_ld;
            if (it > 0 && !ctl_wait(&gctl.gq_empty, (it - 1) & 1, ctl, bad, 55)) break;
#pragma unroll 1
            for (int r = t64; r < 256; r += 64) {
                const int i = a0 * 128 + r;
                put_gate_row<C::GATE_CH>(gq + (r >> 7) * C::GQ_BYTES, r & 127, gseq + (size_t)min(i, p.n - 1) * p.gate_ld, p.gate_ld, i < p.n, p.gate_hl, false);
            }
            fence_proxy_async_smem();
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_u32(&gctl.gq_full));
            for (; kb >= 0; kb = walk.next()) {
                if (!gate_tile(p, a0, kb) && !gate_tile(p, a0 + 1, kb)) continue;
                const uint32_t buf = gkey.slot;
                if (!ctl_wait(&gctl.gk_empty[buf], gkey.phase ^ 1, ctl, bad, 56)) break;
                gkey.next();
#pragma unroll 1
                for (int r = t64; r < 128; r += 64) {
                    const int j = kb * 128 + r;
                    put_gate_row<C::GATE_CH>(gk + buf * C::GK_BYTES, r, gseq + (size_t)min(j, p.n - 1) * p.gate_ld, p.gate_ld, j < p.n, 1.f, C::GATE_CH == 1);
                }
                fence_proxy_async_smem();
                __syncwarp();
                if (lane == 0) mbar_arrive(smem_u32(&gctl.gk_full[buf]));
            }
            ++it;
        }
        if (bad) give_up(p, &ctl, bad, t.A, ord);
        __syncwarp();
    } else if (warp >= 4) {
        // ------------------------------------------------------------------ softmax + epilogue
        reg_inc<REGS_SOFTMAX_2WG>();
        constexpr int NSPLIT = C::NSPLIT, NC = C::NC;
        const int wg = (warp - 4) >> 2;
        const int x = NSPLIT == 2 ? 0 : wg;                  // query tile of this warpgroup
        const int half = NSPLIT == 2 ? wg : 0;               // split rows: its column half of every key tile
        const int row_in_tile = ((warp & 3) << 5) | lane;
        const uint32_t lane_base = (uint32_t)((warp & 3) * 32) << 16;
        const uint32_t t_o = tmem + lane_base + (x ? C::COL_O1 : C::COL_O0) + half * (D / 2);   // its part of the O row
        uint32_t nx = 0;                                     // split rows: exchanges done with the partner half
        // logits in log2 units: sl2 * S, or with a softcap sl2 * tanh(cap_in * S)
        const float sl2 = SOFTCAP ? p.softcap * LOG2E : p.scale * LOG2E;
        const float cap_in = SOFTCAP ? p.scale / p.softcap : 0.f;
        uint32_t ns = 0;                                     // S tiles consumed by this warpgroup
        RingAt<C::NINFO> taken;                              // tiles taken from the ring
        uint32_t ng = 0;                                     // soft gate: tiles whose key assignments this warpgroup has staged
        int it = 0;
        int bad = 0;                                         // where a wait gave up
        // Each turn finds the next item, writes the one before out and then goes through the tiles.  An item's row position and mask
        // are loaded while the item before it ends, so that its first tile need not wait for them (three dependent reads of L2 in
        // the sorted order): its order entry before the wait for the last P V, the mask word before the output is written.
        Item t = {};
        int i = -1;                                          // the row's position in the sequence
        bool valid = false;
        float m_used = -INFINITY, l = 0.f;
        bool finish = false;                                 // an item whose tiles are through
        uint32_t ord = 0;
        for (;; ++ord) {
            Item t_next = {};
            const bool have = next_item<WALK>(p, ctl, ord, true, t_next, bad);
            if (bad) break;
            int i_next = -1;
            uint32_t mi = 0;
            if (have) {
                // its index, or in the sorted layout the position its slot holds (-1: padding)
                i_next = (t_next.A * NQ + x) * 128 + row_in_tile;
                if constexpr (WALK == WALK_SORTED) i_next = dep_load(p.perm_q + (size_t)t_next.hq * p.nqp + i_next);
            }
            auto load_mask = [&]() {
                if constexpr (WALK != WALK_DENSE) mi = (i_next >= 0 && i_next < p.n) ? dep_load(p.mq + (size_t)t_next.hq * p.n + i_next) : 0u;
            };
            if (finish) {
                // ---- epilogue: O / l -> bf16 -> global, lse.  With a partial result to join (window pass of the split layout) the
                // row's logsumexp there is read now, before a thread that shares the row can write the joint one.
                const size_t row = (size_t)t.hq * p.n + (size_t)i;
                float lse_other = -INFINITY;
                if (WALK == WALK_TOKEN && p.join && valid) lse_other = p.lse[row];
                if constexpr (NSPLIT == 2) {
                    // the two halves add their row sums: two exchanges, the leading bf16 part of the sum and its remainder
                    float other = 0.f, rest = l;
                    bool xok = true;
                    for (int piece = 0; piece < 2 && xok; ++piece) {
                        const int par = (int)(nx & 1);
                        const __nv_bfloat16 mine = __float2bfloat16_rn(rest);
                        rest -= __bfloat162float(mine);
                        xval(par, half, row_in_tile) = mine;
                        __syncwarp();
                        if (lane == 0) mbar_arrive(smem_u32(&ctl.xchg[warp & 3]));
                        xok = ctl_wait(&ctl.xchg[warp & 3], (uint32_t)par, ctl, bad, 38);
                        other += __bfloat162float(xval(par, half ^ 1, row_in_tile));
                        ++nx;
                    }
                    if (!xok) break;
                    l += other;
                }
                if (!ctl_wait(&ctl.o_full[x], it & 1, ctl, bad, 40 + x)) break;
                tc_fence_after();
                load_mask();
                const float inv_l = l > 0.f ? 1.f / l : 0.f;        // a row without any pair (possible in a partial pass): zeros, lse = -inf
                float own = inv_l, w_other = 0.f, lse_row = (m_used + lg2_approx(l)) * LN2;
                if (WALK == WALK_TOKEN && p.join) {
                    // the two partial results cover disjoint sets of pairs and join through their logsumexps (Appendix D)
                    const float m = fmaxf(lse_other, lse_row);
                    const float wo = m == -INFINITY ? 0.f : __expf(lse_other - m), wl = m == -INFINITY ? 0.f : __expf(lse_row - m);
                    const float tot = wo + wl, inv = tot > 0.f ? 1.f / tot : 0.f;
                    own = inv_l * wl * inv;
                    w_other = wo * inv;
                    lse_row = tot > 0.f ? m + __logf(tot) : -INFINITY;
                }
                __nv_bfloat16* orow = p.o + (size_t)t.bb * p.o_sb + (size_t)t.h * p.o_sh + (size_t)(valid ? i : 0) * p.o_sn +
                                      half * (D / 2);
#pragma unroll 1
                for (int c = 0; c < D / 16 / NSPLIT; ++c) {
                    uint32_t ov[16];
                    tmem_ld16(t_o + c * 16, ov);
                    tmem_wait_ld();
#pragma unroll
                    for (int e = 0; e < 16; ++e) ov[e] = __float_as_uint(__uint_as_float(ov[e]) * own);
                    const size_t at = row * D + half * (D / 2) + c * 16;
                    if constexpr (WALK == WALK_TOKEN) {
                        if (w_other > 0.f) {               // (a partial result without any pair has unspecified contents)
#pragma unroll
                            for (int e = 0; e < 16; e += 4) {
                                const float4 v4 = *reinterpret_cast<const float4*>(p.join + at + e);
                                ov[e] = __float_as_uint(fmaf(v4.x, w_other, __uint_as_float(ov[e])));
                                ov[e + 1] = __float_as_uint(fmaf(v4.y, w_other, __uint_as_float(ov[e + 1])));
                                ov[e + 2] = __float_as_uint(fmaf(v4.z, w_other, __uint_as_float(ov[e + 2])));
                                ov[e + 3] = __float_as_uint(fmaf(v4.w, w_other, __uint_as_float(ov[e + 3])));
                            }
                        }
                    }
                    if (!valid) continue;
                    if (WALK == WALK_SORTED && p.o32) {
#pragma unroll
                        for (int e = 0; e < 16; e += 8) {
                            uint32_t w[8];
#pragma unroll
                            for (int j = 0; j < 8; ++j) w[j] = ov[e + j];
                            st_global_v8(p.o32 + at + e, w);
                        }
                    } else {
                        uint32_t w[8];
#pragma unroll
                        for (int j = 0; j < 8; ++j) w[j] = pack_bf16x2(__uint_as_float(ov[2 * j]), __uint_as_float(ov[2 * j + 1]));
                        if (p.o_wide) {
                            st_global_v8(orow + c * 16, w);
                        } else {
                            *reinterpret_cast<uint4*>(orow + c * 16) = make_uint4(w[0], w[1], w[2], w[3]);
                            *reinterpret_cast<uint4*>(orow + c * 16 + 8) = make_uint4(w[4], w[5], w[6], w[7]);
                        }
                    }
                }
                if (valid && half == 0) p.lse[row] = lse_row;
                tc_fence_before();
                ++it;
            } else {
                load_mask();
            }
            if (!have) break;
            t = t_next;
            i = i_next;
            valid = i >= 0 && i < p.n;
            const int A = t.A, hq = t.hq, bb = t.bb;
            const int hk = bb * p.Hkv + p.by_G.div(t.h);
            const int a = A * NQ + x;
            TileWalk<WALK> walk;
            if constexpr (WALK == WALK_DENSE) walk.init(p, hq, A * NQ, NQ);
            const TileInfo* tile = nullptr;
            auto next_tile = [&]() -> int {
                if constexpr (WALK == WALK_DENSE) {
                    return walk.next();
                } else {
                    if (!ctl_wait(&ctl.info_full[taken.slot], taken.phase, ctl, bad, 39)) return -1;
                    tile = info + taken.slot;
                    return tile->kb;
                }
            };
            auto tile_read = [&]() {                     // the warp is through with what the ring says of the tile
                if constexpr (WALK != WALK_DENSE) {
                    __syncwarp();
                    if (lane == 0) mbar_arrive(smem_u32(&ctl.info_empty[taken.slot]));
                    taken.next();
                }
            };
            int wmin = 0, wmax = 0;
            if constexpr (WALK == WALK_SORTED) {
                wmin = __reduce_min_sync(0xffffffffu, i < 0 ? 0x7fffffff : i);
                wmax = __reduce_max_sync(0xffffffffu, i);
            }
            if (WALK == WALK_TOKEN) mi &= 0xffffffffu >> (32 - p.K);
            const int dfar = a * 128 - p.w;
            const int f_x = (WALK == WALK_TOKEN && dfar > 0) ? dfar >> 7 : 0;   // tiles b < f_x are far for this query tile
            m_used = -INFINITY;
            l = 0.f;
            bool first = true;
            // soft gate: this row's assignment times lambda / 2 (sigmoid(x) = 1/2 + 1/2 tanh(x / 2))
            constexpr bool GATE_ALU = GATE != 0 && !C::GATE_MMA;  // one query tile: the inner products are taken here
            constexpr int GQ = GATE_ALU ? 2 * GATE : 2;           // 16-byte pieces of an assignment row held per token
            float gi[4 * GQ];
#pragma unroll
            for (int e = 0; e < 4 * GQ; ++e) gi[e] = 0.f;
            if constexpr (GATE_ALU) {
                if (valid) {
                    const float4* gp = reinterpret_cast<const float4*>(p.gate_g + ((size_t)bb * p.n + (size_t)i) * p.gate_ld);
#pragma unroll
                    for (int f = 0; f < GQ; ++f) {
                        if (4 * f < p.gate_ld) {
                            const float4 g0 = dep_load(gp + f);
                            gi[4 * f] = g0.x * p.gate_hl; gi[4 * f + 1] = g0.y * p.gate_hl;
                            gi[4 * f + 2] = g0.z * p.gate_hl; gi[4 * f + 3] = g0.w * p.gate_hl;
                        }
                    }
                }
            }
#pragma unroll 1
            for (;;) {
                const int kb = next_tile();
                if (kb < 0) break;
                TileMask tm;
                if constexpr (WALK == WALK_SORTED) {
                    const bool share = (mi & tile->cls) != 0u;
                    build_tile_mask_sorted(tm, p.w, reinterpret_cast<const int32_t*>(tile->data), share, valid ? i : -1, wmin, wmax, !p.share_only);
                    if (p.gbits_s)
                        exclude_lower_groups(tm, p.gbits_s + ((size_t)hk * (p.nkp / 128) + kb) * p.K * 4, mi & ((1u << tile->pad[0]) - 1u), p.K);
                } else if constexpr (WALK == WALK_DENSE) {
                    build_tile_mask_dense(tm, a, kb, i);
                } else {
                    build_tile_mask(tm, p, a, kb, i, mi, f_x, tile->data);
                }
                tile_read();
                // ---- soft gate (Eq. 2): the score of a distant pair (i - j > w) is multiplied by sigmoid(lambda g_i . g_j).
                // The warpgroup stages the key assignments of its columns in shared memory before S is needed; every
                // thread then reads them with broadcast 16-byte loads, column by column.
                const unsigned char* gb = nullptr;
                bool gated = false;
                const int gj0 = kb * 128 + half * NC;    // first column of this thread's part of the tile
                const int ifar = i - p.w;                           // columns j < ifar are distant for this row
                const bool tile_gated = C::GATE_MMA && gate_tile(p, a, kb);
                if constexpr (GATE_ALU) {
                    // the same decision in all four warps of the warpgroup: does the tile hold a distant pair at all
                    const bool tile_gated = a * 128 + 127 - p.w > gj0;
                    if (tile_gated) {
                        unsigned char* gw = gate_sm + (wg * 2 + (ng & 1)) * C::GATE_BUF_BYTES;
                        const int col = (warp & 3) * 32 + lane;
                        if (col < NC) {
                            const int j = gj0 + col;
                            const float4* gp = reinterpret_cast<const float4*>(p.gate_g + ((size_t)bb * p.n + (size_t)(j < p.n ? j : p.n - 1)) * p.gate_ld);
#pragma unroll
                            for (int f = 0; f < GQ; ++f)
                                reinterpret_cast<float4*>(gw + col * C::GATE_ROW_BYTES)[f] = 4 * f < p.gate_ld ? dep_load(gp + f) : make_float4(0.f, 0.f, 0.f, 0.f);
                        }
                        __syncwarp();
                        if (lane == 0) mbar_arrive(smem_u32(&ctl.gbar[wg]));
                        if (!ctl_wait(&ctl.gbar[wg], ng & 1, ctl, bad, 37)) break;
                        ++ng;
                        gb = gw;
                        gated = __any_sync(0xffffffffu, valid && ifar > gj0);
                    }
                }
                // ---- two query tiles: G first, its factors computed while S is
                uint32_t sr[NC];
                if constexpr (C::GATE_MMA) {
                    if (tile_gated) {
                        if (!ctl_wait(&gctl.g_full[x], ng & 1, ctl, bad, 37)) break;
                        ++ng;
                        tc_fence_after();
                        const uint32_t t_g = tmem + lane_base + (x ? C::COL_S1 : C::COL_S0);
#pragma unroll
                        for (int c = 0; c < NC / 32; ++c) tmem_ld32(t_g + c * 32, *reinterpret_cast<uint32_t(*)[32]>(&sr[c * 32]));
                        tmem_wait_ld();
                        tc_fence_before();
                        __syncwarp();
                        if (lane == 0) mbar_arrive(smem_u32(&gctl.g_taken[x]));
                        const int nfar = ifar - gj0;                    // columns < nfar are distant
                        if (__any_sync(0xffffffffu, nfar < NC)) {
#pragma unroll
                            for (int c = 0; c < NC; ++c) sr[c] = c < nfar ? sr[c] : 0x7f800000u;        // tanh(inf) = 1: factor 1
                        }
#pragma unroll
                        for (int c = 0; c < NC; ++c) sr[c] = __float_as_uint(fmaf(tanh_approx(__uint_as_float(sr[c])), 0.5f, 0.5f));
                    }
                }
                // ---- wait for S
                const int buf = NQ == 2 ? x : (int)(ns & 1);
                const uint32_t par = NQ == 2 ? (ns & 1) : ((ns >> 1) & 1);
                if (!ctl_wait(&ctl.s_full[buf], par, ctl, bad, 30 + x)) break;
                // this thread's NC S columns; its packed P columns overwrite the first half of them
                const uint32_t t_s = tmem + lane_base + (buf ? C::COL_S1 : C::COL_S0) + half * NC;
                tc_fence_after();
                uint32_t pk[NC / 2];
                if (tile_gated) {                    // the factors are in place of the scores
#pragma unroll
                    for (int c = 0; c < NC / 16; ++c) {      // 16 at a time beside the 128 factors (8192 tokens: 742 us, 802 with 32)
                        uint32_t sv[16];
                        tmem_ld16(t_s + c * 16, sv);
                        tmem_wait_ld();
#pragma unroll
                        for (int e = 0; e < 16; e += 2) {
                            const float2 f = __fmul2_rn(make_float2(__uint_as_float(sr[c * 16 + e]), __uint_as_float(sr[c * 16 + e + 1])),
                                                        make_float2(__uint_as_float(sv[e]), __uint_as_float(sv[e + 1])));
                            sr[c * 16 + e] = __float_as_uint(f.x);
                            sr[c * 16 + e + 1] = __float_as_uint(f.y);
                        }
                    }
                } else
#pragma unroll
                for (int c = 0; c < NC / 32; ++c) {
                    tmem_ld32(t_s + c * 32, *reinterpret_cast<uint32_t(*)[32]>(&sr[c * 32]));
                    if constexpr (GATE_ALU) {        // chunk by chunk: 32 scores, then their factors
                        tmem_wait_ld();
                        if (gated) {
                            const bool wide = p.gate_ld == 8;
                            const int nfar = ifar - gj0 < 0 ? 0 : (ifar - gj0 > NC ? NC : ifar - gj0);   // columns < nfar are distant
#pragma unroll
                            for (int e0 = 0; e0 < 32; e0 += 4) {        // four columns in flight
                                float arg[4];
                                if constexpr (GATE == 1) {
                                    float4 k0[4], k1[4];
#pragma unroll
                                    for (int u = 0; u < 4; ++u) {
                                        const float4* kp = reinterpret_cast<const float4*>(gb + (c * 32 + e0 + u) * 32);
                                        k0[u] = kp[0];
                                        k1[u] = wide ? kp[1] : make_float4(0.f, 0.f, 0.f, 0.f);
                                    }
#pragma unroll
                                    for (int u = 0; u < 4; ++u) {
                                        float2 acc = __fmul2_rn(make_float2(gi[0], gi[1]), make_float2(k0[u].x, k0[u].y));
                                        acc = __ffma2_rn(make_float2(gi[2], gi[3]), make_float2(k0[u].z, k0[u].w), acc);
                                        if (wide) {
                                            float2 acb = __fmul2_rn(make_float2(gi[4], gi[5]), make_float2(k1[u].x, k1[u].y));
                                            acb = __ffma2_rn(make_float2(gi[6], gi[7]), make_float2(k1[u].z, k1[u].w), acb);
                                            acc = __fadd2_rn(acc, acb);
                                        }
                                        arg[u] = acc.x + acc.y;
                                    }
                                } else {
                                    // longer assignments: piece by piece, two sums per column
                                    float2 acc[4], acb[4];
#pragma unroll
                                    for (int u = 0; u < 4; ++u) acc[u] = acb[u] = make_float2(0.f, 0.f);
#pragma unroll
                                    for (int f = 0; f < GQ; ++f) {
                                        float4 kf[4];
#pragma unroll
                                        for (int u = 0; u < 4; ++u)
                                            kf[u] = reinterpret_cast<const float4*>(gb + (c * 32 + e0 + u) * C::GATE_ROW_BYTES)[f];
#pragma unroll
                                        for (int u = 0; u < 4; ++u) {
                                            acc[u] = __ffma2_rn(make_float2(gi[4 * f], gi[4 * f + 1]), make_float2(kf[u].x, kf[u].y), acc[u]);
                                            acb[u] = __ffma2_rn(make_float2(gi[4 * f + 2], gi[4 * f + 3]), make_float2(kf[u].z, kf[u].w), acb[u]);
                                        }
                                    }
#pragma unroll
                                    for (int u = 0; u < 4; ++u) arg[u] = (acc[u].x + acc[u].y) + (acb[u].x + acb[u].y);
                                }
#pragma unroll
                                for (int u = 0; u < 4; ++u) {
                                    const float gate = fmaf(tanh_approx(arg[u]), 0.5f, 0.5f);
                                    const float sv = __uint_as_float(sr[c * 32 + e0 + u]);
                                    sr[c * 32 + e0 + u] = __float_as_uint(c * 32 + e0 + u < nfar ? sv * gate : sv);
                                }
                            }
                        }
                    }
                }
                tmem_wait_ld();
                if (SOFTCAP) {
#pragma unroll
                    for (int c = 0; c < NC; ++c) sr[c] = __float_as_uint(tanh_approx(__uint_as_float(sr[c]) * cap_in));
                }
                if (tm.masked) {
#pragma unroll
                    for (int c = 0; c < NC; ++c)
                        sr[c] = ((tm.kw[(NSPLIT == 2 ? half * 2 : 0) + (c >> 5)] >> (c & 31)) & 1u) ? sr[c] : 0xff800000u;      // -inf
                }
                // ---- row maximum of the tile: four independent chains of three-input maxima
                float mx0 = -INFINITY, mx1 = -INFINITY, mx2 = -INFINITY, mx3 = -INFINITY;
#pragma unroll
                for (int c = 0; c < NC; c += 8) {
                    mx0 = max3(mx0, __uint_as_float(sr[c]), __uint_as_float(sr[c + 1]));
                    mx1 = max3(mx1, __uint_as_float(sr[c + 2]), __uint_as_float(sr[c + 3]));
                    mx2 = max3(mx2, __uint_as_float(sr[c + 4]), __uint_as_float(sr[c + 5]));
                    mx3 = max3(mx3, __uint_as_float(sr[c + 6]), __uint_as_float(sr[c + 7]));
                }
                float mraw = max3(mx0, mx1, fmaxf(mx2, mx3));
                if constexpr (NSPLIT == 2) {
                    // the two threads of a row exchange the maxima of their halves and then take the same decisions
                    const int par = (int)(nx & 1);
                    const __nv_bfloat16 mine = __float2bfloat16_rn(mraw);
                    xval(par, half, row_in_tile) = mine;
                    __syncwarp();
                    if (lane == 0) mbar_arrive(smem_u32(&ctl.xchg[warp & 3]));
                    ctl_wait(&ctl.xchg[warp & 3], (uint32_t)par, ctl, bad, 36);
                    mraw = fmaxf(__bfloat162float(mine), __bfloat162float(xval(par, half ^ 1, row_in_tile)));
                    ++nx;
                }
                const float mt = mraw * sl2;                     // log2 units (sl2 > 0; -inf stays -inf)
                // ---- lazy maximum: raise the reference only when it lags by more than the threshold
                float factor = 1.f;
                bool raise = false;
                if (m_used == -INFINITY) {
                    m_used = mt;                                 // nothing accumulated yet for this row
                } else if (mt > m_used + RESCALE_THRESHOLD) {
                    factor = ex2_approx(m_used - mt);
                    m_used = mt;
                    raise = true;
                }
                l *= factor;
                const float msub = m_used == -INFINITY ? 0.f : m_used;
                // ---- probabilities: packed fp32 pairs; part of the exponentials on the FMA/ALU pipes
                const float2 sl2v = make_float2(sl2, sl2), nmv = make_float2(-msub, -msub);
                float2 acc[4];
#pragma unroll
                for (int e = 0; e < 4; ++e) acc[e] = make_float2(0.f, 0.f);
                // The rows of O are brought to a raised reference just before P is handed over (before the exponentials, with all scores
                // held, the registers of this block slow the others down), which the P V waits for.
                auto hand_over = [&](uint64_t* bar, bool rescale) {
                    if (rescale && __any_sync(0xffffffffu, raise) && !first) {
                        // O may only be touched once the previous PV of this query tile has completed.  With two
                        // query tiles its commit precedes s_full; with double-buffered S it has its own barrier.
                        if constexpr (NQ == 1) ctl_wait(&ctl.pv_done, (ns - 1) & 1, ctl, bad, 35);
                        tc_fence_after();
#pragma unroll 1
                        for (int c = 0; c < D / 16 / NSPLIT; ++c) {      // this thread's part of the O row
                            uint32_t ov[16];
                            tmem_ld16(t_o + c * 16, ov);
                            tmem_wait_ld();
#pragma unroll
                            for (int e = 0; e < 16; ++e) ov[e] = __float_as_uint(__uint_as_float(ov[e]) * factor);
                            tmem_st16(t_o + c * 16, ov);
                        }
                    }
                    tmem_wait_st();
                    tc_fence_before();
                    mbar_arrive(smem_u32(bar));
                };
#pragma unroll
                for (int c = 0; c < NC; c += 8) {
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        const float2 xv = __ffma2_rn(make_float2(__uint_as_float(sr[c + 2 * e]),
                                                                 __uint_as_float(sr[c + 2 * e + 1])), sl2v, nmv);
                        float2 pr;
                        if (e >= 4 - EX2_POLY_PER_8 / 2) {
                            pr = ex2_poly2(xv);
                        } else {
                            pr.x = ex2_approx(xv.x);
                            pr.y = ex2_approx(xv.y);
                        }
                        acc[e] = __fadd2_rn(acc[e], pr);
                        pk[(c >> 1) + e] = pack_bf16x2(pr.x, pr.y);
                    }
                    if constexpr (C::SPLIT_P) {
                        static_assert(C::P_FIRST == 96, "the stores below");
                        if (c + 8 == C::P_FIRST) {
                            tmem_st32(t_s, *reinterpret_cast<uint32_t(*)[32]>(&pk[0]));
                            tmem_st16(t_s + 32, *reinterpret_cast<uint32_t(*)[16]>(&pk[32]));
                            hand_over(&ctl.p_full[buf], true);
                        }
                    }
                }
                if constexpr (C::SPLIT_P) {
                    tmem_st16(t_s + 48, *reinterpret_cast<uint32_t(*)[16]>(&pk[48]));
                    hand_over(&ctl.p_rest[buf], false);
                } else {
#pragma unroll
                    for (int c = 0; c < NC / 64; ++c) tmem_st32(t_s + c * 32, *reinterpret_cast<uint32_t(*)[32]>(&pk[c * 32]));
                    hand_over(&ctl.p_full[buf], true);
                }
                l += (acc[0].x + acc[0].y) + (acc[1].x + acc[1].y) + ((acc[2].x + acc[2].y) + (acc[3].x + acc[3].y));
                ++ns;
                first = false;
                if (bad) break;
            }
            if (bad) break;
            tile_read();                                 // the end of the item
            finish = !first;
        }
        if (bad) give_up(p, &ctl, bad, t.A, ord);
    }
    // ---------------------------------------------------------------------- teardown
    tc_fence_before();
    __syncthreads();
    if (*(volatile int*)&ctl.abort_flag) {
        // a role gave up: let copies that were already issued land before the CTA leaves
        const uint64_t t0 = globaltimer_ns();
        while (globaltimer_ns() - t0 < 20000ull) { }
        // ... and take the blocks that have not started out of the queue: each of them would wait as long
        if (threadIdx.x == 0) {
            uint32_t asked = ctl.asked, block;
            for (;;) {
                if (asked > 0) {
                    const uint32_t slot = (asked - 1) & 1;
                    if (!mbar_wait(smem_u32(&ctl.next_full[slot]), ((asked - 1) >> 1) & 1, 1000000ull)) break;
                    if (!clc_answer(smem_u32(&ctl.next[slot]), block)) break;
                    fence_proxy_async_smem();
                }
                const uint32_t slot = asked & 1;
                mbar_arrive_expect_tx(smem_u32(&ctl.next_full[slot]), 16);
                clc_try_cancel(smem_u32(&ctl.next[slot]), smem_u32(&ctl.next_full[slot]));
                ++asked;
            }
        }
        __syncthreads();
    }
    if (warp == 1) tmem_dealloc(tmem, 512);
}

template <int D, bool SOFTCAP, int GATE, int WALK>
static int launch_attn_t(const AttnArgs& a, cudaStream_t st) {
    using C = AttnCfg<D, GATE>;
    CUtensorMap tq, tk, tv;
    int rc;
    constexpr bool sorted = WALK == WALK_SORTED;
    if constexpr (sorted) {
        // gather Q, K, V into the sorted order kept in the workspace; the kernel reads the copies
        char* ws = const_cast<char*>(a.ws);
        if ((rc = launch_gather_sorted(&a.s, a.q, a.k, a.v, a.L, ws, st))) return rc;
        const int HQ = a.s.batch * a.s.Hq, HK = a.s.batch * a.s.Hkv;
        const focus_tensor sq_t{ws + a.L.qs, (int64_t)HQ * a.L.nqp * D, (int64_t)a.L.nqp * D, D};
        const focus_tensor sk_t{ws + a.L.ks, (int64_t)HK * a.L.nkp * D, (int64_t)a.L.nkp * D, D};
        const focus_tensor sv_t{ws + a.L.vs, (int64_t)HK * a.L.nkp * D, (int64_t)a.L.nkp * D, D};
        if ((rc = make_tmap_qkv(&tq, sq_t, 1, HQ, a.L.nqp, D))) return rc;
        if ((rc = make_tmap_qkv(&tk, sk_t, 1, HK, a.L.nkp, D))) return rc;
        if ((rc = make_tmap_qkv(&tv, sv_t, 1, HK, a.L.nkp, D, 128 / C::PARTS))) return rc;
    } else {
        if ((rc = make_tmap_qkv(&tq, a.q, a.s.batch, a.s.Hq, a.s.n, D))) return rc;
        if ((rc = make_tmap_qkv(&tk, a.k, a.s.batch, a.s.Hkv, a.s.n, D))) return rc;
        if ((rc = make_tmap_qkv(&tv, a.v, a.s.batch, a.s.Hkv, a.s.n, D, 128 / C::PARTS))) return rc;
    }
    AttnParams p;
    p.B = a.s.batch; p.Hq = a.s.Hq; p.Hkv = a.s.Hkv; p.G = a.s.Hq / a.s.Hkv; p.n = a.s.n; p.w = a.s.window < a.s.n ? a.s.window : a.s.n; p.K = a.s.K;
    p.nqb = cdiv(a.s.n, 128 * C::NQ);
    p.nqt = cdiv(a.s.n, 128); p.nkt = cdiv(a.s.n, 128); p.nkw = cdiv(p.nkt, 32);
    p.scale = a.scale; p.softcap = a.s.softcap;
    p.mq = a.mq;
    p.gbits = a.ws ? reinterpret_cast<const uint32_t*>(a.ws + a.L.gbits) : nullptr;
    p.live = a.ws ? reinterpret_cast<const uint32_t*>(a.ws + a.L.live) : nullptr;
    p.o = reinterpret_cast<__nv_bfloat16*>(a.o.ptr);
    p.o_sb = a.o.stride_b; p.o_sh = a.o.stride_h; p.o_sn = a.o.stride_n;
    // rows of O on the 32-byte grid: whole sectors per store (a warp's stores go to 32 rows at a time)
    p.o_wide = (uintptr_t)a.o.ptr % 32 == 0 && (a.o.stride_b | a.o.stride_h | a.o.stride_n) % 16 == 0;
    p.lse = a.lse;
    p.status = a.dev_status;
    p.nitems = (long long)a.s.batch * a.s.Hq * p.nqb;
    p.by_heads = Divisor(p.B * p.Hq); p.by_group = Divisor(p.nqb * p.G); p.by_G = Divisor(p.G); p.by_Hkv = Divisor(p.Hkv); p.by_Hq = Divisor(p.Hq);
    p.nqp = a.L.nqp; p.nkp = a.L.nkp; p.nqblk = a.L.nqp / 256;
    p.ipb = 2 / C::NQ;
    p.perm_q = sorted ? reinterpret_cast<const int32_t*>(a.ws + a.L.perm_q) : nullptr;
    p.perm_k = sorted ? reinterpret_cast<const int32_t*>(a.ws + a.L.perm_k) : nullptr;
    p.cls_k = sorted ? reinterpret_cast<const uint32_t*>(a.ws + a.L.cls_k) : nullptr;
    p.ncls_k = sorted ? reinterpret_cast<const int32_t*>(a.ws + a.L.ncls_k) : nullptr;
    p.qrange = sorted ? reinterpret_cast<const int32_t*>(a.ws + a.L.qrange) : nullptr;
    p.order = sorted ? reinterpret_cast<const int32_t*>(a.ws + a.L.order) : nullptr;
    p.counters = a.ws ? reinterpret_cast<const unsigned long long*>(a.ws + a.L.counters) : nullptr;
    p.gate_g = a.gate_g; p.gate_ld = a.gate_ld; p.gate_hl = 0.5f * a.gate_lambda;
    p.local_only = a.local_pass ? 1 : 0;
    p.share_only = (sorted && layout_has_window_pass(a.L.layout)) ? 1 : 0;
    p.gbits_s = (sorted && a.L.layout == FOCUS_LAYOUT_GROUP_MAJOR) ? reinterpret_cast<const uint32_t*>(a.ws + a.L.gbits_s) : nullptr;
    p.o32 = a.o32;
    p.join = a.join;
    p.wait_limit_ns = a.wait_limit_ns;
    p.stall_at = a.stall_at;
    if (sorted) p.nitems = (long long)a.s.batch * a.s.Hq * p.nqblk * p.ipb;
    // K and V of all heads up to half of L2 (126 MB): the order of the items need not keep to one head at a time
    p.by_length = (size_t)a.s.batch * a.s.Hkv * a.s.n * D * 4 <= ((size_t)64 << 20);
    if (p.nitems > 0x7fffffffll) return fail(FOCUS_ERR_UNSUPPORTED, "attention: %lld query blocks exceed 2^31 - 1", p.nitems);
    auto kern = focus_attn_kernel<D, SOFTCAP, GATE, WALK>;
    constexpr uint32_t smem = C::OFF_CTL + (uint32_t)sizeof(SharedCtl) + (C::GATE_MMA ? (uint32_t)sizeof(GateCtl) : 0);
    static_assert(smem <= 227 * 1024, "shared memory of one block");
    if ((rc = check_cuda(allow_smem<focus_attn_kernel<D, SOFTCAP, GATE, WALK>>(smem), "cudaFuncSetAttribute(attn)"))) return rc;
    return check_cuda(launch_dependent(kern, dim3((unsigned)p.nitems), dim3(C::THREADS), smem, st, tq, tk, tv, p), "attention kernel launch");
}

static int launch_attn_one(const AttnArgs& a, cudaStream_t st);

int launch_attn_sm100(const AttnArgs& a, cudaStream_t st) {
    if (a.ws && layout_has_window_pass(a.L.layout) && !a.local_pass) {
        // (1) sharing pairs in the class-sorted order -> o, lse; rows of blocks without key tiles keep lse = -inf
        // (2) window-only pairs in token order, each row joined with what (1) left (a pass of its own for that read and wrote
        // another 1.3 GB at 32 heads x 32768 tokens x 128: 202 us)
        char* ws = const_cast<char*>(a.ws);
        const size_t rows = (size_t)a.s.batch * a.s.Hq * a.s.n;
        int rc = launch_fill_f32(a.lse, rows, -INFINITY, st);
        if (rc) return rc;
        AttnArgs s1 = a;
        s1.o32 = reinterpret_cast<float*>(ws + a.L.o_sorted);
        if ((rc = launch_attn_one(s1, st))) return rc;
        AttnArgs s2 = a;
        s2.local_pass = true;
        s2.join = s1.o32;
        return launch_attn_one(s2, st);
    }
    return launch_attn_one(a, st);
}

template <int D>
static int launch_attn_d(const AttnArgs& a, cudaStream_t st) {
    if (a.gate_g) {      // training-time gated forward: dense causal walk, no softcap
        const int chunks = a.gate_ld <= 8 ? 1 : a.gate_ld / 8;      // 8-float chunks of an assignment row
        if (chunks == 1) return launch_attn_t<D, false, 1, WALK_DENSE>(a, st);
        if (chunks == 2) return launch_attn_t<D, false, 2, WALK_DENSE>(a, st);
        if constexpr (D != 256) return launch_attn_t<D, false, 4, WALK_DENSE>(a, st);
        return fail(FOCUS_ERR_UNSUPPORTED, "the gated forward at D = 256 supports K <= 16");
    }
    const bool cap = a.s.softcap > 0.f;
    if (!a.ws) return cap ? launch_attn_t<D, true, 0, WALK_DENSE>(a, st) : launch_attn_t<D, false, 0, WALK_DENSE>(a, st);
    if (a.local_pass || !layout_is_sorted(a.L.layout))
        return cap ? launch_attn_t<D, true, 0, WALK_TOKEN>(a, st) : launch_attn_t<D, false, 0, WALK_TOKEN>(a, st);
    return cap ? launch_attn_t<D, true, 0, WALK_SORTED>(a, st) : launch_attn_t<D, false, 0, WALK_SORTED>(a, st);
}

static int launch_attn_one(const AttnArgs& a, cudaStream_t st) {
    switch (a.s.D) {
        case 64: return launch_attn_d<64>(a, st);
        case 128: return launch_attn_d<128>(a, st);
        case 256: return launch_attn_d<256>(a, st);
    }
    return fail(FOCUS_ERR_UNSUPPORTED, "D (%d) must be 64, 128 or 256", a.s.D);
}

}  // namespace focus
