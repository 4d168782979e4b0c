// focus_sinkhorn: the Sinkhorn normalisation of the soft group assignments (paper Sec. 2 "Learned grouping"):
// Q = exp(S / tau), then N times "divide each column by its sum over the tokens, divide each row by its sum over
// the groups".
//
// Every iterate has the form Q = diag(r) exp(S / tau) diag(c).  A column division replaces c_g by
// 1 / sum_i r_i E_ig and a row division replaces r_i by 1 / sum_g E_ig c_g, so one pass over the scores per
// iteration is enough: with the current column offsets a token computes its row offset (a log-sum-exp over K
// values), its normalised row Q_i (every entry in (0, 1]) and adds that row into the column sums that give the next
// column offsets.  Offsets are kept as logarithms, so nothing overflows at a small temperature; the very first
// column sum is taken relative to the column maximum.  Column sums are accumulated in fp64.
//
// Two forms.  While a sequence's rows fit in the shared memory of the blocks that are resident at once, one cooperative
// launch does the whole call (sinkhorn_team_kernel): every row is read once, and what separates two iterations is a
// barrier between the blocks of a sequence.  Longer sequences take one launch per iteration over the matrix in L2.
#include "common.cuh"

#include <type_traits>

namespace focus {

constexpr int SK_THREADS = 256;
constexpr int SK_MAX_BLOCKS = 148 * 8;

// order-preserving map of a float onto unsigned integers (0 sorts below every float)
__device__ __forceinline__ uint32_t ordered_of(float f) {
    const uint32_t b = __float_as_uint(f);
    return (b & 0x80000000u) ? ~b : (b | 0x80000000u);
}
__device__ __forceinline__ float float_of_ordered(uint32_t o) {
    return __uint_as_float((o & 0x80000000u) ? (o & 0x7fffffffu) : ~o);
}

// workspace of one sequence: double T[iters + 1][32] (column sums of pass 0, 1, ...), then uint32 M[32] (column maxima)
// (then, for all sequences, the words of the one-launch form)
__host__ __device__ inline size_t sk_seq_bytes(int iters) { return (size_t)(iters + 1) * 32 * sizeof(double) + 32 * sizeof(uint32_t); }

template <int KMAX>
__device__ __forceinline__ void load_row(const float* __restrict__ S, size_t tok, float (&x)[KMAX]) {
    const float4* p = reinterpret_cast<const float4*>(S + tok * KMAX);
#pragma unroll
    for (int c = 0; c < KMAX / 4; ++c) {
        const float4 v = __ldg(p + c);
        x[4 * c] = v.x; x[4 * c + 1] = v.y; x[4 * c + 2] = v.z; x[4 * c + 3] = v.w;
    }
}

template <int KMAX>
__global__ void __launch_bounds__(SK_THREADS)
sinkhorn_colmax_kernel(const float* __restrict__ S, int n, int K, int iters, unsigned char* __restrict__ ws) {
    const int b = blockIdx.y;
    uint32_t* M = reinterpret_cast<uint32_t*>(ws + (size_t)b * sk_seq_bytes(iters) + (size_t)(iters + 1) * 32 * sizeof(double));
    const float* Sb = S + (size_t)b * n * KMAX;
    float mx[KMAX];
#pragma unroll
    for (int g = 0; g < KMAX; ++g) mx[g] = -INFINITY;
    for (int tok = blockIdx.x * SK_THREADS + threadIdx.x; tok < n; tok += gridDim.x * SK_THREADS) {
        float x[KMAX];
        load_row<KMAX>(Sb, (size_t)tok, x);
#pragma unroll
        for (int g = 0; g < KMAX; ++g) mx[g] = fmaxf(mx[g], x[g]);
    }
#pragma unroll
    for (int g = 0; g < KMAX; ++g) {
        float m = mx[g];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
        if ((threadIdx.x & 31) == 0 && g < K && m > -INFINITY) atomicMax(M + g, ordered_of(m));
    }
}

// MODE 0: column sums of exp((S - M) / tau).  MODE 1: a row division followed by the next column sums.
// MODE 2: the last row division; writes the assignments.
template <int KMAX, int MODE>
__global__ void __launch_bounds__(SK_THREADS)
sinkhorn_pass_kernel(const float* __restrict__ S, int n, int K, int iters, int pass, float inv_tau,
                     unsigned char* __restrict__ ws, float* __restrict__ out) {
    __shared__ double red[SK_THREADS / 32][KMAX];
    __shared__ float colmax_s[KMAX], voff_s[KMAX];
    const int b = blockIdx.y;
    unsigned char* wsb = ws + (size_t)b * sk_seq_bytes(iters);
    double* T = reinterpret_cast<double*>(wsb);
    const uint32_t* M = reinterpret_cast<const uint32_t*>(wsb + (size_t)(iters + 1) * 32 * sizeof(double));
    const float* Sb = S + (size_t)b * n * KMAX;
    if (threadIdx.x < KMAX) {
        const int g = threadIdx.x;
        float cm = 0.f, v = 0.f;
        if (g < K) {
            cm = float_of_ordered(M[g]);
            // column offset after `pass` column divisions, relative to the column maximum:
            // -log of the first column sum, then minus the log of every later one
            double acc = 0.0;
            for (int m = 0; m < pass; ++m) acc -= log(T[(size_t)m * 32 + g]);
            v = (float)acc;
        }
        colmax_s[g] = cm;
        voff_s[g] = v;
    }
    __syncthreads();
    float tsum[KMAX];
#pragma unroll
    for (int g = 0; g < KMAX; ++g) tsum[g] = 0.f;
    for (int tok = blockIdx.x * SK_THREADS + threadIdx.x; tok < n; tok += gridDim.x * SK_THREADS) {
        float x[KMAX];
        load_row<KMAX>(Sb, (size_t)tok, x);
        if (MODE == 0) {
#pragma unroll
            for (int g = 0; g < KMAX; ++g)
                if (g < K) tsum[g] += expf((x[g] - colmax_s[g]) * inv_tau);
        } else {
            float mx = -INFINITY;
#pragma unroll
            for (int g = 0; g < KMAX; ++g) {
                x[g] = (x[g] - colmax_s[g]) * inv_tau + voff_s[g];
                if (g < K) mx = fmaxf(mx, x[g]);
            }
            float se = 0.f;
#pragma unroll
            for (int g = 0; g < KMAX; ++g) {
                x[g] = g < K ? expf(x[g] - mx) : 0.f;
                se += x[g];
            }
            const float inv = 1.f / se;
#pragma unroll
            for (int g = 0; g < KMAX; ++g) x[g] *= inv;
            if (MODE == 1) {
#pragma unroll
                for (int g = 0; g < KMAX; ++g) tsum[g] += x[g];
            } else {
                float4* o = reinterpret_cast<float4*>(out + ((size_t)b * n + tok) * KMAX);
#pragma unroll
                for (int c = 0; c < KMAX / 4; ++c) o[c] = make_float4(x[4 * c], x[4 * c + 1], x[4 * c + 2], x[4 * c + 3]);
            }
        }
    }
    if (MODE != 2) {
#pragma unroll
        for (int g = 0; g < KMAX; ++g) {
            float s = tsum[g];
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
            if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5][g] = (double)s;
        }
        __syncthreads();
        if (threadIdx.x < K) {
            double s = 0.0;
            for (int w = 0; w < SK_THREADS / 32; ++w) s += red[w][threadIdx.x];
            atomicAdd(T + (size_t)pass * 32 + threadIdx.x, s);
        }
    }
}

// ---- one launch for the whole call: the P blocks of a sequence (a "team") keep its rows in shared memory, `chunk`
// tokens per block, and walk the iterations together.  Between two iterations stands one exchange: every block publishes
// its K column sums and adds up the P x K numbers of its team.  A number, a double whole, travels as two 8-byte words, each half
// of its bits and the exchange's ordinal, written and polled whole, so that neither a fence nor
// a counter stands between writing and reading it (fp64 atomics into one sum, a fence and an arrival counter took 3.5 us
// per exchange), and the order of every sum is fixed.  What bounds it is latency: of the ~2.3 us of an iteration a third
// is the words' way through L2, the rest instruction issue and block barriers.  The launch is cooperative, so
// that all blocks of a team run at once.
constexpr int SKT_THREADS = 512;
constexpr int SKT_TOKENS = 8 * SKT_THREADS;          // tokens per block at most: fp32 column sums of a thread over 8 rows
constexpr int SKT_BLOCKS = 160;                      // blocks per team at most (the workspace has words for as many)
constexpr size_t SKT_SMEM = 200 * 1024;
constexpr long long SKT_LEAD = 500;                  // cycles before the first poll
constexpr long long SKT_LIMIT = 4000000000ll;        // cycles of a wait: two seconds

// words of one sequence's exchanges: two sets, taken in turn.  A block writes set e mod 2 for exchange e + 2 after it has
// read everybody's e + 1, which each of them wrote after reading everybody's e.
static int skt_max_blocks(int n) { return cdiv(n, SKT_THREADS) < SKT_BLOCKS ? cdiv(n, SKT_THREADS) : SKT_BLOCKS; }
// Every block has 128-byte lines of its own.
__host__ __device__ constexpr size_t skt_stride(int ld) { return ld < 8 ? 128 : (size_t)ld * 16; }
static size_t skt_words_bytes(const focus_shape* s) { return 2 * skt_max_blocks(s->n) * skt_stride(focus_soft_ld(s->K)); }

__device__ __forceinline__ void put_word(void* p, double v, unsigned int tag) {
    const unsigned long long bits = (unsigned long long)__double_as_longlong(v);
    asm volatile("st.relaxed.gpu.global.v2.b64 [%0], {%1, %2};" ::"l"(p), "l"((bits & 0xffffffff00000000ull) | tag), "l"(bits << 32 | tag) : "memory");
}
__device__ __forceinline__ bool get_word(const void* p, unsigned int tag, double& v) {
    unsigned long long a, b;
    asm volatile("ld.relaxed.gpu.global.v2.b64 {%0, %1}, [%2];" : "=l"(a), "=l"(b) : "l"(p) : "memory");
    v = __longlong_as_double((long long)((a & 0xffffffff00000000ull) | b >> 32));
    return (unsigned int)a == tag && (unsigned int)b == tag;
}

// log2 of a positive double to 1e-15, in less time than the library's (it stands between two iterations): Tang's table
// method.  tab[k] = (c, -log2 c) with c a float near 1 / (1 + (k + 1/2) / 32); u = m c - 1 for the mantissa m is below 1/60, exact
// but for one rounding, and log1p(u) is summed to its eighth term (the ninth is below 1e-17).
__device__ __forceinline__ double2 log2_entry(int k) {
    const float c = 1.f / (1.f + (k + 0.5f) / 32.f);
    return make_double2((double)c, -log2((double)c));
}
__device__ __forceinline__ double log2_table(double x, const double2* tab) {
    if (!(x >= 2.2250738585072014e-308 && x < INFINITY)) return log2(x);           // zero, denormal, infinity, NaN
    const long long bits = __double_as_longlong(x);
    const int e = (int)(bits >> 52) - 1023;
    const double m = __longlong_as_double((bits & 0x000fffffffffffffll) | 0x3ff0000000000000ll);
    const double2 t = tab[(int)(bits >> 47) & 31];
    const double u = fma(m, t.x, -1.0), u2 = u * u;
    // -1/2 + u/3 - u^2/4 + ... - u^6/8, in pairs so that the chain is short
    const double p01 = fma(u, 1.0 / 3, -0.5), p23 = fma(u, 1.0 / 5, -0.25), p45 = fma(u, 1.0 / 7, -1.0 / 6);
    const double tail = u2 * fma(u2, fma(u2, fma(u2, -0.125, p45), p23), p01);
    return ((double)e + t.y) + 1.4426950408889634 * (u + tail);
}
__device__ __forceinline__ float ex2f(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ float rcpf(float x) {
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// v[0..N) of the 32 lanes combined: lane l ends with the result of value l / (32 / N) in v[0]
template <int N, bool MAX>
__device__ __forceinline__ void reduce_lanes(float (&v)[N]) {
    const int lane = threadIdx.x & 31;
    int off = 16;
#pragma unroll
    for (int w = N / 2; w >= 1; w /= 2, off /= 2) {
        const bool up = lane & off;
#pragma unroll
        for (int i = 0; i < w; ++i) {
            const float r = __shfl_xor_sync(0xffffffffu, up ? v[i] : v[i + w], off);
            const float mine = up ? v[i + w] : v[i];
            v[i] = MAX ? fmaxf(mine, r) : mine + r;
        }
    }
    for (; off >= 1; off /= 2) {
        const float r = __shfl_xor_sync(0xffffffffu, v[0], off);
        v[0] = MAX ? fmaxf(v[0], r) : v[0] + r;
    }
}

// BWD = false: out = the assignments.  BWD = true: the column sums again, then the derivative of the assignments
// from d_in to out (the passes of sinkhorn_bwd_pass_kernel and sinkhorn_bwd_last_kernel below).
// LATE: diagnostic, waits of late_limit cycles, and the first block of a sequence comes late by four of them to exchange late_at.
template <int KMAX, bool BWD, bool LATE>
__global__ void __launch_bounds__(SKT_THREADS, 1)
sinkhorn_team_kernel(const float* S, int n, int K, int iters, float tau, float inv_tau, unsigned char* __restrict__ ws,
                     unsigned char* __restrict__ words, size_t words_bytes, const float* d_in, float* out, int P, int chunk,
                     long long late_limit, unsigned int late_at) {
    extern __shared__ float4 rows_s[];               // [KMAX / 4][chunk] scores, then as many of the derivative
    constexpr int NW = SKT_THREADS / 32, PIECES = KMAX / 4;
    __shared__ float red[NW][KMAX];
    __shared__ float colmax_s[KMAX], voff_s[KMAX], pend_sub_s[KMAX], pend_inv_s[KMAX], ct_s[KMAX];
    __shared__ double team_s[NW][KMAX];
    __shared__ int failed_s;
    const int b = blockIdx.x / P, rank = blockIdx.x % P, tok0 = rank * chunk;
    const int cnt = min(chunk, n - tok0);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    double* const T = reinterpret_cast<double*>(ws + (size_t)b * sk_seq_bytes(iters));       // BWD: sums of pass 0 .. iters - 1
    words += (size_t)b * words_bytes;
    float4* const dcache = rows_s + (size_t)PIECES * chunk;
    auto get = [&](const float4* c, int i, float (&x)[KMAX]) {
#pragma unroll
        for (int q = 0; q < PIECES; ++q) {
            const float4 v = c[(size_t)q * chunk + i];
            x[4 * q] = v.x; x[4 * q + 1] = v.y; x[4 * q + 2] = v.z; x[4 * q + 3] = v.w;
        }
    };
    auto put = [&](float4* c, int i, const float (&x)[KMAX]) {
#pragma unroll
        for (int q = 0; q < PIECES; ++q) c[(size_t)q * chunk + i] = make_float4(x[4 * q], x[4 * q + 1], x[4 * q + 2], x[4 * q + 3]);
    };
    __shared__ double2 tab_s[32];
    if (threadIdx.x < 32) tab_s[threadIdx.x] = log2_entry(threadIdx.x);
    if (threadIdx.x == 0) failed_s = 0;

    // the exchange: the warps' values (red) become the block's, the blocks' the team's; collect(g, value) runs in lane g
    // of the first warp.  Thread t polls the words of group t mod KMAX.
    unsigned int ordinal = 0;
    auto exchange = [&](auto is_max, auto collect) {
        constexpr bool MAX = decltype(is_max)::value;
        constexpr int PARTS = 32 / KMAX;
        auto combine = [](double x, double y) { return MAX ? fmax(x, y) : x + y; };
        // lane l: value l mod KMAX of the warps, PARTS lanes a value
        auto over_warps = [&](auto& vals) {
            double v = (double)vals[lane / KMAX][lane % KMAX];
#pragma unroll
            for (int w = PARTS; w < NW; w += PARTS) v = combine(v, (double)vals[w + lane / KMAX][lane % KMAX]);
#pragma unroll
            for (int off = 16; off >= KMAX; off /= 2) v = combine(v, __shfl_xor_sync(0xffffffffu, v, off));
            return v;
        };
        // A wait that runs out leaves the block with sums that are not numbers, hence with such offsets and such sums to publish from
        // then on: nobody goes on with sums that lack somebody's.  (A maximum passes over what is not a number; see there.)
        const double none = __longlong_as_double(0x7fffffffffffffffll);
        ++ordinal;
        unsigned char* const set = words + (size_t)(ordinal & 1) * P * skt_stride(KMAX);
        if (LATE && ordinal == late_at && rank == 0 && threadIdx.x == 0)
            for (const long long t0 = clock64(); clock64() - t0 < 4 * late_limit;) { }
        __syncthreads();                             // red holds the warps' values
        if (warp == 0) {
            const double v = over_warps(red);
            if (lane < KMAX) put_word(set + (size_t)rank * skt_stride(KMAX) + lane * 16, v, ordinal);
        }
        double v = MAX ? -INFINITY : 0.0;
        if (!failed_s) {
            constexpr int STEP = SKT_THREADS / KMAX, PER = (SKT_BLOCKS + STEP - 1) / STEP;
            double got[PER];
            bool seen[PER];
#pragma unroll
            for (int j = 0; j < PER; ++j) {
                got[j] = v;
                seen[j] = threadIdx.x / KMAX + j * STEP >= P;
            }
            // A poll that comes too early makes the next one take 1.4 us instead of 0.4, and a block that is late by that
            // much makes the others' polls come too early in the next exchange; so wait out most of the words' way first.
            // Forward and derivative, 500 cycles against none: 131072 x 8 83 and 87 us, 30000 x 8 70 and 105, 8192 x 8 70
            // and 98; 900 cycles cost another 5 us each.
            const long long t0 = clock64();
            while (P > 1 && clock64() - t0 < SKT_LEAD) { }
            for (bool all = false; !all;) {
                all = true;
#pragma unroll
                for (int j = 0; j < PER; ++j) {
                    const int q = threadIdx.x / KMAX + j * STEP;
                    if (!seen[j]) all &= seen[j] = get_word(set + (size_t)q * skt_stride(KMAX) + threadIdx.x % KMAX * 16, ordinal, got[j]);
                }
                if (!all && clock64() - t0 > (LATE ? late_limit : SKT_LIMIT)) {
                    failed_s = 1;
                    got[0] = none;
                    break;
                }
            }
#pragma unroll
            for (int j = 0; j < PER; ++j) v = combine(v, got[j]);
        } else {
            v = none;
        }
#pragma unroll
        for (int off = 16; off >= KMAX; off /= 2) v = combine(v, __shfl_xor_sync(0xffffffffu, v, off));
        if (lane < KMAX) team_s[warp][lane] = v;
        __syncthreads();
        if (warp == 0) {
            const double v = over_warps(team_s);
            if (lane < KMAX) collect(lane, v);
        }
        __syncthreads();
    };
    auto store_warp = [&](float (&v)[KMAX]) {
        if (lane % (32 / KMAX) == 0) red[warp][lane / (32 / KMAX)] = v[0];
    };

    // ---- rows to shared memory, column maxima
    {
        float mx[KMAX];
#pragma unroll
        for (int g = 0; g < KMAX; ++g) mx[g] = -INFINITY;
        const float4* src = reinterpret_cast<const float4*>(S + ((size_t)b * n + tok0) * KMAX);
        const float4* dsrc = BWD ? reinterpret_cast<const float4*>(d_in + ((size_t)b * n + tok0) * KMAX) : nullptr;
        for (int i = threadIdx.x; i < cnt; i += SKT_THREADS)
#pragma unroll
            for (int q = 0; q < PIECES; ++q) {
                const float4 v = src[(size_t)i * PIECES + q];
                rows_s[(size_t)q * chunk + i] = v;
                if (BWD) {
                    const float4 d = dsrc[(size_t)i * PIECES + q];           // entries beyond K are ignored
                    dcache[(size_t)q * chunk + i] = make_float4(4 * q < K ? d.x : 0.f, 4 * q + 1 < K ? d.y : 0.f,
                                                                4 * q + 2 < K ? d.z : 0.f, 4 * q + 3 < K ? d.w : 0.f);
                }
                mx[4 * q] = fmaxf(mx[4 * q], v.x); mx[4 * q + 1] = fmaxf(mx[4 * q + 1], v.y);
                mx[4 * q + 2] = fmaxf(mx[4 * q + 2], v.z); mx[4 * q + 3] = fmaxf(mx[4 * q + 3], v.w);
            }
        reduce_lanes<KMAX, true>(mx);
        store_warp(mx);
    }
    exchange(std::true_type{}, [&](int g, double m) {
        colmax_s[g] = m > -INFINITY && !failed_s ? (float)m : float_of_ordered(0u);         // no maximum: NaN
        voff_s[g] = g < K ? 0.f : -INFINITY;
        ct_s[g] = pend_sub_s[g] = 0.f;
        pend_inv_s[g] = g < K ? 1.f : 0.f;
    });
    // the cached scores become S - M, 0 beyond K (where the offsets of minus infinity leave nothing).  Log2 units are
    // (S - M) * log2(e) / tau, the factor in two floats: a factor rounded once would shift every exponent alike
    const double per_tau = 1.4426950408889634 / (double)tau;
    const float c_hi = (float)per_tau, c_lo = (float)(per_tau - (double)c_hi);
    // A difference whose exponent overflows (minus infinity among them) has weight 0.  It is kept at the lowest value whose
    // exponent is finite: c_lo may be negative, and times minus infinity it would add plus infinity to the exponent.  A row
    // with no other entry has no assignment and becomes NaN, as (-inf) - (-inf) makes it in the passes below; NaN stays NaN.
    const float lowest = -3.4e38f / fmaxf(c_hi, 1.f);
    for (int i = threadIdx.x; i < cnt; i += SKT_THREADS) {
        float x[KMAX];
        get(rows_s, i, x);
        bool closed = true;
#pragma unroll
        for (int g = 0; g < KMAX; ++g) {
            x[g] = g < K ? x[g] - colmax_s[g] : 0.f;
            if (g < K) closed &= x[g] < lowest;
        }
#pragma unroll
        for (int g = 0; g < KMAX; ++g) {
            if (x[g] < lowest) x[g] = lowest;
            if (g < K && closed) x[g] = __int_as_float(0x7fffffff);
        }
        put(rows_s, i, x);
    }
    auto log2_units = [&](float x, float off) { return fmaf(x, c_hi, fmaf(x, c_lo, off)); };
    // ---- column sums of pass 0 .. iters - 1.  Lane g of the first warp keeps column g's offset in double: minus the logs
    // of the sums so far.
    double acc = 0.0, sum = 1.0;                     // and the last sum collected
    // Z = softmax over the groups of the scores plus offsets, as exponentials and the reciprocal of their sum
    auto softmax_row = [&](float (&x)[KMAX]) {
        float mx = -INFINITY;
#pragma unroll
        for (int g = 0; g < KMAX; ++g) {
            x[g] = log2_units(x[g], voff_s[g]);
            mx = fmaxf(mx, x[g]);
        }
        float se = 0.f;
#pragma unroll
        for (int g = 0; g < KMAX; ++g) {
            x[g] = ex2f(x[g] - mx);
            se += x[g];
        }
        return rcpf(se);
    };
    for (int pass = 0; pass < iters; ++pass) {
        float tsum[KMAX];
#pragma unroll
        for (int g = 0; g < KMAX; ++g) tsum[g] = 0.f;
        for (int i = threadIdx.x; i < cnt; i += SKT_THREADS) {
            float x[KMAX];
            get(rows_s, i, x);
            if (pass == 0) {
#pragma unroll
                for (int g = 0; g < KMAX; ++g) tsum[g] += ex2f(log2_units(x[g], 0.f));
            } else {
                const float inv = softmax_row(x);
#pragma unroll
                for (int g = 0; g < KMAX; ++g) tsum[g] = fmaf(x[g], inv, tsum[g]);
            }
        }
        reduce_lanes<KMAX, false>(tsum);
        store_warp(tsum);
        exchange(std::false_type{}, [&](int g, double total) {
            if (g < K) {
                sum = total;
                acc -= log2_table(sum, tab_s);
            }
            // a row's softmax does not see what all offsets have in common (about log2(n / K) per pass): leave it out, so
            // that a small number is rounded to fp32
            const double common = __shfl_sync(KMAX == 32 ? 0xffffffffu : (1u << KMAX) - 1u, acc, 0);
            if (g >= K) return;
            voff_s[g] = (float)(BWD && iters == 1 ? acc : acc - common);      // (Y_0 below wants the offset itself)
            if (BWD) {
                T[(size_t)pass * 32 + g] = sum;      // the same value from every block; read back by this thread
                ct_s[g] = (float)sum;                // for the first pass of the derivative, t = iters - 1
            }
        });
    }
    float4* const o = reinterpret_cast<float4*>(out + ((size_t)b * n + tok0) * KMAX);
    if constexpr (!BWD) {
        // ---- the last row division
        for (int i = threadIdx.x; i < cnt; i += SKT_THREADS) {
            float x[KMAX];
            get(rows_s, i, x);
            const float inv = softmax_row(x);
#pragma unroll
            for (int q = 0; q < PIECES; ++q)
                o[(size_t)i * PIECES + q] = make_float4(x[4 * q] * inv, x[4 * q + 1] * inv, x[4 * q + 2] * inv, x[4 * q + 3] * inv);
        }
    } else {
        // ---- the iterations in reverse
        for (int t = iters - 1; t >= 0; --t) {
            float tsum[KMAX];
#pragma unroll
            for (int g = 0; g < KMAX; ++g) tsum[g] = 0.f;
            for (int i = threadIdx.x; i < cnt; i += SKT_THREADS) {
                float x[KMAX], d[KMAX];
                get(rows_s, i, x);
                get(dcache, i, d);
                const float inv = softmax_row(x);
                float dot = 0.f, rinv = t >= 1 ? 0.f : 1.f;
#pragma unroll
                for (int g = 0; g < KMAX; ++g) {
                    x[g] *= inv;                     // Z_t
                    d[g] = (d[g] - pend_sub_s[g]) * pend_inv_s[g];
                    dot = fmaf(d[g], x[g], dot);
                    if (t >= 1) rinv = fmaf(x[g], ct_s[g], rinv);         // 1 / r_t (see sinkhorn_bwd_pass_kernel)
                }
#pragma unroll
                for (int g = 0; g < KMAX; ++g) {
                    const float e = d[g] - dot;
                    tsum[g] = fmaf(e, x[g], tsum[g]);
                    d[g] = e * rinv;
                }
                put(dcache, i, d);
            }
            reduce_lanes<KMAX, false>(tsum);
            store_warp(tsum);
            exchange(std::false_type{}, [&](int g, double total) {
                if (g < K) {
                    pend_sub_s[g] = (float)total;
                    pend_inv_s[g] = (float)(1.0 / sum);              // sum = T[t]
                    if (t >= 1) {
                        acc += log2_table(sum, tab_s);
                        sum = T[(size_t)(t - 1) * 32 + g];
                        ct_s[g] = (float)sum;
                    }
                }
                const double common = __shfl_sync(KMAX == 32 ? 0xffffffffu : (1u << KMAX) - 1u, acc, 0);
                if (g < K && t >= 1) voff_s[g] = (float)(t == 1 ? acc : acc - common);
            });
        }
        // dS = (e * Z_0 - B_0 * Y_0) / tau, e as pass 0 left it, B_0 in pend_sub_s
        for (int i = threadIdx.x; i < cnt; i += SKT_THREADS) {
            float x[KMAX], e[KMAX], y[KMAX];
            get(rows_s, i, x);
            get(dcache, i, e);
#pragma unroll
            for (int g = 0; g < KMAX; ++g) y[g] = ex2f(log2_units(x[g], voff_s[g]));            // Y_0 (may underflow to 0: then its term vanishes)
            const float inv = softmax_row(x);
#pragma unroll
            for (int g = 0; g < KMAX; ++g) e[g] = g < K ? (e[g] * (x[g] * inv) - pend_sub_s[g] * y[g]) * inv_tau : 0.f;
#pragma unroll
            for (int q = 0; q < PIECES; ++q) o[(size_t)i * PIECES + q] = make_float4(e[4 * q], e[4 * q + 1], e[4 * q + 2], e[4 * q + 3]);
        }
    }
    if (failed_s) {                                  // a wait ran out: no number that looks like a result
        const float bad = __int_as_float(0x7fffffff);
        for (int i = threadIdx.x; i < cnt * PIECES; i += SKT_THREADS) o[i] = make_float4(bad, bad, bad, bad);
    }
}

// Runs the call as one cooperative launch if the rows of every sequence fit in its team's shared memory and the context has the
// multiprocessors for all teams at once; `done` says whether it did.  A team has one block per 512 tokens, at most its share of
// the multiprocessors.
template <int KMAX, bool BWD, bool LATE = false>
static int launch_team(const focus_shape* s, const float* S, float tau, int iters, unsigned char* ws, const float* d_in, float* out,
                       cudaStream_t st, bool& done, long long late_limit = 0, unsigned int late_at = 0) {
    done = false;
    int rc;
    const int sms = launch_multiprocessors(st);      // (a capture takes a cooperative launch without asking whether its blocks fit)
    // (from about 1e36 on the lowest finite exponent of a row no longer stands for weight 0)
    if (s->batch > sms || tau > 1e30f) return 0;
    int P = sms / s->batch;
    if (P > skt_max_blocks(s->n)) P = skt_max_blocks(s->n);
    const int chunk = cdiv(cdiv(s->n, P), SKT_THREADS) * SKT_THREADS;        // whole rounds of the threads
    const size_t smem = (size_t)chunk * KMAX * sizeof(float) * (BWD ? 2 : 1);
    if (chunk > SKT_TOKENS || smem > SKT_SMEM) return 0;
    P = cdiv(s->n, chunk);                           // no block without tokens
    auto kern = sinkhorn_team_kernel<KMAX, BWD, LATE>;
    if ((rc = check_cuda(allow_smem<sinkhorn_team_kernel<KMAX, BWD, LATE>>(SKT_SMEM), "cudaFuncSetAttribute(sinkhorn)"))) return rc;
    cudaLaunchAttribute coop;
    coop.id = cudaLaunchAttributeCooperative;
    coop.val.cooperative = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(P * s->batch);
    cfg.blockDim = dim3(SKT_THREADS);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = &coop;
    cfg.numAttrs = 1;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, kern, S, s->n, s->K, iters, tau, 1.f / tau, ws, ws + s->batch * sk_seq_bytes(iters),
                                         skt_words_bytes(s), d_in, out, P, chunk, late_limit, late_at);
    if (e == cudaErrorCooperativeLaunchTooLarge) {   // a partition of the multiprocessors that does not hold the teams at once
        cudaGetLastError();                          // (not an error of the caller's)
        return 0;
    }
    done = true;
    return check_cuda(e, "sinkhorn launch");
}

size_t sinkhorn_workspace_bytes(const focus_shape* s, int iters) { return (size_t)s->batch * (sk_seq_bytes(iters) + skt_words_bytes(s)); }

template <int KMAX>
static int launch_sk(const focus_shape* s, const float* S, float tau, int iters, unsigned char* ws, float* out, cudaStream_t st) {
    const int n = s->n, K = s->K;
    int nblk = cdiv(n, SK_THREADS);
    if (nblk > SK_MAX_BLOCKS) nblk = SK_MAX_BLOCKS;
    const dim3 grid(nblk, s->batch);
    const float inv_tau = 1.f / tau;
    int rc = check_cuda(cudaMemsetAsync(ws, 0, sinkhorn_workspace_bytes(s, iters), st), "cudaMemsetAsync(sinkhorn workspace)");
    bool done = false;
    if (rc || (rc = launch_team<KMAX, false>(s, S, tau, iters, ws, nullptr, out, st, done)) || done) return rc;
    sinkhorn_colmax_kernel<KMAX><<<grid, SK_THREADS, 0, st>>>(S, n, K, iters, ws);
    sinkhorn_pass_kernel<KMAX, 0><<<grid, SK_THREADS, 0, st>>>(S, n, K, iters, 0, inv_tau, ws, nullptr);
    for (int pass = 1; pass < iters; ++pass)
        sinkhorn_pass_kernel<KMAX, 1><<<grid, SK_THREADS, 0, st>>>(S, n, K, iters, pass, inv_tau, ws, nullptr);
    sinkhorn_pass_kernel<KMAX, 2><<<grid, SK_THREADS, 0, st>>>(S, n, K, iters, iters, inv_tau, ws, out);
    return check_cuda(cudaGetLastError(), "sinkhorn kernel launch");
}

int launch_sinkhorn_stalled(const focus_shape* s, const float* S, float tau, int iters, void* ws, float* out, long long limit, int stall_at,
                            cudaStream_t st) {
    if (s->K > 4) return fail(FOCUS_ERR_UNSUPPORTED, "the stalled exchange takes K <= 4");
    unsigned char* w = reinterpret_cast<unsigned char*>(ws);
    int rc = check_cuda(cudaMemsetAsync(w, 0, sinkhorn_workspace_bytes(s, iters), st), "cudaMemsetAsync(sinkhorn workspace)");
    bool done = false;
    if (rc || (rc = launch_team<4, false, true>(s, S, tau, iters, w, nullptr, out, st, done, limit, (unsigned int)stall_at))) return rc;
    return done ? FOCUS_OK : fail(FOCUS_ERR_UNSUPPORTED, "the sequence does not fit the one-launch form");
}

int launch_sinkhorn(const focus_shape* s, const float* S, float tau, int iters, void* ws, float* out, cudaStream_t st) {
    unsigned char* w = reinterpret_cast<unsigned char*>(ws);
    if (s->K <= 4) return launch_sk<4>(s, S, tau, iters, w, out, st);
    if (s->K <= 8) return launch_sk<8>(s, S, tau, iters, w, out, st);
    if (s->K <= 16) return launch_sk<16>(s, S, tau, iters, w, out, st);
    return launch_sk<32>(s, S, tau, iters, w, out, st);
}

// ---- backward: d loss / d S from d loss / d g (paper Sec. 2 "Learned grouping": the Sinkhorn steps are differentiated
// through, step by step in reverse).  With X_0 = exp(S / tau) and per iteration t: c_t = column sums of X_t,
// Y_t = X_t / c_t, r_t = row sums of Y_t, Z_t = Y_t / r_t = X_{t+1}, a division by a sum along an axis has the
// derivative dX = (dZ - sum(dZ * Z)) / sum(X) along that axis.  Every X_t row follows from its score row and the
// column sums the forward passes leave in the workspace, so nothing but those sums is taped: pass t of the
// backward recomputes the row's X_t, applies the column step left over from iteration t + 1 (its column sums are
// complete by then), then the row step of iteration t, and adds the row into the column sums iteration t needs.
// For t = 0 the division by r_0 is left to the last kernel, which needs only Z_0 = Y_0 / r_0 and Y_0: r_0 itself
// underflows for a row whose scores all lie far below the column maxima.
//
// B = double [iters][32] per sequence: column sums of d * Y_t.
template <int KMAX>
__global__ void __launch_bounds__(SK_THREADS)
sinkhorn_bwd_pass_kernel(const float* __restrict__ S, int n, int K, int iters, int t, float inv_tau,
                         const unsigned char* __restrict__ ws, double* __restrict__ B, const float* __restrict__ d_in,
                         float* __restrict__ d_out) {
    __shared__ double red[SK_THREADS / 32][KMAX];
    __shared__ float colmax_s[KMAX], voff_s[KMAX], pend_sub_s[KMAX], pend_inv_s[KMAX], ct_s[KMAX];
    const int b = blockIdx.y;
    const unsigned char* wsb = ws + (size_t)b * sk_seq_bytes(iters);
    const double* T = reinterpret_cast<const double*>(wsb);
    const uint32_t* M = reinterpret_cast<const uint32_t*>(wsb + (size_t)(iters + 1) * 32 * sizeof(double));
    double* Bb = B + (size_t)b * iters * 32;
    const float* Sb = S + (size_t)b * n * KMAX;
    const bool pending = t + 1 < iters;            // the column step of iteration t + 1 has not been applied yet
    if (threadIdx.x < KMAX) {
        const int g = threadIdx.x;
        float cm = 0.f, v = 0.f, ps = 0.f, pi = 0.f;
        if (g < K) {
            cm = float_of_ordered(M[g]);
            // log Y_t = (S - M) / tau - sum_{m <= t} log T[m]  (+ the row's own offset when t >= 1)
            double acc = 0.0;
            for (int m = 0; m <= t; ++m) acc -= log(T[(size_t)m * 32 + g]);
            v = (float)acc;
            if (pending) {
                ps = (float)Bb[(size_t)(t + 1) * 32 + g];
                pi = (float)(1.0 / T[(size_t)(t + 1) * 32 + g]);
            }
        }
        colmax_s[g] = cm; voff_s[g] = v; pend_sub_s[g] = ps; pend_inv_s[g] = pi;
        ct_s[g] = (g < K && t >= 1) ? (float)T[(size_t)t * 32 + g] : 0.f;
    }
    __syncthreads();
    float tsum[KMAX];
#pragma unroll
    for (int g = 0; g < KMAX; ++g) tsum[g] = 0.f;
    for (int tok = blockIdx.x * SK_THREADS + threadIdx.x; tok < n; tok += gridDim.x * SK_THREADS) {
        float x[KMAX], d[KMAX];
        load_row<KMAX>(Sb, (size_t)tok, x);
        load_row<KMAX>(d_in + (size_t)b * n * KMAX, (size_t)tok, d);
        // Z_t = softmax over the groups of log Y_t up to the row's offset; r_t = the sum that normalises it
        float mx = -INFINITY;
#pragma unroll
        for (int g = 0; g < KMAX; ++g) {
            x[g] = (x[g] - colmax_s[g]) * inv_tau + voff_s[g];
            if (g < K) mx = fmaxf(mx, x[g]);
        }
        float se = 0.f;
#pragma unroll
        for (int g = 0; g < KMAX; ++g) {
            x[g] = g < K ? expf(x[g] - mx) : 0.f;
            se += x[g];
        }
        const float inv = 1.f / se;
        float dot = 0.f;
#pragma unroll
        for (int g = 0; g < KMAX; ++g) {
            x[g] *= inv;                                           // Z_t
            d[g] = g < K ? (pending ? (d[g] - pend_sub_s[g]) * pend_inv_s[g] : d[g]) : 0.f;
            dot = fmaf(d[g], x[g], dot);
        }
        // 1 / r_t for t >= 1: the row of X_t = Z_{t-1} sums to one, Y_t = X_t / c_t = Z_t r_t, so
        // sum_g Y_t,g c_t,g = 1 = r_t sum_g Z_t,g c_t,g
        float rinv = 1.f;
        if (t >= 1) {
            float zc = 0.f;
#pragma unroll
            for (int g = 0; g < KMAX; ++g) zc = fmaf(x[g], ct_s[g], zc);
            rinv = zc;
        }
#pragma unroll
        for (int g = 0; g < KMAX; ++g) {
            const float e = d[g] - dot;
            tsum[g] += e * x[g];                                   // (d - dot) / r_t * Y_t = (d - dot) * Z_t
            d[g] = g < K ? e * rinv : 0.f;                         // t = 0: left undivided
        }
        float4* o = reinterpret_cast<float4*>(d_out + ((size_t)b * n + tok) * KMAX);
#pragma unroll
        for (int c = 0; c < KMAX / 4; ++c) o[c] = make_float4(d[4 * c], d[4 * c + 1], d[4 * c + 2], d[4 * c + 3]);
    }
#pragma unroll
    for (int g = 0; g < KMAX; ++g) {
        float s = tsum[g];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5][g] = (double)s;
    }
    __syncthreads();
    if (threadIdx.x < K) {
        double s = 0.0;
        for (int w = 0; w < SK_THREADS / 32; ++w) s += red[w][threadIdx.x];
        atomicAdd(Bb + (size_t)t * 32 + threadIdx.x, s);
    }
}

// dS = ((d - dot_0) * Z_0 - B_0 * Y_0) / tau, with e = d - dot_0 as pass 0 left it
template <int KMAX>
__global__ void __launch_bounds__(SK_THREADS)
sinkhorn_bwd_last_kernel(const float* __restrict__ S, int n, int K, int iters, float inv_tau,
                         const unsigned char* __restrict__ ws, const double* __restrict__ B, const float* __restrict__ d_in,
                         float* __restrict__ d_out) {
    __shared__ float colmax_s[KMAX], voff_s[KMAX], b0_s[KMAX];
    const int b = blockIdx.y;
    const unsigned char* wsb = ws + (size_t)b * sk_seq_bytes(iters);
    const double* T = reinterpret_cast<const double*>(wsb);
    const uint32_t* M = reinterpret_cast<const uint32_t*>(wsb + (size_t)(iters + 1) * 32 * sizeof(double));
    const float* Sb = S + (size_t)b * n * KMAX;
    if (threadIdx.x < KMAX) {
        const int g = threadIdx.x;
        colmax_s[g] = g < K ? float_of_ordered(M[g]) : 0.f;
        voff_s[g] = g < K ? (float)(-log(T[g])) : 0.f;
        b0_s[g] = g < K ? (float)B[(size_t)b * iters * 32 + g] : 0.f;
    }
    __syncthreads();
    for (int tok = blockIdx.x * SK_THREADS + threadIdx.x; tok < n; tok += gridDim.x * SK_THREADS) {
        float x[KMAX], e[KMAX];
        load_row<KMAX>(Sb, (size_t)tok, x);
        load_row<KMAX>(d_in + (size_t)b * n * KMAX, (size_t)tok, e);
        float mx = -INFINITY;
#pragma unroll
        for (int g = 0; g < KMAX; ++g) {
            x[g] = (x[g] - colmax_s[g]) * inv_tau + voff_s[g];     // log Y_0
            if (g < K) mx = fmaxf(mx, x[g]);
        }
        float se = 0.f, y[KMAX];
#pragma unroll
        for (int g = 0; g < KMAX; ++g) {
            y[g] = g < K ? expf(x[g]) : 0.f;                       // Y_0 (may underflow to 0: then its term vanishes)
            x[g] = g < K ? expf(x[g] - mx) : 0.f;
            se += x[g];
        }
        const float inv = 1.f / se;
#pragma unroll
        for (int g = 0; g < KMAX; ++g) e[g] = g < K ? (e[g] * (x[g] * inv) - b0_s[g] * y[g]) * inv_tau : 0.f;
        float4* o = reinterpret_cast<float4*>(d_out + ((size_t)b * n + tok) * KMAX);
#pragma unroll
        for (int c = 0; c < KMAX / 4; ++c) o[c] = make_float4(e[4 * c], e[4 * c + 1], e[4 * c + 2], e[4 * c + 3]);
    }
}

size_t sinkhorn_bwd_workspace_bytes(const focus_shape* s, int iters) {
    return sinkhorn_workspace_bytes(s, iters) + (size_t)s->batch * iters * 32 * sizeof(double);
}

template <int KMAX>
static int launch_sk_bwd(const focus_shape* s, const float* S, float tau, int iters, unsigned char* ws, const float* dG, float* dS,
                         cudaStream_t st) {
    const int n = s->n, K = s->K;
    int nblk = cdiv(n, SK_THREADS);
    if (nblk > SK_MAX_BLOCKS) nblk = SK_MAX_BLOCKS;
    const dim3 grid(nblk, s->batch);
    const float inv_tau = 1.f / tau;
    int rc = check_cuda(cudaMemsetAsync(ws, 0, sinkhorn_bwd_workspace_bytes(s, iters), st), "cudaMemsetAsync(sinkhorn workspace)");
    if (rc) return rc;
    double* B = reinterpret_cast<double*>(ws + sinkhorn_workspace_bytes(s, iters));
    bool done = false;
    if ((rc = launch_team<KMAX, true>(s, S, tau, iters, ws, dG, dS, st, done)) || done) return rc;
    // the forward's column sums again (no assignments written)
    sinkhorn_colmax_kernel<KMAX><<<grid, SK_THREADS, 0, st>>>(S, n, K, iters, ws);
    sinkhorn_pass_kernel<KMAX, 0><<<grid, SK_THREADS, 0, st>>>(S, n, K, iters, 0, inv_tau, ws, nullptr);
    for (int pass = 1; pass < iters; ++pass)
        sinkhorn_pass_kernel<KMAX, 1><<<grid, SK_THREADS, 0, st>>>(S, n, K, iters, pass, inv_tau, ws, nullptr);
    for (int t = iters - 1; t >= 0; --t)
        sinkhorn_bwd_pass_kernel<KMAX><<<grid, SK_THREADS, 0, st>>>(S, n, K, iters, t, inv_tau, ws, B, t == iters - 1 ? dG : dS, dS);
    sinkhorn_bwd_last_kernel<KMAX><<<grid, SK_THREADS, 0, st>>>(S, n, K, iters, inv_tau, ws, B, dS, dS);
    return check_cuda(cudaGetLastError(), "sinkhorn backward kernel launch");
}

int launch_sinkhorn_bwd(const focus_shape* s, const float* S, float tau, int iters, void* ws, const float* dG, float* dS,
                        cudaStream_t st) {
    unsigned char* w = reinterpret_cast<unsigned char*>(ws);
    if (s->K <= 4) return launch_sk_bwd<4>(s, S, tau, iters, w, dG, dS, st);
    if (s->K <= 8) return launch_sk_bwd<8>(s, S, tau, iters, w, dG, dS, st);
    if (s->K <= 16) return launch_sk_bwd<16>(s, S, tau, iters, w, dG, dS, st);
    return launch_sk_bwd<32>(s, S, tau, iters, w, dG, dS, st);
}

}  // namespace focus
