// The sampling kernel with top-k / top-p, behind the streaming kernel.
#pragma once

#include "cfgzip_kernels.cuh"

namespace cfgzip {

// ---------------------------------------------------------------------------------------
// Second kernel of a sampling step with top-k / top-p: keeps, of the row's allowed tokens in the
// order (value, largest first; equal values by token id, lowest first), the first top_k (0 = all) and of those the
// shortest beginning whose weight reaches top_p times the weight of what top_k kept (>= 1: all), then draws among
// the kept tokens by inverse CDF in token order with the row's uniform number.
// Weights are 40-bit fixed-point integers (exp((z - M) / T) * 2^40), so every sum is exact whatever the order of the
// addends: the result is deterministic. A token whose weight is zero in that format can change neither a cumulative
// weight nor the draw.
//
// Ways through, all exact:
//   short  The streaming kernel has published the largest logit of every run of tokens; with top_k of every chunk of 31 to 64
//          vectors. The k-th largest of those is a bar that at least k tokens reach, and, the chunks being many, not many more
//          (k = 50: some 60), and only the chunks that reach it are read. For top-p alone the bar is where the run maxima by
//          themselves already weigh enough, or nearly (checked afterwards), and one pass over the row collects the tokens at or
//          above it. Up to kFiltThreads tokens get a lane or more each, which sums over all of them: their order needs no sort.
//   long   Otherwise (a flat distribution, a large k), with one filter: a pass that counts the tokens in 8192 steps of the
//          distance from the row maximum (one shared-memory addition a token; the weight of a step follows from its count to
//          better than 0.1 %), which says about where the cut falls; and a pass that sums, exactly and chunk by chunk, what
//          lies above a window of some 200 tokens around it and lists the tokens of the window. The exact sums then say whether
//          the cut lies in the window, and where; if it does not, they say where to lay the next one.
//   search Where three do not hold it (many equal logits), or with both filters, the kept set is { key > tau } plus the first m tokens,
//          in token order, with key == tau, where key is an order-preserving integer image of the logit; tau comes out of a
//          radix search over the row, twelve bits a pass.
// Bound: latency of a chain of block-wide steps, most of them executed once or twice, beside one or two passes over a row
// that is in the L2: loops stay rolled and steps that come up more than once are functions, which keeps the code a third of
// what it was inlined and unrolled. Collecting every token that carries weight first took 78 us of the step for 64 rows of
// 151936 bf16 logits at T = 0.7 (15000 such tokens a row), and some 30 passes over the row where they did not fit. With top_k this
// takes 9 of a step of 23.4 (a pass over the whole row, a claim on the list for every token and a sort: 13 of 27; the claims alone, one
// after the other, took 9000 of 19000 cycles). With top-p alone the same rows take 66 us (606), 256 rows that allow nearly
// everything 174 (1366).
// Where it is slower than collecting everything was: top-p alone on short rows of which every token that carries weight fitted
// one list (up to some 12000): 128 bf16 rows of 20032 with 1 % allowed 24 -> 37 us, with 10 % 31 -> 50 (with 90 % 147 -> 47). One
// row in a hundred that misses its guessed bar sets the time: count, window, list and the sort of some 500 tokens (10 us) one
// after the other. A lower bar to begin with lost 20 % with 90 % allowed; a second, lower bar for such rows gained 10 to 20 %
// in four of sixteen cases and lost as much in two.
//
// Thresholds (all ways are exact, what they choose is checked; they decide the time only): `0.04` and `0.6` of the guessed bar: with
// 0.02 or 0.01 256 rows of 151936 take 223 and 229 us instead of 203, 277 rows of 28864 75 instead of 58; kFiltWindow 200 tokens around
// the cut: 1 % of flat rows need a second window; kFiltWindowMost 800 tokens to a side: without it 277 rows of 28864 163 us instead of
// 58; `0.4` of the list's length as the lower bound on allowed tokens that skips counting them, `0.9` of what top-p leaves out as
// the weight that need not be listed, `0.25` of the list as the most tokens a guessed bar may be expected to pass, three tries, and
// top_k up to an eighth of the list: set once and not varied since.
// ---------------------------------------------------------------------------------------
// Threads of a block: much of the work is the same for every warp (scans, set-up) and takes issue slots once per warp; 256
// threads and two blocks per SM still keep 32 KB of loads in flight per SM and overlap one row's serial steps with another's.
constexpr int kFiltThreads = 256;
constexpr int kFiltWarps = kFiltThreads / 32;
constexpr int kFiltPeers = 8;       // most blocks that share a row
constexpr int kFiltList = 2048;     // tokens of the lists
constexpr int kFiltBits = 12, kFiltBuckets = 1 << kFiltBits;
constexpr int kFiltSteps = 8192, kFiltCoarse = kFiltThreads, kFiltFine = kFiltSteps / kFiltCoarse;  // the long way's steps
constexpr int kFiltWindow = 200;    // tokens the window of the long way aims at
constexpr unsigned int kFiltWindowMost = 800;  // and holds at most to either side, whole coarse steps
constexpr int kFiltTries = 3;       // windows before the search
constexpr int kFiltChunks = 512;    // most chunks of the draw's pass
constexpr int kFiltMaxima = 2048;   // most chunks whose maxima the streaming kernel leaves (of its own chunks)
constexpr float kFixOne = 1099511627776.f;  // 2^40

// Order-preserving integer image of a logit and its inverse. bf16 logits only use the upper half of the float's
// bits, so their keys are 16 bits wide.
template <int DT>
__device__ __forceinline__ uint32_t logit_key(float z) {
    z = z == 0.f ? 0.f : z;  // -0.0 and +0.0 are the same value
    const uint32_t b = __float_as_uint(z);
    const uint32_t k = (b & 0x80000000u) ? ~b : (b | 0x80000000u);
    return DT == kBF16 ? k >> 16 : k;
}
template <int DT>
__device__ __forceinline__ float key_logit(uint32_t k) {
    if (DT == kBF16) k = (k << 16) | ((k & 0x8000u) ? 0u : 0xFFFFu);  // the lower half of a negative value's key is all ones
    return __uint_as_float((k & 0x80000000u) ? (k & 0x7FFFFFFFu) : ~k);
}
// 2^40 exp2((z - M) scale), truncated, for z <= M (-inf: 0): the mantissa shifted into place, as a conversion to 64 bits is
// slower (its leading one from bit 63 down by 23 and by as many as the exponent is below zero).
__device__ __forceinline__ unsigned long long fixed_weight(float z, float M, float scale) {
    const uint32_t b = __float_as_uint(ex2f((z - M) * scale));
    unsigned long long w;
    asm("{\n\t.reg .b64 t;\n\tmov.b64 t, {%1, %2};\n\tshr.b64 %0, t, %3;\n\t}"
        : "=l"(w)
        : "r"(0u), "r"((b << 8) | 0x80000000u), "r"(150u - (b >> 23)));
    return w;
}

struct CountMass {
    unsigned int n;
    unsigned long long w;
};
__device__ __forceinline__ void operator+=(CountMass& a, const CountMass& b) {
    a.n += b.n;
    a.w += b.w;
}

// Shared memory of a block.
struct FiltShared {
    union {
        struct {  // count and weight of the buckets; weights as two 32-bit halves, which keeps every atomic a native one
            unsigned int n[kFiltBuckets], lo[kFiltBuckets], hi[kFiltBuckets];
        } hist;
        struct {  // tokens in every step of the distance from the row maximum; count and weight of kFiltFine of them together
            unsigned int n[kFiltSteps];
            uint2 coarse[kFiltCoarse];
        } steps;
        struct {
            uint2 list[kFiltList];                // logit, token id
            unsigned long long order[kFiltList];  // the list in order: key from the top, token id
            unsigned long long weight[kFiltList];
            struct {                // the draw's pass: kept weight above the cut and number of ties of every chunk
                unsigned long long above[kFiltChunks];
                unsigned int ties[kFiltChunks];
            } chunk;
        };
    };
    uint16_t chunks[kFiltMaxima];    // short way with top_k: the chunks whose largest logit reaches the bar
    unsigned int n_chunks;
    unsigned int bar[kFiltThreads];  // count or weight of the run maxima, by distance from the row maximum
    unsigned long long pick[8];  // result of a search, written into every block of the cluster by the first
    unsigned long long scan_w[2][kFiltWarps];
    unsigned int scan_n[2][kFiltWarps];
    unsigned long long peer_w[kFiltPeers];  // weight of the tokens of a block's share
    float warp_max[kFiltWarps], warp_sum[kFiltWarps];
    unsigned int list_n[1 + kFiltTries];  // of the short way's list and the windows' (they share their space, not their counts)
    uint32_t cut_key;
    int cut_id;
    unsigned int n_kept;
    unsigned long long kept_w, topk_w;
};

// Exclusive prefix of one (count, weight) pair per thread in thread order; total to everybody. The two sets of partial sums
// are used in turn (`turn` flips with every call of this and the next), so that one barrier per call is enough.
struct FiltScan {
    CountMass before, total;
};
__device__ __noinline__ FiltScan filt_scan(CountMass v, FiltShared& sh, int turn) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    CountMass inc = v;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const unsigned int un = __shfl_up_sync(0xFFFFFFFFu, inc.n, d);
        const unsigned long long uw = __shfl_up_sync(0xFFFFFFFFu, inc.w, d);
        if (lane >= d) inc += CountMass{un, uw};
    }
    if (lane == 31) {
        sh.scan_n[turn][warp] = inc.n;
        sh.scan_w[turn][warp] = inc.w;
    }
    __syncthreads();
    CountMass front{inc.n - v.n, inc.w - v.w}, all{0u, 0ull};
#pragma unroll
    for (int i = 0; i < kFiltWarps; ++i) {
        const CountMass t{sh.scan_n[turn][i], sh.scan_w[turn][i]};
        if (i < warp) front += t;
        all += t;
    }
    return FiltScan{front, all};
}
// The total alone: the warps' sums by integer reductions of 24 bits of the weight at a time (below 2^61).
__device__ __noinline__ CountMass filt_total(CountMass v, FiltShared& sh, int turn) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const unsigned int n = __reduce_add_sync(0xFFFFFFFFu, v.n);
    const unsigned int w0 = __reduce_add_sync(0xFFFFFFFFu, uint32_t(v.w) & 0xFFFFFFu),
                       w1 = __reduce_add_sync(0xFFFFFFFFu, uint32_t(v.w >> 24) & 0xFFFFFFu),
                       w2 = __reduce_add_sync(0xFFFFFFFFu, uint32_t(v.w >> 48));
    if (lane == 0) {
        sh.scan_n[turn][warp] = n;
        sh.scan_w[turn][warp] = w0 + (static_cast<unsigned long long>(w1) << 24) + (static_cast<unsigned long long>(w2) << 48);
    }
    __syncthreads();
    CountMass all{0u, 0ull};
#pragma unroll
    for (int i = 0; i < kFiltWarps; ++i) all += CountMass{sh.scan_n[turn][i], sh.scan_w[turn][i]};
    return all;
}

// How rows are cut into chunks (host): for the longest lead a row can have.
struct FiltGeom {
    int pieces, chunk, n_chunks, per_block;
};
inline FiltGeom filt_geom(int V, int n_peers) {
    FiltGeom g;
    g.pieces = (V + 7 + 256 * kFiltChunks - 1) / (256 * kFiltChunks);
    g.chunk = 256 * g.pieces;
    g.n_chunks = (V + 7 + g.chunk - 1) / g.chunk;
    g.per_block = (g.n_chunks + n_peers - 1) / n_peers;
    return g;
}

// The row as a block sees it. Rows are gone over eight tokens at a time from token -lead on, so that the eight are one vector
// of the row wherever the row starts. A chunk is 256 tokens (more only where that would be more than kFiltChunks of them);
// every block of the cluster takes a run of chunks, [c_begin, c_end).
struct FiltRow {
    const char* rowp;
    int V, lead, pieces, chunk, n_chunks, c_begin, c_end;
    float M, scale;
    float z_zero;  // a token takes part when its logit is at least this
    uint32_t crank, n_peers;
};

// Eight consecutive logits of the row from token t0 on (t0 + lead a multiple of 8), -inf outside the row.
template <int DT>
struct FiltOct {
    uint4 a, b;
};
template <int DT>
struct FiltNone {  // -inf in every element of a word
    static constexpr uint32_t word = DT == kBF16 ? 0xFF80FF80u : 0xFF800000u;
};
template <int DT>
__device__ __noinline__ FiltOct<DT> filt_edge(const char* rowp, int t0, int end) {  // rare: some of the eight lie outside
    constexpr int kPer = DT == kBF16 ? 2 : 1;
    uint32_t r[8];
#pragma unroll
    for (int q = 0; q < 8 / kPer; ++q) r[q] = FiltNone<DT>::word;
#pragma unroll
    for (int q = 0; q < 8; ++q)
        if (octet_has(t0, q, end)) {
            if (DT == kBF16) {
                const uint32_t x = __ldcg(reinterpret_cast<const unsigned short*>(rowp) + (t0 + q));
                r[q / kPer] = (q & 1) ? (r[q / kPer] & 0xFFFFu) | (x << 16) : (r[q / kPer] & 0xFFFF0000u) | x;
            } else {
                r[q] = __ldcg(reinterpret_cast<const unsigned int*>(rowp) + (t0 + q));
            }
        }
    FiltOct<DT> o;
    o.a = make_uint4(r[0], r[1], r[2], r[3]);
    o.b = DT == kF32 ? make_uint4(r[4], r[5], r[6], r[7]) : o.a;
    return o;
}
template <int DT>
__device__ __forceinline__ FiltOct<DT> filt_load(const char* rowp, int t0, int end) {
    constexpr uint32_t kNone = FiltNone<DT>::word;
    FiltOct<DT> o;
    o.a = o.b = make_uint4(kNone, kNone, kNone, kNone);
    octet_loads(
        t0, end,
        [&] {
            const char* p = rowp + int64_t(t0) * (DT == kBF16 ? 2 : 4);
            o.a = __ldcg(reinterpret_cast<const uint4*>(p));
            if (DT == kF32) o.b = __ldcg(reinterpret_cast<const uint4*>(p + 16));
        },
        [&] { o = filt_edge<DT>(rowp, t0, end); });
    return o;
}
template <int DT>
__device__ __forceinline__ void filt_floats(const FiltOct<DT>& o, float (&e)[8]) {
    const uint32_t r[8] = {o.a.x, o.a.y, o.a.z, o.a.w, o.b.x, o.b.y, o.b.z, o.b.w};
#pragma unroll
    for (int q = 0; q < 8; ++q)
        e[q] = DT == kF32 ? __uint_as_float(r[q]) : __uint_as_float((q & 1) ? r[q / 2] & 0xFFFF0000u : r[q / 2] << 16);
}
// Some of the eight tokens, bit q for token t0 + q, one after the other: f(token, logit).
template <typename F>
__device__ __forceinline__ void filt_each(const float (&e)[8], int t0, uint32_t which, F&& f) {
#pragma unroll 1
    while (which) {
        const int q = __ffs(int(which)) - 1;
        which &= which - 1u;
        const bool q0 = q & 1, q1 = q & 2;
        const float x = q1 ? (q0 ? e[3] : e[2]) : (q0 ? e[1] : e[0]), y = q1 ? (q0 ? e[7] : e[6]) : (q0 ? e[5] : e[4]);
        f(t0 + q, (q & 4) ? y : x);
    }
}
__device__ __forceinline__ uint32_t filt_at_least(const float (&e)[8], float least) {
    uint32_t m = 0u;
#pragma unroll
    for (int q = 0; q < 8; ++q) m |= e[q] >= least ? 1u << q : 0u;
    return m;
}
// The block's share eight tokens at a time, 128 bytes of loads in flight per thread: f(first token, logits). The bodies are
// free of branches (a masked logit is -inf and weighs nothing): what few tokens need comes after, through filt_each.
template <int DT, typename F>
__device__ __forceinline__ void filt_visit(const FiltRow& w, F&& f) {
    constexpr int kStep = kFiltThreads * 8;
    const int t_end = min(w.c_end * w.chunk - w.lead, w.V);
    constexpr int kHalf = DT == kBF16 ? 4 : 2;
#pragma unroll 1
    for (int t0 = w.c_begin * w.chunk - w.lead + int(threadIdx.x) * 8; t0 < t_end; t0 += 2 * kHalf * kStep) {
        FiltOct<DT> o[2 * kHalf];
#pragma unroll
        for (int r = 0; r < 2 * kHalf; ++r) o[r] = filt_load<DT>(w.rowp, t0 + r * kStep, t_end);
#pragma unroll 1
        for (int r = 0; r < kHalf; ++r) {  // (two bodies in the code: side by side they hide each other's latencies)
            FiltOct<DT> x = o[0], y = o[kHalf];
#pragma unroll
            for (int k = 1; k < kHalf; ++k) {
                if (r == k) x = o[k];
                if (r == k) y = o[kHalf + k];
            }
            float e[8], f8[8];
            filt_floats<DT>(x, e);
            filt_floats<DT>(y, f8);
            f(t0 + r * kStep, e);
            f(t0 + (kHalf + r) * kStep, f8);
        }
    }
}
// The same chunk by chunk, a warp each: f(first token, logits, sums of the chunk, this lane's part). The sums of a chunk (certain
// weight, number) go to the cluster's first block.
template <int DT, typename F>
__device__ __forceinline__ void filt_chunks(const FiltRow& w, FiltShared& sh, F&& f) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t above0 = peer_shared(sh.chunk.above, 0u), ties0 = peer_shared(sh.chunk.ties, 0u);
    // the warp's pieces (256 tokens) one after the other, four loads in flight
    int c = w.c_begin + warp, piece = 0, c_next = c, piece_next = 0;
    auto fetch = [&]() {
        const FiltOct<DT> o = filt_load<DT>(w.rowp, c_next * w.chunk + piece_next * 256 + lane * 8 - w.lead, c_next < w.c_end ? w.V : -8);
        if (++piece_next == w.pieces) {
            piece_next = 0;
            c_next += kFiltWarps;
        }
        return o;
    };
    CountMass v{0u, 0ull};
#pragma unroll 1
    while (c < w.c_end) {
        const FiltOct<DT> o0 = fetch(), o1 = fetch(), o2 = fetch(), o3 = fetch();
#pragma unroll 1
        for (int r = 0; r < 4 && c < w.c_end; ++r) {
            float e[8];
            filt_floats<DT>(r == 0 ? o0 : r == 1 ? o1 : r == 2 ? o2 : o3, e);
            f(c * w.chunk + piece * 256 + lane * 8 - w.lead, e, v);
            if (++piece == w.pieces) {
                v.n = __reduce_add_sync(0xFFFFFFFFu, v.n);
                const unsigned int w0 = __reduce_add_sync(0xFFFFFFFFu, uint32_t(v.w) & 0xFFFFFFu),
                                   w1 = __reduce_add_sync(0xFFFFFFFFu, uint32_t(v.w >> 24) & 0xFFFFFFu),
                                   w2 = __reduce_add_sync(0xFFFFFFFFu, uint32_t(v.w >> 48));
                if (lane == 0) {
                    st_peer_u64(above0 + uint32_t(c) * 8u,
                                w0 + (static_cast<unsigned long long>(w1) << 24) + (static_cast<unsigned long long>(w2) << 48));
                    st_peer_u32(ties0 + uint32_t(c) * 4u, v.n);
                }
                v = CountMass{0u, 0ull};
                piece = 0;
                c += kFiltWarps;
            }
        }
    }
}
// A token into one of the lists of the cluster's first block.
__device__ __noinline__ void filt_push(FiltShared& sh, int which, int t, float z) {
    const unsigned int at = add_peer_u32(peer_shared(&sh.list_n[which], 0u), 1u);
    if (at < kFiltList) {
        st_peer_u64(peer_shared(sh.list, 0u) + at * 8u, (static_cast<unsigned long long>(uint32_t(t)) << 32) | __float_as_uint(z));
    }
}

__device__ __noinline__ void hist_clear(FiltShared& sh, int bytes) {
    uint4* h = reinterpret_cast<uint4*>(&sh.hist);
    __syncthreads();
#pragma unroll 4
    for (int i = threadIdx.x; i < bytes / 16; i += kFiltThreads) h[i] = make_uint4(0u, 0u, 0u, 0u);
    __syncthreads();
}
__device__ __forceinline__ void hist_add(FiltShared& sh, uint32_t bucket, unsigned long long w) {
    atomicAdd(&sh.hist.n[bucket], 1u);
    const uint32_t lo = static_cast<uint32_t>(w);
    uint32_t hi = static_cast<uint32_t>(w >> 32);
    if (lo) {
        const uint32_t old = atomicAdd(&sh.hist.lo[bucket], lo);
        hi += (old + lo) < old ? 1u : 0u;  // the carry out of the lower half
    }
    if (hi) atomicAdd(&sh.hist.hi[bucket], hi);
}

// Threads that share a token when a block handles n <= kFiltThreads of them side by side.
__device__ __forceinline__ int lanes_per_token(unsigned int n) {
    return n <= kFiltThreads / 8u ? 8 : n <= kFiltThreads / 4u ? 4 : n <= kFiltThreads / 2u ? 2 : 1;
}

// The n tokens of the list into sh.order, by (key from the top, token id) and as one integer each. Up to kFiltThreads of them:
// every token counts those in front of it, 1 to 8 lanes a token; more: a bitonic sort. Called by all threads of the block.
template <int DT>
__device__ __noinline__ void filt_sort(FiltShared& sh, unsigned int n) {
    const int tid = threadIdx.x;
    auto entry = [&](unsigned int i) {
        const uint2 e = sh.list[i];
        return (static_cast<unsigned long long>(~logit_key<DT>(__uint_as_float(e.x))) << 32) | e.y;
    };
    unsigned long long* const v = sh.weight;  // (free until the order is known)
    if (n <= unsigned(kFiltThreads)) {
        if (unsigned(tid) < n) v[tid] = entry(tid);
        __syncthreads();
        const int lanes = lanes_per_token(n);
        const unsigned int i = tid / lanes, sub = tid & (lanes - 1);
        const unsigned long long me = i < n ? v[i] : 0ull;
        unsigned int rank = 0u;
#pragma unroll 8
        for (unsigned int k = sub; k < n; k += lanes) rank += v[k] < me ? 1u : 0u;
#pragma unroll 1
        for (int d = lanes >> 1; d >= 1; d >>= 1) rank += __shfl_xor_sync(0xFFFFFFFFu, rank, d);
        if (i < n && sub == 0) sh.order[rank] = me;
        __syncthreads();
        return;
    }
    unsigned int size = kFiltThreads * 2;
    while (size < n) size *= 2;
    for (unsigned int i = tid; i < size; i += kFiltThreads) sh.order[i] = i < n ? entry(i) : ~0ull;
    __syncthreads();
#pragma unroll 1
    for (unsigned int k = 2; k <= size; k *= 2)
#pragma unroll 1
        for (unsigned int d = k / 2; d >= 1; d /= 2) {
            for (unsigned int p = tid; p < size / 2; p += kFiltThreads) {
                const unsigned int x = p + (p & ~(d - 1u)), y = x + d;  // (d is a power of two)
                const unsigned long long vx = sh.order[x], vy = sh.order[y];
                if ((vx > vy) == ((x & k) == 0u)) {
                    sh.order[x] = vy;
                    sh.order[y] = vx;
                }
            }
            __syncthreads();
        }
}

// top_p's share of a weight, rounded up; at least one unit so that one token is kept
__device__ __forceinline__ unsigned long long filt_target(unsigned long long S, float top_p) {
    const unsigned long long t = static_cast<unsigned long long>(ceil(static_cast<double>(S) * static_cast<double>(top_p)));
    return t < 1ull ? 1ull : (t > S ? S : t);
}
// u times the kept weight, rounded down: the first token whose cumulative weight exceeds it is drawn
__device__ __forceinline__ unsigned long long filt_threshold(unsigned long long S_kept, float u) {
    const unsigned long long t = static_cast<unsigned long long>(static_cast<double>(u) * static_cast<double>(S_kept));
    return t >= S_kept ? S_kept - 1ull : t;
}

// The first bucket b with carry + sum(0 .. b) > threshold, over the histograms of all blocks of the cluster, by count or by
// weight. Threshold: `thr`, or, with top_p > 0, that share of the weight of all buckets less one. Left in the sh.pick of every
// block: [0] the bucket, all ones if there is none, [1] [2] count and weight in front of it (carry included), [3] [4] in it,
// [5] the threshold. Called by all threads of the cluster.
__device__ __noinline__ void hist_pick(FiltShared& sh, uint32_t crank, uint32_t n_peers, CountMass carry, bool by_weight,
                                       unsigned long long thr, float top_p, int turn) {
    constexpr int kPer = kFiltBuckets / kFiltThreads;  // consecutive buckets per thread
    static_assert(kPer % 4 == 0, "16-byte reads");
    const int tid = threadIdx.x;
    cluster_barrier();
    if (crank == 0u) {
        CountMass h[kPer];
#pragma unroll
        for (int b = 0; b < kPer; ++b) h[b] = CountMass{0u, 0ull};
#pragma unroll 1
        for (uint32_t p = 0; p < n_peers; ++p)
#pragma unroll
            for (int half = 0; half < kPer / 4; ++half) {
                const int at = tid * kPer + half * 4;
                const uint4 vn = ld_peer_v4(peer_shared(sh.hist.n + at, p)), vl = ld_peer_v4(peer_shared(sh.hist.lo + at, p)),
                            vh = ld_peer_v4(peer_shared(sh.hist.hi + at, p));
                h[half * 4 + 0] += CountMass{vn.x, (static_cast<unsigned long long>(vh.x) << 32) | vl.x};
                h[half * 4 + 1] += CountMass{vn.y, (static_cast<unsigned long long>(vh.y) << 32) | vl.y};
                h[half * 4 + 2] += CountMass{vn.z, (static_cast<unsigned long long>(vh.z) << 32) | vl.z};
                h[half * 4 + 3] += CountMass{vn.w, (static_cast<unsigned long long>(vh.w) << 32) | vl.w};
            }
        CountMass mine{0u, 0ull};
#pragma unroll
        for (int b = 0; b < kPer; ++b) mine += h[b];
        if (tid == 0) sh.pick[0] = ~0ull;
        const FiltScan s = filt_scan(mine, sh, turn);  // (its barrier also orders the line above before the writes below)
        if (top_p > 0.f) thr = filt_target(s.total.w, top_p) - 1ull;
        if (tid == 0) sh.pick[5] = thr;
        CountMass run = s.before;
        run += carry;
#pragma unroll
        for (int b = 0; b < kPer; ++b) {
            const unsigned long long below = by_weight ? run.w : run.n, here = by_weight ? h[b].w : h[b].n;
            if (below <= thr && thr < below + here) {
                sh.pick[0] = static_cast<unsigned long long>(tid * kPer + b);
                sh.pick[1] = run.n;
                sh.pick[2] = run.w;
                sh.pick[3] = h[b].n;
                sh.pick[4] = h[b].w;
            }
            run += h[b];
        }
        __syncthreads();
        for (int i = tid; i < 8 * int(n_peers - 1u); i += kFiltThreads)
            st_peer_u64(peer_shared(&sh.pick[i & 7], 1u + uint32_t(i >> 3)), sh.pick[i & 7]);
    }
    cluster_barrier();
}

// Where the steps say that the running count (or weight, in units of 2^-24 of the largest) passes `goal`, as a window of
// logits: above .x surely kept, from .y on to be looked at. Called by all
// threads of the cluster. Every block sums its steps kFiltFine at a time, the first block finds the coarse step and then the
// step, and takes as many steps to either side as hold some kFiltWindow tokens at the density found there.
template <int DT>
__device__ __noinline__ float2 filt_window(FiltShared& sh, const FiltRow& w, bool by_count, unsigned long long goal, float steps,
                                           int turn) {
    const int tid = threadIdx.x, lane = tid & 31;
    const float per_step = -w.scale / steps;  // powers of two from a step to the next
    auto step_weight = [&](int step) { return ex2f((0.5f + float(step)) * per_step); };  // of a token in the middle of it
    __syncthreads();
    {
        unsigned int n = 0u;
        float wt = 0.f;
        const float ratio = ex2f(per_step);
#pragma unroll 1
        for (int q = 0; q < kFiltFine; q += 4) {
            const int step = tid * kFiltFine + ((q + 4 * tid) & (kFiltFine - 1));  // (eight lanes on eight groups of banks)
            const uint4 c = *reinterpret_cast<const uint4*>(sh.steps.n + step);
            const unsigned int here = c.x + c.y + c.z + c.w;
            if (here) {
                n += here;
                const float x = fmaf(fmaf(fmaf(float(c.w), ratio, float(c.z)), ratio, float(c.y)), ratio, float(c.x));
                wt = fmaf(x, step_weight(step), wt);
            }
        }
        sh.steps.coarse[tid] = make_uint2(n, __float_as_uint(wt));
    }
    cluster_barrier();
    if (w.crank == 0u) {
        unsigned int n = 0u;
        float wt = 0.f;
#pragma unroll
        for (uint32_t p = 0; p < uint32_t(kFiltPeers); ++p)  // (unrolled: all in flight at once)
            if (p < w.n_peers) {
                const uint32_t at = peer_shared(&sh.steps.coarse[tid], p);
                n += ld_peer_u32(at);
                wt += __uint_as_float(ld_peer_u32(at + 4u));
            }
        if (tid == 0) sh.pick[0] = ~0ull;
        const CountMass mine{n, __float2ull_rz(wt * 16777216.f)};
        const FiltScan s = filt_scan(mine, sh, turn);
        const unsigned long long below = by_count ? s.before.n : s.before.w, here = by_count ? mine.n : mine.w;
        if (below <= goal && goal < below + here) {
            sh.pick[0] = static_cast<unsigned long long>(tid);
            sh.pick[1] = goal - below;
            sh.pick[2] = n;
            sh.pick[3] = s.before.n;
        }
        __syncthreads();
        // Where few tokens lie around the goal, below a peak, their density says little about the steps further down: the window
        // ends where the coarse steps in front of it hold kFiltWindowMost tokens on either side.
        const unsigned int through = s.before.n + n, goal_n = unsigned(sh.pick[3]);
        const int skip = __syncthreads_count(through + kFiltWindowMost <= goal_n),
                  reach = __syncthreads_count(through <= goal_n + kFiltWindowMost);
        if (tid < 32 && sh.pick[0] != ~0ull) {  // the step inside the coarse step, a lane each
            static_assert(kFiltFine == 32, "a lane per step");
            const int step = int(sh.pick[0]) * kFiltFine + lane;
            unsigned int c = 0u;
#pragma unroll
            for (uint32_t p = 0; p < uint32_t(kFiltPeers); ++p)
                if (p < w.n_peers) c += ld_peer_u32(peer_shared(&sh.steps.n[step], p));
            const unsigned long long x = by_count ? c : __float2ull_rz(float(c) * step_weight(step) * 16777216.f);
            unsigned long long inc = x;
#pragma unroll 1
            for (int d = 1; d < 32; d <<= 1) {
                const unsigned long long up = __shfl_up_sync(0xFFFFFFFFu, inc, d);
                if (lane >= d) inc += up;
            }
            const uint32_t past = __ballot_sync(0xFFFFFFFFu, inc > sh.pick[1]);
            const int in = past ? __ffs(int(past)) - 1 : kFiltFine - 1;
            const int at = int(sh.pick[0]) * kFiltFine + in;
            const float wide = fminf(0.5f * kFiltWindow * kFiltFine / float(unsigned(sh.pick[2])), float(kFiltSteps));
            const float first = fmaxf(float(at) - wide, float(skip * kFiltFine)),
                        beyond = fminf(float(at) + 1.f + wide, float(max(reach, int(sh.pick[0]) + 1) * kFiltFine));
            if (lane == in) {
                float hi = first > 0.f ? w.M - first / steps : INFINITY;
                float lo = beyond < float(kFiltSteps - 1) ? w.M - beyond / steps : w.z_zero;
                if (DT == kBF16) {
                    // all tokens of a step may be equal here and the next value several steps away: where the goal falls near
                    // an end of the step, the value beyond that end belongs into the window too
                    const uint32_t key = logit_key<DT>(w.M - (float(at) + 0.5f) / steps);
                    const unsigned long long into = sh.pick[1] - min(sh.pick[1], inc - x);
                    if (3ull * into < x) hi = fmaxf(hi, key_logit<DT>(key + 3u));
                    if (3ull * into > 2ull * x) lo = fminf(lo, key_logit<DT>(key - 2u));
                }
                sh.pick[6] = (static_cast<unsigned long long>(__float_as_uint(hi)) << 32) | __float_as_uint(fmaxf(lo, w.z_zero));
            }
        }
        if (tid == 0 && sh.pick[0] == ~0ull)  // nothing is cut away
            sh.pick[6] = (static_cast<unsigned long long>(__float_as_uint(w.z_zero)) << 32) | __float_as_uint(w.z_zero);
        __syncthreads();
        if (tid > 0 && tid < int(w.n_peers)) st_peer_u64(peer_shared(&sh.pick[6], uint32_t(tid)), sh.pick[6]);
    }
    cluster_barrier();
    return make_float2(__uint_as_float(uint32_t(sh.pick[6] >> 32)), __uint_as_float(uint32_t(sh.pick[6])));
}

// How the kept set ends: { key > tau } and, with key == tau, the first m tokens in token order that are not beyond id_cut.
struct FiltCut {
    uint32_t tau;
    int id_cut;
    unsigned int m;
    unsigned long long w_tie;
};

// Way 2: tau and m by radix search over the row, one filter after the other. Called by all threads of the cluster.
template <int DT>
__device__ __noinline__ FiltCut filt_search(const FiltRow& w, FiltShared& sh, int top_k, float top_p) {
    const uint32_t key_max = logit_key<DT>(w.M);
    const int bits = 32 - __clz(int(key_max - logit_key<DT>(w.z_zero)));  // of key_max - key
    FiltCut cut{0u, w.V, 0xFFFFFFFFu, 0ull};
    bool have = false;
    CountMass above{0u, 0ull}, ties{0u, 0ull};
    unsigned long long S = 0ull, target = 0ull;
    int turn = 0;
#pragma unroll 1
    for (int filter = 0; filter < 2; ++filter) {
        const bool by_weight = filter == 1;
        if (by_weight ? !(top_p < 1.f) : top_k <= 0) continue;
        if (by_weight && have) {
            target = filt_target(S, top_p);
            if (above.w < target) {  // reached among the ties at tau itself
                if (cut.w_tie > 0ull) {
                    const unsigned long long q = (target - above.w + cut.w_tie - 1ull) / cut.w_tie;
                    if (q < cut.m) cut.m = unsigned(q < 1ull ? 1ull : q);
                }
                continue;
            }
        }
        // the largest key whose tokens, with those above it, together count (weigh) more than the threshold
        unsigned long long thr = by_weight ? target - 1ull : static_cast<unsigned long long>(top_k) - 1ull, prefix = 0ull;
        CountMass front{0u, 0ull}, at{0u, 0ull};
        bool found = true;
        int hi = bits;
        do {
            const int lo = max(0, hi - kFiltBits);
            hist_clear(sh, sizeof(sh.hist));
            filt_visit<DT>(w, [&](int t0, const float (&e)[8]) {
                filt_each(e, t0, filt_at_least(e, w.z_zero), [&](int, float z) {
                    const unsigned long long x = key_max - logit_key<DT>(z);
                    if ((x >> hi) == prefix)
                        hist_add(sh, uint32_t(x >> lo) & ((1u << (hi - lo)) - 1u), fixed_weight(z, w.M, w.scale));
                });
            });
            // (without a cut so far the target follows from the weight of everything, which the first round sums)
            hist_pick(sh, w.crank, w.n_peers, front, by_weight, thr, by_weight && !have && hi == bits ? top_p : 0.f, turn);
            turn ^= 1;
            if (sh.pick[0] == ~0ull) {  // (a top_k beyond everything that carries weight cuts nothing away)
                found = false;
                break;
            }
            thr = sh.pick[5];
            prefix = (prefix << (hi - lo)) | sh.pick[0];
            front = CountMass{static_cast<unsigned int>(sh.pick[1]), sh.pick[2]};
            at = CountMass{static_cast<unsigned int>(sh.pick[3]), sh.pick[4]};
            hi = lo;
        } while (hi > 0);
        if (!found) continue;
        above = front;
        ties = at;
        cut.tau = key_max - uint32_t(prefix);
        cut.w_tie = fixed_weight(key_logit<DT>(cut.tau), w.M, w.scale);
        unsigned long long q = ties.n;  // all the ties unless fewer reach the threshold
        if (!by_weight)
            q = static_cast<unsigned long long>(top_k) - above.n;
        else if (cut.w_tie > 0ull)
            q = (thr + 1ull - above.w + cut.w_tie - 1ull) / cut.w_tie;
        cut.m = unsigned(q < 1ull ? 1ull : (q > ties.n ? ties.n : q));
        S = above.w + static_cast<unsigned long long>(cut.m) * cut.w_tie;
        have = true;
    }
    return cut;
}

// How many tokens the row's class mask allows, or all ones where `least` (every thread's part of a lower bound) says too many for
// the list. A lane per class: the masks that get here allow few of them. Called by all threads of the block.
__device__ __noinline__ unsigned int filt_allowed(const StepArgs& a, const PartDev& P, int row, float least, FiltShared& sh) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    __syncthreads();
#pragma unroll 1
    for (int d = 16; d >= 1; d >>= 1) least += __shfl_xor_sync(0xFFFFFFFFu, least, d);
    if (lane == 0) sh.warp_sum[warp] = least;
    __syncthreads();
    least = 0.f;
#pragma unroll
    for (int i = 0; i < kFiltWarps; ++i) least += sh.warp_sum[i];
    if (least > 0.4f * kFiltList) return ~0u;  // (it usually says half and less)
    const uint32_t* cm = a.class_mask + int64_t(row) * a.cm_stride;
    unsigned int n = 0u;
#pragma unroll 4
    for (int k = tid; k < P.K; k += kFiltThreads)
        if ((ld_after_wait(cm + (k >> 5)) >> (k & 31)) & 1u) n += unsigned(__ldg(P.off + k + 1) - __ldg(P.off + k));
    n = __reduce_add_sync(0xFFFFFFFFu, n);
    __syncthreads();
    if (lane == 0) sh.warp_sum[warp] = __uint_as_float(n);
    __syncthreads();
    n = 0u;
#pragma unroll
    for (int i = 0; i < kFiltWarps; ++i) n += __float_as_uint(sh.warp_sum[i]);
    return n;
}

// One row per cluster of blocks (1 to 8 of them: a short batch has fewer rows than the device has multiprocessors).
// Every block goes over its share of the row; what they find meets in the shared memory of the cluster's first block.
// FINE: with top_k, from the maxima of the chunks.
template <int DT, bool FINE>
__global__ void __launch_bounds__(kFiltThreads, 2) k_sample_filtered(const __grid_constant__ StepArgs a, const FiltGeom geom,
                                                                     int top_k, float top_p) {
    extern __shared__ __align__(16) unsigned char filt_smem[];
    FiltShared& sh = *reinterpret_cast<FiltShared*>(filt_smem);
    // (without a row plan the row is known, and what follows from it reads no memory, while the kernel in front finishes)
    pdl_launch_dependents();
    if (a.group_rows) pdl_wait();
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    FiltRow w;
    w.n_peers = cluster_blocks();
    w.crank = cluster_rank();
    const int slot = blockIdx.x / w.n_peers;  // the blocks of a cluster are neighbours along x
    const int g = slot / kGroupRows, j = slot - g * kGroupRows;
    // (every way out before the cluster's barriers depends on the row alone, so the blocks of a cluster take it together)
    if (a.n_groups && g >= ld_after_wait(a.n_groups)) return;
    int row;
    if (a.group_rows) {
        row = a.group_rows[g * kGroupRows + j];
    } else {
        row = g * kGroupRows + j;
        if (row >= a.B) row = -1;
    }
    if (row < 0) return;
    const float scale = a.scale, zero_at = 41.f / scale;
    w.scale = scale;
    w.V = a.V;
    w.rowp = reinterpret_cast<const char*>(a.logits) + int64_t(row) * a.row_stride * (DT == kBF16 ? 2 : 4);
    w.lead = (8 - row_head<DT>(w.rowp, 8)) & 7;
    w.pieces = geom.pieces;
    w.chunk = geom.chunk;
    w.n_chunks = geom.n_chunks;
    w.c_begin = min(int(w.crank) * geom.per_block, w.n_chunks);
    w.c_end = min(w.c_begin + geom.per_block, w.n_chunks);
    if (tid < 1 + kFiltTries) sh.list_n[tid] = 0u;
    sh.bar[tid] = 0u;
    if (tid == 0) sh.n_chunks = 0u;
    if (!a.group_rows) pdl_wait();
    PartDev P = a.p0;
    if (a.group_part) {
        P = a.parts[a.group_part[g]];
    } else if (a.row_part) {
        const int part = a.row_part[row];
        if (part < 0 || part >= a.n_parts || !a.parts[part].live || a.parts[part].V != a.V) return;  // counted by the step kernel
        P = a.parts[part];
    }
    // the run states the streaming kernel published: the row maximum, and the maxima and sums of up to four runs per thread
    // for the bar of the short way (leaving runs out only lowers the bar)
    // (top_k: the maxima of the chunks, and the few tokens outside the vectors)
    const Partial* src = row_slots(a, g, j);
    const float* const maxima = a.chunk_max + int64_t(row) * a.n_chunks;
    const int n_states = FINE ? a.n_chunks : group_states(a, g);
    const int fine_head = FINE && a.shifted ? row_head<DT>(w.rowp, a.V) : 0, fine_end = fine_head + ((a.V - fine_head) & ~7);
    const int edge_t = tid < 8 ? tid : fine_end + tid - 8;
    float edge_z = -INFINITY;
    if (FINE && tid < 16 && (tid < 8 ? edge_t < fine_head : edge_t < a.V)) edge_z = ldcg_elem<DT>(w.rowp, edge_t);
    const float u = ld_after_wait(a.u + row);  // needed late
    constexpr int kKeep = 4;
    float run_m[kKeep], run_s[kKeep], M = edge_z;
#pragma unroll
    for (int q = 0; q < kKeep; ++q) {
        const int k = tid + q * kFiltThreads;
        float2 r = make_float2(-INFINITY, 0.f);
        if (k < n_states) {
            if (FINE) r.x = __ldcg(maxima + k);
            else r = __ldcg(reinterpret_cast<const float2*>(src + k));
        }
        run_m[q] = r.x;
        run_s[q] = r.y;
        M = fmaxf(M, r.x);
    }
#pragma unroll 1
    for (int k = tid + kKeep * kFiltThreads; k < n_states; k += kFiltThreads) M = fmaxf(M, __ldcg(FINE ? maxima + k : &src[k].m));
    M = float_from_order_key(__reduce_max_sync(0xFFFFFFFFu, float_order_key(M)));
    if (lane == 0) sh.warp_max[warp] = M;
    __syncthreads();
    M = float_from_order_key(__reduce_max_sync(0xFFFFFFFFu, float_order_key(sh.warp_max[lane & (kFiltWarps - 1)])));
    if (!(M > kRefFloor)) {
        // nothing allowed, or only -inf allowed: the lowest allowed token (if any) and -inf logs
        if (warp == 0 && w.crank == 0) {
            unsigned long long cand = first_allowed_share(a, P, row, lane, 32);
#pragma unroll 1
            for (int d = 16; d >= 1; d >>= 1) {
                const unsigned long long other = __shfl_xor_sync(0xFFFFFFFFu, cand, d);
                cand = other < cand ? other : cand;
            }
            if (lane == 0) write_row_outputs(a, row, -INFINITY, 0.f, cand);
        }
        return;
    }
    cluster_arrive();  // this block runs and its lists are empty (waited for before anything is pushed)
    w.M = M;
    // (below M - 40 / scale the fixed-point weight is zero; the extra unit covers the rounding of the threshold itself)
    w.z_zero = fmaxf(key_logit<DT>(logit_key<DT>(M - zero_at)), kRefFloor);
    int turn = 0;
    auto write_draw = [&](int token, float zt, unsigned long long S_kept, int repv) {
        const float l = logf(static_cast<float>(S_kept) * (1.f / kFixOne));
        a.argmax[row] = token;
        if (a.rep) a.rep[row] = repv;
        if (a.lse) a.lse[row] = fmaf(M, a.inv_t, l);
        if (a.logp_argmax) a.logp_argmax[row] = (zt - M) * a.inv_t - l;
    };

    // ---- way 0 (short): the bar
    int way = 1;
    float z_bar = w.z_zero;
    bool guess = false;   // top-p alone: whether the tokens above the bar weigh enough has to be seen
    float run_sum = 1.f;  // top-p alone: the weight of all tokens, relative to the largest, by the run sums
    if (top_k <= kFiltList / 8) {
        // The run maxima by distance from M, in kFiltThreads steps of the range of weights: their number (top-k), or their
        // weight in units of 2^-20 (top-p; rounded down, which only lowers the bar). For top-p the weight of all tokens is not
        // known exactly yet: the run sums give it to about 1e-5, the bar allows 1e-3.
        const float steps = float(kFiltThreads) * scale * (1.f / 41.5f);
        float sum = 0.f;
#pragma unroll
        for (int q = 0; q < kKeep; ++q)
            if (run_m[q] >= w.z_zero) {
                const float e = ex2f((run_m[q] - M) * scale);
                atomicAdd(&sh.bar[min(int((M - run_m[q]) * steps), kFiltThreads - 1)], top_k > 0 ? 1u : uint32_t(e * 1048576.f));
                sum += run_s[q] * e;
            }
        if constexpr (!FINE) {  // (their weight counts all the same; chunk maxima have none, and top_k needs none)
#pragma unroll 1
            for (int k = tid + kKeep * kFiltThreads; k < n_states; k += kFiltThreads) {
                const int4 raw = __ldcg(reinterpret_cast<const int4*>(src + k));
                if (__int_as_float(raw.x) >= w.z_zero) sum += __int_as_float(raw.y) * ex2f((__int_as_float(raw.x) - M) * scale);
            }
        }
        uint32_t goal = uint32_t(top_k) - 1u;
        if (top_k == 0) {
#pragma unroll
            for (int d = 16; d >= 1; d >>= 1) sum += __shfl_xor_sync(0xFFFFFFFFu, sum, d);
            if (lane == 0) sh.warp_sum[warp] = sum;
        }
        if (tid == 0) sh.pick[0] = ~0ull;
        __syncthreads();
        if (top_k == 0) {
            sum = 0.f;
#pragma unroll
            for (int i = 0; i < kFiltWarps; ++i) sum += sh.warp_sum[i];
            run_sum = sum;
            goal = uint32_t(fminf(fmaf(sum * top_p, 1.001f * 1048576.f, 2.f), 4294967040.f));  // (past any sum of run maxima: not found)
        }
        // the first step at which the running sum passes the goal; every warp finds its steps' part of it
        const uint32_t here = sh.bar[tid];
        uint32_t inc = here;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const uint32_t up = __shfl_up_sync(0xFFFFFFFFu, inc, d);
            if (lane >= d) inc += up;
        }
        if (lane == 31) sh.scan_n[turn][warp] = inc;
        __syncthreads();
        uint32_t before = inc - here, all = 0u;
#pragma unroll
        for (int i = 0; i < kFiltWarps; ++i) {
            before += i < warp ? sh.scan_n[turn][i] : 0u;
            all += sh.scan_n[turn][i];
        }
        // The run maxima fall short by little (two heavy tokens in one run, runs of few allowed tokens): a bar that leaves out run
        // maxima of 4 % of the weight top_p leaves out will do almost always, and the pass over the row says whether it did.
        // (Where the runs say so, that is: the part of them that reaches the bar tells how many tokens do, the weight of the others
        // how much lies below it.)
        if (top_k == 0 && goal >= all && float(all) >= 0.6f * float(goal)) {
            guess = true;
            goal = all - 1u - min(all - 1u, uint32_t(0.04f * (1.f - top_p) * run_sum * 1048576.f));
        }
        turn ^= 1;
        if (before <= goal && goal - before < here) sh.pick[0] = static_cast<unsigned long long>(tid);
        __syncthreads();
        const bool found = sh.pick[0] != ~0ull;
        if (found || top_k > 0) way = 0;  // (fewer runs with a token than top_k: collect every token)
        // (a little lower than the step's own edge, as the steps are computed in floating point; the last step holds
        // everything further off, rounded or not)
        if (found && sh.pick[0] + 1ull < kFiltThreads)
            z_bar = fmaxf(w.z_zero, M - (float(sh.pick[0]) + 1.01f) / steps - fabsf(M) * 1e-6f);
        if (guess) {
            z_bar = fmaxf(w.z_zero, fminf(z_bar, M + log2f(0.04f * (1.f - top_p) * run_sum) / scale));  // (nor single tokens of that weight)
            int reach = 0;
            float below = 0.f;
#pragma unroll
            for (int q = 0; q < kKeep; ++q) {
                reach += __syncthreads_count(run_m[q] >= z_bar);
                if (run_m[q] >= w.z_zero && run_m[q] < z_bar) below += run_s[q] * ex2f((run_m[q] - M) * scale);
            }
#pragma unroll
            for (int d = 16; d >= 1; d >>= 1) below += __shfl_xor_sync(0xFFFFFFFFu, below, d);
            if (lane == 0) sh.warp_sum[warp] = below;
            __syncthreads();
            below = 0.f;
#pragma unroll
            for (int i = 0; i < kFiltWarps; ++i) below += sh.warp_sum[i];
            const float runs = float(n_states), seen = fminf(runs, float(kKeep * kFiltThreads)), part = float(reach) / seen;
            if (part >= 1.f || -runs * log1pf(-part) > 0.25f * kFiltList || below * (runs / seen) / (1.f - part) > 0.5f * (1.f - top_p) * run_sum)
                way = 1, guess = false;
        }
        // Rows that allow no more tokens than the list holds (a run's sum, relative to its own maximum, is at most its tokens: most
        // other rows are told without counting): the tokens that one of them may weigh without all of them together
        // weighing what top_p leaves out need not be listed. (1 % of 57591 tokens, 308 f32 rows, T = 0.7, top-p 0.95: 110 -> 78 us)
        if (way == 1 && top_k == 0) {
            float least = 0.f;
#pragma unroll
            for (int q = 0; q < kKeep; ++q) least += run_s[q];
            const unsigned int allowed = filt_allowed(a, P, row, least, sh);
            if (allowed <= unsigned(kFiltList)) {
                way = 0;
                z_bar = fmaxf(w.z_zero, M - fabsf(M) * 1e-6f + fminf(0.f, log2f(0.9f * (1.f - top_p) * run_sum / float(allowed)) / scale));
            }
        }
    }
    cluster_wait();

    // ---- ways 0 and 1: a list of at most kFiltList tokens that holds the cut
    CountMass front{0u, 0ull};  // what lies above the listed tokens
    FiltCut cut{0u, a.V, 0xFFFFFFFFu, 0ull};
    unsigned int n = 0u;
    int tries = 0;  // windows looked at
    float2 window = make_float2(INFINITY, INFINITY);
    if (way == 1 && top_k > 0 && top_p < 1.f) way = 2;
#pragma unroll 1
    while (way < 2) {
        if (way == 0) {
            unsigned long long mine = 0ull;
            auto push = [&](int t, float z) { filt_push(sh, 0, t, z); };
            if constexpr (FINE) {
                // the chunks that reach the bar, dealt to the blocks by their number and there to the warps; 32 vectors at a time,
                // four loads in flight
                auto mine_too = [&](int c) { return (uint32_t(c) & (w.n_peers - 1u)) == w.crank; };
#pragma unroll
                for (int q = 0; q < kKeep; ++q)
                    if (run_m[q] >= z_bar && mine_too(tid + q * kFiltThreads)) sh.chunks[atomicAdd(&sh.n_chunks, 1u)] = uint16_t(tid + q * kFiltThreads);
#pragma unroll 1
                for (int k = tid + kKeep * kFiltThreads; k < n_states; k += kFiltThreads)
                    if (mine_too(k) && __ldcg(maxima + k) >= z_bar) sh.chunks[atomicAdd(&sh.n_chunks, 1u)] = uint16_t(k);
                if (w.crank == 0u && edge_z >= z_bar) push(edge_t, edge_z);
                __syncthreads();
                const int vecs = a.chunk_tokens >> 3, halves = (vecs + 31) >> 5, units = int(sh.n_chunks) * halves;
                constexpr int kFlight = 4;
#pragma unroll 1
                for (int i0 = warp; i0 < units; i0 += kFlight * kFiltWarps) {
                    FiltOct<DT> o[kFlight];
                    int t0[kFlight];
#pragma unroll
                    for (int r = 0; r < kFlight; ++r) {
                        const int i = i0 + r * kFiltWarps;
                        const int v = (halves == 2 ? (i & 1) * 32 : 0) + lane;
                        t0[r] = -1;
                        o[r].a = o[r].b = make_uint4(FiltNone<DT>::word, FiltNone<DT>::word, FiltNone<DT>::word, FiltNone<DT>::word);
                        if (i < units && v < vecs) {
                            const int t = fine_head + int(sh.chunks[halves == 2 ? i >> 1 : i]) * a.chunk_tokens + 8 * v;
                            if (t < fine_end) {
                                t0[r] = t;
                                const char* p = w.rowp + int64_t(t) * (DT == kBF16 ? 2 : 4);
                                o[r].a = __ldcg(reinterpret_cast<const uint4*>(p));
                                if (DT == kF32) o[r].b = __ldcg(reinterpret_cast<const uint4*>(p + 16));
                            }
                        }
                    }
                    // one claim on the list for the warp's tokens
                    uint32_t over = 0u;
#pragma unroll
                    for (int r = 0; r < kFlight; ++r) {
                        float e[8];
                        filt_floats<DT>(o[r], e);
                        over |= filt_at_least(e, z_bar) << (8 * r);
                    }
                    const unsigned int here = __popc(over);
                    unsigned int inc = here;
#pragma unroll
                    for (int d = 1; d < 32; d <<= 1) {
                        const unsigned int up = __shfl_up_sync(0xFFFFFFFFu, inc, d);
                        if (lane >= d) inc += up;
                    }
                    unsigned int at = 0u;
                    if (lane == 31 && inc) at = add_peer_u32(peer_shared(&sh.list_n[0], 0u), inc);
                    at = __shfl_sync(0xFFFFFFFFu, at, 31) + inc - here;
                    const uint32_t list0 = peer_shared(sh.list, 0u);
#pragma unroll 1
                    for (int r = 0; r < kFlight && over >> (8 * r); ++r) {
                        float e[8];
                        filt_floats<DT>(r == 0 ? o[0] : r == 1 ? o[1] : r == 2 ? o[2] : o[3], e);
                        filt_each(e, r == 0 ? t0[0] : r == 1 ? t0[1] : r == 2 ? t0[2] : t0[3], (over >> (8 * r)) & 0xFFu, [&](int t, float z) {
                            if (at < unsigned(kFiltList))
                                st_peer_u64(list0 + at * 8u, (static_cast<unsigned long long>(uint32_t(t)) << 32) | __float_as_uint(z));
                            ++at;
                        });
                    }
                }
            } else if (top_k > 0)
                filt_visit<DT>(w, [&](int t0, const float (&e)[8]) { filt_each(e, t0, filt_at_least(e, z_bar), push); });
            else
                filt_visit<DT>(w, [&](int t0, const float (&e)[8]) {
#pragma unroll
                    for (int q = 0; q < 8; ++q) mine += fixed_weight(e[q], M, scale);
                    filt_each(e, t0, filt_at_least(e, z_bar), push);
                });
            if (top_k == 0) {  // the weight of everything
                const unsigned long long all = filt_total(CountMass{0u, mine}, sh, turn).w;
                turn ^= 1;
                if (tid == 0) st_peer_u64(peer_shared(&sh.peer_w[w.crank], 0u), all);
            }
        } else {
            if (tries == 0) {
                const bool by_count = top_k > 0;
                // For top-p the steps need not reach down to weight zero: what lies more than `range` powers of two below M weighs
                // at most V 2^-range, half of what top_p leaves out.
                const float range = by_count ? 41.5f : fminf(41.5f, log2f(2.f * float(a.V) / ((1.f - top_p) * run_sum)) + 1.f);
                const float steps = float(kFiltSteps) * scale / range;
                const float z_low = fmaxf(w.z_zero, M - range / scale);
                hist_clear(sh, sizeof(sh.steps.n));
                filt_visit<DT>(w, [&](int, const float (&e)[8]) {
#pragma unroll
                    for (int q = 0; q < 8; ++q)
                        if (e[q] >= z_low) atomicAdd(&sh.steps.n[min(int((M - e[q]) * steps), kFiltSteps - 1)], 1u);
                });
                window = filt_window<DT>(sh, w, by_count,
                                         by_count ? static_cast<unsigned long long>(top_k) - 1ull
                                                  : __float2ull_rz(run_sum * top_p * 16777216.f),
                                         steps, turn);
                turn ^= 1;
            }
            // (a top_k beyond everything that carries weight cuts nothing away: the window is empty then)
            unsigned long long total = 0ull;
            filt_chunks<DT>(w, sh, [&](int t0, const float (&e)[8], CountMass& v) {
#pragma unroll
                for (int q = 0; q < 8; ++q) {
                    const unsigned long long wt = fixed_weight(e[q], M, scale);
                    const bool above = e[q] >= window.x;
                    v.w += above ? wt : 0ull;
                    total += wt;
                }
                const uint32_t above = filt_at_least(e, window.x), listed = filt_at_least(e, window.y) & ~above;
                v.n += __popc(above);
                filt_each(e, t0, listed, [&](int t, float z) { filt_push(sh, 1 + tries, t, z); });
            });
            const unsigned long long all = filt_total(CountMass{0u, total}, sh, turn).w;
            turn ^= 1;
            if (tid == 0) st_peer_u64(peer_shared(&sh.peer_w[w.crank], 0u), all);
        }
        cluster_barrier();  // everything has arrived
        n = ld_peer_u32(peer_shared(&sh.list_n[way + tries], 0u));  // (the same in every block of the cluster)
        if (way == 0 && (!guess || n > unsigned(kFiltList))) {
            if (n <= unsigned(kFiltList)) break;
            way = top_k > 0 && top_p < 1.f ? 2 : 1;  // (both filters: way 1 takes one only)
            continue;
        }
        // does the cut lie among the listed tokens? (or at their end, when nothing is cut away)
        if (w.crank == 0u) {
            front = CountMass{0u, 0ull};
            if (way == 1) {
                CountMass mine{0u, 0ull};
#pragma unroll 1
                for (int c = tid; c < w.n_chunks; c += kFiltThreads) mine += CountMass{sh.chunk.ties[c], sh.chunk.above[c]};
                front = filt_total(mine, sh, turn);
                turn ^= 1;
            }
            unsigned long long listed = 0ull, S = 0ull;
            if (n <= unsigned(kFiltList))
                for (unsigned int i = tid; i < n; i += kFiltThreads) listed += fixed_weight(__uint_as_float(sh.list[i].x), M, scale);
            listed = filt_total(CountMass{0u, listed}, sh, turn).w;
            turn ^= 1;
            for (uint32_t p = 0; p < w.n_peers; ++p) S += sh.peer_w[p];
            const unsigned long long target = filt_target(S, top_p);
            const bool ok = n <= unsigned(kFiltList) &&
                            (top_k > 0 ? (front.n < unsigned(top_k) && unsigned(top_k) <= front.n + n) || (n == 0u && front.n <= unsigned(top_k))
                                       : front.w < target && target <= front.w + listed);
            // A top-p cut beside the window (1 % of flat bf16 rows, whose next value is a hundred tokens away): the exact sums say
            // on which side and by how much weight, the window's own density how far. One more pass, the search takes ten.
            const bool again = !ok && way == 1 && top_k == 0 && n <= unsigned(kFiltList) && tries + 1 < kFiltTries;
            if (again && tid == 0) {
                const float per_token = (fminf(window.x, M) - window.y) / float(n + 1u);
                const bool up = front.w >= target;
                const float edge = up ? window.x : window.y;
                const float miss = static_cast<float>(up ? front.w - target : target - front.w - listed) * (1.f / kFixOne);
                const float wide = (1.25f * miss * ex2f((M - edge) * scale) + 0.5f * kFiltWindow) * per_token;
                float hi = up ? edge + wide : edge, lo = up ? edge : edge - wide;
                if (DT == kBF16) {  // (a value or two further on at least)
                    const uint32_t key = logit_key<DT>(edge);
                    if (up) hi = fmaxf(hi, key_logit<DT>(key + 2u));
                    else lo = fminf(lo, key_logit<DT>(key - 2u));
                }
                sh.pick[6] = (static_cast<unsigned long long>(__float_as_uint(hi)) << 32) | __float_as_uint(fmaxf(lo, w.z_zero));
            }
            __syncthreads();
            if (tid < int(w.n_peers)) {
                st_peer_u64(peer_shared(&sh.pick[7], uint32_t(tid)), ok ? 1ull : again ? 2ull : 0ull);
                if (again && tid > 0) st_peer_u64(peer_shared(&sh.pick[6], uint32_t(tid)), sh.pick[6]);
            }
        }
        cluster_barrier();
        if (sh.pick[7] == 1ull) break;
        if (sh.pick[7] == 2ull) {
            window = make_float2(__uint_as_float(uint32_t(sh.pick[6] >> 32)), __uint_as_float(uint32_t(sh.pick[6])));
            ++tries;
        } else {
            ++way;
        }
    }

    if (way < 2) {
        cluster_arrive();  // this thread has read the first block's count
        if (w.crank != 0u) {
            cluster_wait();
            return;
        }
        if (way == 0 && n <= unsigned(kFiltThreads)) {
            // Few tokens, one lane or more each: a token's place in the order and the weight in front of it, then the cut, then the kept
            // weight up to its place in token order.
            unsigned long long* const kept_weight = reinterpret_cast<unsigned long long*>(sh.list);  // (read once, by this thread)
            if (unsigned(tid) < n) {
                const uint2 e = sh.list[tid];
                sh.order[tid] = (static_cast<unsigned long long>(~logit_key<DT>(__uint_as_float(e.x))) << 32) | e.y;
                sh.weight[tid] = fixed_weight(__uint_as_float(e.x), M, scale);
            }
            __syncthreads();
            const int lanes = lanes_per_token(n);
            const unsigned int i = tid / lanes, sub = tid & (lanes - 1);
            const bool have = i < n;
            const unsigned long long me = have ? sh.order[i] : 0ull, mine = have ? sh.weight[i] : 0ull;
            const uint32_t id = uint32_t(me);
            const int repv = have ? __ldg(P.trep + id) : -1;  // (asked for early: one of them is the row's)
            unsigned int rank = 0u;
            unsigned long long before = 0ull;
#pragma unroll 4
            for (unsigned int k = sub; k < n; k += lanes)
                if (sh.order[k] < me) {
                    ++rank;
                    before += sh.weight[k];
                }
#pragma unroll 1
            for (int d = lanes >> 1; d >= 1; d >>= 1) {
                rank += __shfl_xor_sync(0xFFFFFFFFu, rank, d);
                before += __shfl_xor_sync(0xFFFFFFFFu, before, d);
            }
            const unsigned int end = top_k > 0 ? min(unsigned(top_k), n) : n;
            unsigned long long target = ~0ull;
            if (top_p < 1.f) {
                unsigned long long S = 0ull;
                if (top_k > 0) {
                    if (have && sub == 0 && rank + 1 == end) sh.topk_w = before + mine;
                    __syncthreads();
                    S = sh.topk_w;
                } else {
                    for (uint32_t p = 0; p < w.n_peers; ++p) S += sh.peer_w[p];
                }
                target = filt_target(S, top_p);
            }
            const bool kept = have && rank < end && before < target;
            if (have && sub == 0) {
                kept_weight[i] = kept ? mine : 0ull;
                if (kept && (rank + 1 == end || before + mine >= target)) sh.kept_w = before + mine;  // the last one that is kept
            }
            __syncthreads();
            const unsigned long long S_kept = sh.kept_w, thr = filt_threshold(S_kept, u);
            unsigned long long cum = 0ull;
#pragma unroll 4
            for (unsigned int k = sub; k < n; k += lanes) cum += uint32_t(sh.order[k]) <= id ? kept_weight[k] : 0ull;
#pragma unroll 1
            for (int d = lanes >> 1; d >= 1; d >>= 1) cum += __shfl_xor_sync(0xFFFFFFFFu, cum, d);
            cluster_wait();  // (long since complete: no block may leave while another reads its shared memory)
            if (kept && sub == 0 && mine > 0ull && cum - mine <= thr && thr < cum)
                write_draw(int(id), key_logit<DT>(~uint32_t(me >> 32)), S_kept, repv);
            return;
        }
        // the listed tokens in order, with the weight in front of each
        filt_sort<DT>(sh, n);
        const unsigned int per = (n + kFiltThreads - 1) / kFiltThreads, i0 = min(tid * per, n), i1 = min(i0 + per, n);
        unsigned long long sum = 0ull;
#pragma unroll 1
        for (unsigned int i = i0; i < i1; ++i) {
            const unsigned long long wt = fixed_weight(key_logit<DT>(~uint32_t(sh.order[i] >> 32)), M, scale);
            sh.weight[i] = wt;
            sum += wt;
        }
        unsigned long long before = front.w + filt_scan(CountMass{0u, sum}, sh, turn).before.w;
        turn ^= 1;
        const unsigned int end = top_k > 0 ? min(unsigned(top_k) - min(unsigned(top_k), front.n), n) : n;  // how many top_k keeps
        unsigned long long target = ~0ull;
        if (top_p < 1.f) {
            unsigned long long S = 0ull;
            if (top_k > 0) {  // (way 0)
                unsigned long long b = before;
#pragma unroll 1
                for (unsigned int i = i0; i < i1; ++i) {
                    b += sh.weight[i];
                    if (i + 1 == end) sh.topk_w = b;
                }
                __syncthreads();
                S = sh.topk_w;
            } else {
                for (uint32_t p = 0; p < w.n_peers; ++p) S += sh.peer_w[p];
            }
            target = filt_target(S, top_p);
        }
#pragma unroll 1
        for (unsigned int i = i0; i < min(i1, end); ++i) {
            const unsigned long long after = before + sh.weight[i];
            if (before < target && (i + 1 == end || after >= target)) {  // the last token that is kept
                sh.n_kept = i + 1;
                sh.kept_w = after;
                sh.cut_key = ~uint32_t(sh.order[i] >> 32);
                sh.cut_id = int(uint32_t(sh.order[i]));
            }
            before = after;
        }
        if (way == 0 || n > 0u) {
            __syncthreads();
            cut.tau = sh.cut_key;
            cut.id_cut = sh.cut_id;
            const unsigned int n_kept = sh.n_kept;
            // into the sums of their chunks
            if (way == 0) {
                for (int c = tid; c < w.n_chunks; c += kFiltThreads) {
                    sh.chunk.above[c] = 0ull;
                    sh.chunk.ties[c] = 0u;
                }
                __syncthreads();
            }
            for (unsigned int i = tid; i < n_kept; i += kFiltThreads)
                atomicAdd(&sh.chunk.above[(int(uint32_t(sh.order[i])) + w.lead) / w.chunk], sh.weight[i]);
            __syncthreads();
        }
        cluster_wait();
    } else {
        cut = filt_search<DT>(w, sh, top_k, top_p);
        filt_chunks<DT>(w, sh, [&](int t0, const float (&e)[8], CountMass& v) {
            filt_each(e, t0, filt_at_least(e, w.z_zero), [&](int, float z) {
                const uint32_t key = logit_key<DT>(z);
                if (key > cut.tau) v.w += fixed_weight(z, M, scale);
                else if (key == cut.tau) v.n += 1u;
            });
        });
        cluster_barrier();
        if (w.crank != 0u) return;
    }

    // ---- the draw, in token order: the chunk that holds it, then the token
    const unsigned int m = cut.m;
    const unsigned long long w_tie = cut.w_tie;
    auto kept_ties = [&](unsigned int before, unsigned int here) { return min(here, m > before ? m - before : 0u); };
    static_assert(kFiltChunks == 2 * kFiltThreads, "two chunks per thread");
    unsigned int ties0 = 0u, ties1 = 0u;
    unsigned long long above0 = 0ull, above1 = 0ull;
    if (2 * tid < w.n_chunks) ties0 = sh.chunk.ties[2 * tid], above0 = sh.chunk.above[2 * tid];
    if (2 * tid + 1 < w.n_chunks) ties1 = sh.chunk.ties[2 * tid + 1], above1 = sh.chunk.above[2 * tid + 1];
    unsigned int tie_base = 0u;
    if (w_tie > 0ull) {
        tie_base = filt_scan(CountMass{ties0 + ties1, 0ull}, sh, turn).before.n;
        turn ^= 1;
    }
    above0 += static_cast<unsigned long long>(kept_ties(tie_base, ties0)) * w_tie;
    above1 += static_cast<unsigned long long>(kept_ties(tie_base + ties0, ties1)) * w_tie;
    const FiltScan s = filt_scan(CountMass{0u, above0 + above1}, sh, turn);
    const unsigned long long S_kept = s.total.w, thr = filt_threshold(S_kept, u);
    if (s.before.w <= thr && thr < s.before.w + above0 + above1) {  // the one thread with the chunk that holds the draw
        const bool second = thr >= s.before.w + above0;
        sh.pick[0] = static_cast<unsigned long long>(2 * tid + (second ? 1 : 0));
        sh.pick[1] = s.before.w + (second ? above0 : 0ull);
        sh.pick[2] = tie_base + (second ? ties0 : 0u);
    }
    __syncthreads();
    if (warp != 0) return;
    unsigned long long run = sh.pick[1];
    unsigned int tie_run = unsigned(sh.pick[2]);
#pragma unroll 1
    for (int piece = 0; piece < w.pieces && run <= thr; ++piece) {
        const int t0 = int(sh.pick[0]) * w.chunk + piece * 256 + lane * 8 - w.lead;
        float e[8];
        filt_floats<DT>(filt_load<DT>(w.rowp, t0, w.V), e);
        unsigned int t_mine = 0u;
        filt_each(e, t0, filt_at_least(e, w.z_zero), [&](int, float z) { t_mine += logit_key<DT>(z) == cut.tau ? 1u : 0u; });
        unsigned int t_inc = t_mine;
#pragma unroll 1
        for (int d = 1; d < 32; d <<= 1) {
            const unsigned int up = __shfl_up_sync(0xFFFFFFFFu, t_inc, d);
            if (lane >= d) t_inc += up;
        }
        unsigned int seen = tie_run + t_inc - t_mine;
        auto weight_of = [&](int t, float z) {  // 0 for a token that is not kept; in token order
            const uint32_t key = logit_key<DT>(z);
            const bool in = key > cut.tau || (key == cut.tau && seen++ < m && t <= cut.id_cut);
            return in ? fixed_weight(z, M, scale) : 0ull;
        };
        unsigned long long w_mine = 0ull;
        filt_each(e, t0, filt_at_least(e, w.z_zero), [&](int t, float z) { w_mine += weight_of(t, z); });
        unsigned long long inc = w_mine;
#pragma unroll 1
        for (int d = 1; d < 32; d <<= 1) {
            const unsigned long long up = __shfl_up_sync(0xFFFFFFFFu, inc, d);
            if (lane >= d) inc += up;
        }
        unsigned long long cum = run + inc - w_mine;
        if (cum <= thr && thr < cum + w_mine) {
            seen = tie_run + t_inc - t_mine;
            filt_each(e, t0, filt_at_least(e, w.z_zero), [&](int t, float z) {
                const unsigned long long wt = weight_of(t, z);
                if (cum <= thr && thr < cum + wt) write_draw(t, z, S_kept, __ldg(P.trep + t));
                cum += wt;
            });
        }
        run += __shfl_sync(0xFFFFFFFFu, inc, 31);
        tie_run += __shfl_sync(0xFFFFFFFFu, t_inc, 31);
    }
}

}  // namespace cfgzip
