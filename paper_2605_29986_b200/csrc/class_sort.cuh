// Class lists on the GPU: the tokens sorted by class, ascending inside a class, and where every class starts. A stable
// radix sort of the token ids by class id, nine bits a pass: one pass up to 512 classes, two up to 262144. Every block
// takes a run of consecutive tokens of the current order, every warp of it a run of those, 32 at a time; lanes of one
// digit are found with a match, so that a class that holds most of the vocabulary costs one counter update per warp and
// round. (One warp walking all tokens in order took 1.77 ms at V = 128256; this: about 20 us.)
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>

namespace cfgzip {

constexpr int kSortBits = 9, kSortDigits = 1 << kSortBits;
constexpr int kSortWarps = 8, kSortThreads = kSortWarps * 32;

// Tokens per block: 1024 keeps 126 blocks busy at V = 128256; more only where the digit counts of all blocks would
// outgrow a scan by one block (1024 blocks).
inline int sort_tile(int V) { return 1024 * std::max(1, (V + (1 << 20) - 1) >> 20); }
inline int sort_blocks(int V) { return (V + sort_tile(V) - 1) / sort_tile(V); }
// words: one list of token ids, the digit counts of every block, alignment
inline size_t class_sort_scratch_words(int V) { return size_t(V) + size_t(sort_blocks(V)) * kSortDigits + 4; }

struct SortArgs {
    const int32_t* c;          // token -> class
    const int32_t* n_classes;  // dev, or null: K
    int V, K, tile, n_blocks, pass;
    int32_t *list, *other;     // the last pass writes `list`; the passes before it take turns
    int32_t* counts;           // [kSortDigits * n_blocks], digit by digit
};

__device__ __forceinline__ int sort_last_pass(const SortArgs& a) {
    const int top = (a.n_classes ? __ldg(a.n_classes) : a.K) - 1;
    return top > 0 ? (31 - __clz(top)) / kSortBits : 0;
}
__device__ __forceinline__ const int32_t* sort_source(const SortArgs& a, int last) {  // null: the tokens in order
    return a.pass == 0 ? nullptr : ((last - a.pass) & 1 ? a.list : a.other);
}

// Visit the tokens of this warp's part of the block's tile in order, 32 at a time: f(token, digit, lanes of that digit).
template <typename F>
__device__ __forceinline__ void sort_visit(const SortArgs& a, const int32_t* src, F&& f) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, part = a.tile / kSortWarps;
    const int begin = blockIdx.x * a.tile + warp * part, end = min(begin + part, a.V);
    for (int i0 = begin; i0 < end; i0 += 32) {
        const int i = i0 + lane;
        const bool have = i < end;
        const int t = have ? (src ? src[i] : i) : -1;
        const int d = have ? (a.c[t] >> (kSortBits * a.pass)) & (kSortDigits - 1) : kSortDigits + lane;  // no token: nobody's equal
        f(t, d, __match_any_sync(0xFFFFFFFFu, d));
    }
}

// The digits of every warp's part of the tile, counted by the warp's own lanes.
__device__ __forceinline__ void sort_warp_counts(const SortArgs& a, const int32_t* src, int32_t (&s_count)[kSortWarps][kSortDigits]) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int d = lane; d < kSortDigits; d += 32) s_count[warp][d] = 0;
    __syncwarp();
    sort_visit(a, src, [&](int t, int d, unsigned peers) {
        if (t >= 0 && lane == __ffs(int(peers)) - 1) s_count[warp][d] += __popc(peers);
        __syncwarp();
    });
    __syncthreads();
}

static __global__ void __launch_bounds__(kSortThreads) k_sort_count(const __grid_constant__ SortArgs a) {
    __shared__ int32_t s_count[kSortWarps][kSortDigits];
    const int last = sort_last_pass(a);
    if (a.pass > last) return;
    sort_warp_counts(a, sort_source(a, last), s_count);
    for (int d = threadIdx.x; d < kSortDigits; d += kSortThreads) {
        int n = 0;
#pragma unroll
        for (int w = 0; w < kSortWarps; ++w) n += s_count[w][d];
        a.counts[d * a.n_blocks + blockIdx.x] = n;
    }
}

// Exclusive prefix sum of the counts, one block, sixteen values per thread and round.
static __global__ void __launch_bounds__(1024) k_sort_scan(const __grid_constant__ SortArgs a) {
    __shared__ int s_warp[32];
    if (a.pass > sort_last_pass(a)) return;
    constexpr int kPer = 16;
    const int n = kSortDigits * a.n_blocks, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;  // n is a multiple of 16
    int carry = 0;
    for (int base = 0; base < n; base += 1024 * kPer) {
        const int i = base + tid * kPer;
        int4 v[kPer / 4];
        int mine = 0;
#pragma unroll
        for (int q = 0; q < kPer / 4; ++q) {
            v[q] = i < n ? reinterpret_cast<const int4*>(a.counts + i)[q] : make_int4(0, 0, 0, 0);
            mine += v[q].x + v[q].y + v[q].z + v[q].w;
        }
        int inc = mine;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const int up = __shfl_up_sync(0xFFFFFFFFu, inc, d);
            if (lane >= d) inc += up;
        }
        if (lane == 31) s_warp[warp] = inc;
        __syncthreads();
        int run = carry + inc - mine;
        for (int w = 0; w < 32; ++w) {
            if (w < warp) run += s_warp[w];
            carry += s_warp[w];
        }
        if (i < n)
#pragma unroll
            for (int q = 0; q < kPer / 4; ++q) {
                const int4 in = v[q];
                v[q] = make_int4(run, run + in.x, run + in.x + in.y, run + in.x + in.y + in.z);
                run += in.x + in.y + in.z + in.w;
                reinterpret_cast<int4*>(a.counts + i)[q] = v[q];
            }
        __syncthreads();
    }
}

static __global__ void __launch_bounds__(kSortThreads) k_sort_place(const __grid_constant__ SortArgs a) {
    __shared__ int32_t s_at[kSortWarps][kSortDigits];
    const int last = sort_last_pass(a);
    if (a.pass > last) return;
    const int32_t* src = sort_source(a, last);
    int32_t* dst = (last - a.pass) & 1 ? a.other : a.list;
    sort_warp_counts(a, src, s_at);
    for (int d = threadIdx.x; d < kSortDigits; d += kSortThreads) {  // counts of the warps -> where each of them starts
        int at = a.counts[d * a.n_blocks + blockIdx.x];
#pragma unroll
        for (int w = 0; w < kSortWarps; ++w) {
            const int n = s_at[w][d];
            s_at[w][d] = at;
            at += n;
        }
    }
    __syncthreads();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    sort_visit(a, src, [&](int t, int d, unsigned peers) {
        const int at = t >= 0 ? s_at[warp][d] : 0;
        __syncwarp();
        if (t >= 0) {
            dst[at + __popc(peers & ((1u << lane) - 1u))] = t;
            if (lane == __ffs(int(peers)) - 1) s_at[warp][d] = at + __popc(peers);
        }
        __syncwarp();
    });
}

// off[k] = first place of class k in the sorted list; every entry past the last class reads V (`entries` of them in all).
static __global__ void __launch_bounds__(256) k_class_bounds(const __grid_constant__ SortArgs a, int32_t* off, int entries) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    const int K = a.n_classes ? __ldg(a.n_classes) : a.K;
    if (i < a.V) {
        const int k = a.c[a.list[i]];
        if (i == 0 || a.c[a.list[i - 1]] != k) off[k] = i;
    }
    if (i >= K && i < entries) off[i] = a.V;
}

// ---- a partition's other tables from its two vectors, which are checked on the way (*bad: set when c or r do not describe
// a partition; ids out of range are replaced by 0 then, so that nothing behind this reads past a table) ------------------
// c16: c in 16 bits, padded to n entries with K; null when K does not fit
static __global__ void __launch_bounds__(256) k_load_tokens(int32_t* c, uint16_t* c16, int V, int n, int K, int32_t* bad) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= n) return;
    int k = K;
    if (t < V) {
        k = c[t];
        if (k < 0 || k >= K) {
            *bad = 1;
            c[t] = k = 0;
        }
    }
    if (c16) c16[t] = uint16_t(k);
}
// (c[r[k]] == k for every k also says that no class is empty)
static __global__ void __launch_bounds__(256) k_load_classes(const int32_t* c, const int32_t* r, int32_t* trep, int V, int K, int32_t* bad) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < K) {
        const int t = r[i];
        if (t < 0 || t >= V || c[t] != i) *bad = 1;
    }
    if (i < V) trep[i] = r[c[i]];
}

// c: token -> class, ids 0 .. K-1 without gaps. K: host value, or 0 with n_classes on the device (then up to V classes and
// V + 1 entries of off, else K + 1). scratch: class_sort_scratch_words(V) words. Launches only.
inline void class_sort(const int32_t* c, int V, const int32_t* n_classes, int K, int32_t* off, int32_t* tok, int32_t* scratch,
                       cudaStream_t st) {
    SortArgs a{};
    a.c = c;
    a.n_classes = n_classes;
    a.V = V;
    a.K = K;
    a.tile = sort_tile(V);
    a.n_blocks = sort_blocks(V);
    a.list = tok;
    a.counts = reinterpret_cast<int32_t*>((reinterpret_cast<uintptr_t>(scratch) + 15) & ~uintptr_t(15));
    a.other = a.counts + size_t(a.n_blocks) * kSortDigits;
    const int most = n_classes ? V : K;
    for (a.pass = 0; a.pass == 0 || ((most - 1) >> (kSortBits * a.pass)) > 0; ++a.pass) {
        k_sort_count<<<a.n_blocks, kSortThreads, 0, st>>>(a);
        k_sort_scan<<<1, 1024, 0, st>>>(a);
        k_sort_place<<<a.n_blocks, kSortThreads, 0, st>>>(a);
    }
    const int entries = most + 1;
    k_class_bounds<<<(std::max(V, entries) + 255) / 256, 256, 0, st>>>(a, off, entries);
}

}  // namespace cfgzip
