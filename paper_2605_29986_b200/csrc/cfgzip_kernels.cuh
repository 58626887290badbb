// Kernels of the decode-step path. All of them are bandwidth- or latency-bound
// scans: no tensor cores. Notation: V tokens, K classes, B rows, VW = ceil(V/32),
// KW = ceil(K/32); an "octet" is 8 consecutive tokens of one row (16 bytes of bf16,
// 32 bytes of f32, one byte of vocab mask).
#pragma once

#include <cuda.h>

#include "cfgzip_device.cuh"
#include "ranges.h"

namespace cfgzip {

// kMasksRows: rows on 16-byte boundaries, KW a multiple of 4 (the pipelined kernel copies every row, the others read four words
// at a time). kMasksBlock, groups of consecutive rows in the pipelined kernel and under several masks: the rows of a group are one piece
// of memory on a 16-byte boundary and are copied as such. kMasksStaged: any, word by word. (Three in four class counts leave the rows
// off these boundaries; us, word by word / the block: 96 bf16 rows of 128256 in 2080 classes 17.1 / 15.2, in 8224 20.1 / 16.6, 64 f32 rows in
// 16416 28.9 / 22.3.)
enum : int { kMasksStaged = 0, kMasksRows = 1, kMasksBlock = 2 };
constexpr uint32_t kMaskPiece = 2048;  // bytes of such a copy

// Arguments of one step (expand / fused), shared by the dense, sparse and generic kernels.
struct StepArgs {
    const PartDev* parts;
    int32_t part0;
    int32_t n_parts;
    const int32_t* row_part;    // dev [B] or null
    // row groups (dense kernels): null = implicit groups of 32 consecutive rows using part0
    const int32_t* group_part;  // dev [n_groups]
    const int32_t* group_rows;  // dev [n_groups * 32], -1 = empty slot, valid slots first
    const int32_t* n_groups;    // dev scalar
    const int32_t* group_w;     // dev [max_groups + 1] or null: row batches in the groups in front of each (the total from n_groups
                                // on); where the groups are more than the fewest they could be, the blocks of the launch are
                                // shared out by it (group_share), at most S per group
    int32_t max_groups;
    int32_t blocks;             // group_w: blocks of the streaming launch
    int32_t S_even;             // group_w: blocks of every group where the groups are the fewest they could be
    const uint32_t* class_mask;
    int64_t cm_stride;
    void* logits;
    int64_t row_stride;         // elements
    uint32_t* vocab_mask;       // nullable
    int64_t vm_stride;
    int32_t* argmax;
    int32_t* rep;
    float* logp_argmax;
    float* lse;
    int32_t B, V, VW;
    int32_t S;                  // CTAs that share one group (dense) or one row (sparse)
    int32_t slots;              // dense: published states per row (S * WT + 1)
    int32_t per_split;          // octets (dense) or vocab-mask words (sparse) per CTA
    int32_t WT;                 // dense: warps side by side along the vocabulary
    int32_t table_words;        // dense: shared-memory words of the bit-sliced class table
    int32_t stage_stride;       // dense: words per row of the class-mask staging area, 0 = no staging
    int32_t depth;              // pipelined dense kernel: stages per warp
    int32_t cm_bulk;            // how the class masks reach the class table: kMasksStaged, kMasksRows or kMasksBlock
    int32_t wide;               // every row of the logits starts on a 32-byte boundary: f32 octets go back as one 32-byte store
    int32_t stage_alias;        // pipelined dense kernel: the class-mask staging area lies over the start of the rings
    int32_t hold_warps;         // stage_alias: warps whose ring it covers; they start their copies after the table is built
    int32_t run_chunks;         // sampling step: every warp slot of the pipelined kernel takes one contiguous run of this
                                // many chunks, so that the published states of a row follow the token order
    int32_t chunk_tokens;       // tokens of one chunk of the pipelined kernel (256 or 512): sampling kernel's run length unit
    int32_t prefetch_items;     // pipelined kernel without a row plan: work items per warp whose logits are asked into the L2
                                // before the wait for the kernel in front (a hint; nothing is read until after the wait)
    int32_t rot_chunks;         // pipelined kernel, greedy step: the round-robin deal of a row batch's chunks starts this many
                                // warp slots further on for every next row batch of the group
    int32_t expire_test;        // test hook: the pipelined kernel reports its first completed wait as run out
    int32_t fold;               // pipelined kernel: the last block of a row group folds the group's states and writes the
                                // rows' results itself (no second kernel); tickets[g] counts the group's finished blocks
    int32_t fold_off;           // fold: byte offset, in dynamic shared memory, of the block's own (row, warp) states, which
                                // are merged to one state per row before they are published; 0 = warps publish directly
    int32_t* row_mode;          // automatic mode: dev [B], written by the class-list kernel, which runs first (1 = the row
                                // allowed so few tokens that that kernel finished it), read by the kernels after it; else null
    int32_t auto_permille;      // automatic mode: a row stays with the class lists when under this many thousandths of its tokens are allowed
    int32_t masks_per_row;      // > 0: several class masks per logits row (register dense kernel only): row r of the masks,
                                // vocab masks and results belongs to logits row r / masks_per_row, and the logits are not modified
    int32_t tail_state;         // sampling kernel: the last state of a row stands for the octets past the last whole vector
    int32_t head_state;         // sampling kernel: the first state of a row stands for the tokens in front of its first vector
                                // (rows off the vector grid)
    int32_t shifted;            // rows start anywhere: the vectors of a row begin at row_head tokens, not at token 0
    float scale;                // log2(e) / temperature: the sums are of exp(z / T); log2(e) in a greedy step
    float inv_t;                // 1 / temperature
    const float* u;             // sampling step: dev [B] uniform numbers in [0, 1), else null
    PartDev p0;                 // descriptor of part0 (saves a dependent load when rows do not mix partitions)
    Partial* partials;
    unsigned int* tickets;
    int32_t* status;            // [0] empty rows, [1] bad tokens, [2] bad rows, [3] copies that never arrived
    float* chunk_max;           // sampling step with top_k: dev [B][n_chunks] largest masked logit of every chunk; else null
    int32_t n_chunks;
};

// kMasksBlock: how much of group g is copied, whole 16 bytes (up to three words of the last row may be left).
__device__ __forceinline__ uint32_t mask_block_bytes(const StepArgs& a, int g) {
    const int rows = min(kGroupRows, a.B - g * kGroupRows);
    return (uint32_t(rows - 1) * uint32_t(a.cm_stride) + uint32_t(a.p0.KW)) * 4u & ~15u;
}

// Tokens in front of the first vector boundary of a row that may start anywhere (16 bytes for bf16, 32 for f32: an
// octet is one vector either way), and how many whole vectors follow.
template <int DT>
__device__ __forceinline__ int row_head(const char* rowp, int V) {
    constexpr unsigned ES = DT == kBF16 ? 2 : 4, kVec = 8 * ES;
    const unsigned past = unsigned(reinterpret_cast<uintptr_t>(rowp)) & (kVec - 1u);
    return min(V, int(((kVec - past) & (kVec - 1u)) / ES));
}

// The logits row behind row r of the masks and results (they differ when a logits row has several masks).
__device__ __forceinline__ int64_t logits_row(const StepArgs& a, int r) { return a.masks_per_row > 0 ? r / a.masks_per_row : r; }

// The two halves separately, for a kernel that sets itself up (nothing read from memory) while the kernel in
// front of it is still running and only then waits for it.
__device__ __forceinline__ void pdl_launch_dependents() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

__device__ __forceinline__ void pdl_prologue() {
    // Let the next kernel of the stream start its launch early, then wait until everything
    // launched before this kernel has completed. Both are no-ops without the launch attribute.
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
}

template <int DT>
__device__ __forceinline__ float ldcg_elem(const void* base, int64_t idx) {
    if (DT == kBF16) return __uint_as_float(uint32_t(__ldcg(reinterpret_cast<const unsigned short*>(base) + idx)) << 16);
    return __ldcg(reinterpret_cast<const float*>(base) + idx);
}

// Turn a merged row state into the row's outputs. `pos` is an octet index (pos_is_token
// false: the first allowed token of that octet whose value equals m is the choice) or the
// token index itself.
template <int DT>
__device__ void finalize_row(const StepArgs& a, const PartDev& P, int row, float m, float s, int pos,
                             bool pos_is_token) {
    if (row < 0) return;
    int tok = -1, repv = -1;
    float lsev = -INFINITY, lpa = -INFINITY;
    if (pos != kNoPos) {
        if (pos_is_token) {
            tok = pos;
        } else {
            const uint32_t* cm = a.class_mask + int64_t(row) * a.cm_stride;
            const void* base = reinterpret_cast<const char*>(a.logits) + int64_t(row) * a.row_stride * (DT == kBF16 ? 2 : 4);
            for (int j = 0; j < 8 && tok < 0; ++j) {
                const int t = 8 * pos + j;
                if (t >= a.V) break;
                const int k = P.c32[t];
                if (((cm[k >> 5] >> (k & 31)) & 1u) && ldcg_elem<DT>(base, t) == m) tok = t;
            }
        }
        if (tok >= 0) repv = P.trep[tok];
        if (m > kRefFloor && s > 0.f) {
            const float l = logf(s);
            lsev = m + l;
            lpa = -l;
        }
    } else {
        atomicAdd(a.status + 0, 1);
    }
    a.argmax[row] = tok;
    if (a.rep) a.rep[row] = repv;
    if (a.lse) a.lse[row] = lsev;
    if (a.logp_argmax) a.logp_argmax[row] = lpa;
}

// Same for a whole warp whose lanes all hold the row's merged state (octet position): lanes
// 0..15 test the 16 tokens from the winning octet on side by side. A row without a position either
// allows nothing or holds only -inf at its allowed tokens: the class lists give its lowest
// allowed token. Needs first_allowed_share / write_row_outputs (defined below).
template <int DT>
__device__ __forceinline__ void warp_finalize_row(const StepArgs& a, const PartDev& P, int row, float m, float s,
                                                  int pos, int lane);

// Eight tokens handled one element at a time: ragged tail of a row, or unaligned logits.
template <int DT>
__device__ __forceinline__ void octet_scalar(void* row_base, int o, int V, uint32_t byte, float (&f)[8]) {
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        const int t = 8 * o + j;
        f[j] = -INFINITY;
        if (t < V) {
            if ((byte >> j) & 1u)
                f[j] = load_elem<DT>(row_base, t);
            else
                store_neg_inf<DT>(row_base, t);
        }
    }
}

// Fill the 32 row slots of group g and return the partition the group uses.
__device__ __forceinline__ int group_rows_setup(const StepArgs& a, int g, int* s_row, int tid) {
    if (tid < kGroupRows) {
        int row;
        if (a.group_rows) {
            row = a.group_rows[g * kGroupRows + tid];
        } else {
            row = g * kGroupRows + tid;
            if (row >= a.B) row = -1;
        }
        s_row[tid] = row;
    }
    return a.group_part ? a.group_part[g] : a.part0;
}

// Copy words [k0, k1) of the class-mask rows of the group's 32 row slots to shared memory (`stage`, rows
// stage_stride words apart). A warp takes one row at a time with coalesced loads, four rows
// and two 32-word spans per pass, so up to eight loads per thread are in flight together.
__device__ __forceinline__ void stage_class_masks(const StepArgs& a, const int* s_row, uint32_t* stage, int warp, int lane, int n_warps,
                                                  int k0, int k1) {
    for (int r0 = warp; r0 < kGroupRows; r0 += 4 * n_warps) {
        for (int kw0 = k0 + lane; kw0 < k1; kw0 += 64) {
            uint32_t v[4][2];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int r = r0 + q * n_warps;
                const int row = r < kGroupRows ? s_row[r] : -1;
#pragma unroll
                for (int u = 0; u < 2; ++u) {
                    const int kw = kw0 + 32 * u;
                    v[q][u] = (row >= 0 && kw < k1) ? ld_after_wait(a.class_mask + int64_t(row) * a.cm_stride + kw) : 0u;
                }
            }
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int r = r0 + q * n_warps;
#pragma unroll
                for (int u = 0; u < 2; ++u) {
                    const int kw = kw0 + 32 * u;
                    if (r < kGroupRows && kw < k1) stage[r * a.stage_stride + kw - k0] = v[q][u];
                }
            }
        }
    }
}

// Bit-sliced class table of one row group: T[k] bit r = "row slot r allows class k", entries 32 k0 .. 32 k1 - 1.
// Entries K .. 32*(KW+1)-1 are zero, so that the padding class id K looks up "nobody" (k1 = KW + 1 writes them).
// The 32x32 bit blocks come from a staging area that starts with word k0 of every row; a stage_stride that is odd (or even
// and no multiple of 4) spreads its column reads over 32 (16) banks. BLOCK: words from `staged` on (counted through the
// area) are not in it and are read from global memory.
template <bool BLOCK, int U = 4>
__device__ __forceinline__ void build_class_table(const StepArgs& a, int K, int KW, const int* s_row, uint32_t* T, const uint32_t* stage,
                                                  int warp, int lane, int n_warps, int k0, int k1, int staged) {
    const uint32_t tail = (K & 31) ? (1u << (K & 31)) - 1u : 0xFFFFFFFFu;
    const int row = s_row[lane];
    for (int kw0 = k0 + warp; kw0 < k1; kw0 += n_warps * U) {
        uint32_t x[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int kw = kw0 + u * n_warps, at = lane * a.stage_stride + kw - k0;
            x[u] = 0u;
            if (kw < k1 && kw < KW && row >= 0) {
                if (!BLOCK || at < staged) x[u] = stage[at];
                else x[u] = ld_after_wait(a.class_mask + int64_t(row) * a.cm_stride + kw);
            }
            if (kw == KW - 1) x[u] &= tail;
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int kw = kw0 + u * n_warps;
            const uint32_t t = warp_transpose32(x[u], lane);  // independent chains: their shuffles overlap
            if (kw < k1) T[kw * 32 + lane] = t;
        }
    }
}
// The table as many words at a time as the staging area holds: all of them, or kMaskSlice (16416 classes a lane per row, read where
// they lie, word by word, took 29 of 43 us of a call with 8 x 16 masks). NARROW: where the table leaves no room for that, as many as it does
// (with a width the compiler does not know all slices are slower, 64 rows in 50000 classes 195 us instead of 160). Called by all threads
// of the block, which meet before the table is read.
constexpr int kMaskSlice = 128;
template <bool NARROW = false>
__device__ __forceinline__ void build_class_table_staged(const StepArgs& a, int K, int KW, const int* s_row, uint32_t* T, uint32_t* stage,
                                                         int warp, int lane, int n_warps) {
    const int span = NARROW ? a.stage_stride - 1 : a.stage_stride >= KW ? KW + 1 : kMaskSlice;
    for (int k0 = 0; k0 <= KW; k0 += span) {
        if (k0) __syncthreads();  // (the words before have been taken)
        stage_class_masks(a, s_row, stage, warp, lane, n_warps, k0, min(k0 + span, KW));
        __syncthreads();
        build_class_table<false>(a, K, KW, s_row, T, stage, warp, lane, n_warps, k0, min(k0 + span, KW + 1), 0);
    }
}
// The same as a function, for the kernel that hardly needs it: inlined there it cost the batches that do not up to 7 % (96 rows of
// 128256 bf16 in 8192 classes 14.9 -> 16.1 us).
__device__ __noinline__ void build_class_table_staged_call(const StepArgs& a, int K, int KW, uint32_t rows_at, uint32_t table_at,
                                                           uint32_t stage_at) {
    auto words = [](uint32_t at) { return reinterpret_cast<uint32_t*>(__cvta_shared_to_generic(at)); };
    build_class_table_staged(a, K, KW, reinterpret_cast<const int*>(words(rows_at)), words(table_at), words(stage_at), threadIdx.x >> 5,
                             threadIdx.x & 31, blockDim.x >> 5);
}
// For tables that leave no room for a whole slice: narrower ones, or every word where it lies. (A function for the same reason: inlined in
// k_step_dense it cost the tables that do not need it a quarter, 64 rows in 50000 classes 160 -> 205 us.)
__device__ __noinline__ void build_class_table_narrow_call(const StepArgs& a, int K, int KW, uint32_t rows_at, uint32_t table_at,
                                                           uint32_t stage_at) {
    auto words = [](uint32_t at) { return reinterpret_cast<uint32_t*>(__cvta_shared_to_generic(at)); };
    const int* const s_row = reinterpret_cast<const int*>(words(rows_at));
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, n_warps = blockDim.x >> 5;
    if (a.stage_stride) build_class_table_staged<true>(a, K, KW, s_row, words(table_at), words(stage_at), warp, lane, n_warps);
    else build_class_table<true, 8>(a, K, KW, s_row, words(table_at), words(stage_at), warp, lane, n_warps, 0, KW + 1, 0);
}

// The same table from a staging area whose rows are 16-byte aligned and stage_stride (a
// multiple of 4, with stage_stride/4 odd) words apart: a lane reads four words of its row at
// once, which spreads the eight lanes of a quarter warp over all 32 banks.
__device__ __forceinline__ void build_class_table_quads(const StepArgs& a, const PartDev& P, const int* s_row, uint32_t* T,
                                                        const uint32_t* stage, int warp, int lane, int n_warps) {
    const uint32_t tail = (P.K & 31) ? (1u << (P.K & 31)) - 1u : 0xFFFFFFFFu;
    const bool have = s_row[lane] >= 0;
    for (int q = warp; 4 * q < P.KW; q += n_warps) {  // KW is a multiple of 4 here
        uint4 x = make_uint4(0, 0, 0, 0);
        if (have) x = *reinterpret_cast<const uint4*>(stage + lane * a.stage_stride + 4 * q);
        if (4 * q + 4 == P.KW) x.w &= tail;
        const uint32_t t0 = warp_transpose32(x.x, lane), t1 = warp_transpose32(x.y, lane);
        const uint32_t t2 = warp_transpose32(x.z, lane), t3 = warp_transpose32(x.w, lane);
        uint32_t* dst = T + (4 * q) * 32 + lane;
        dst[0] = t0; dst[32] = t1; dst[64] = t2; dst[96] = t3;
    }
    if (warp == 0) T[P.KW * 32 + lane] = 0u;  // the padding class
}

// The same straight from the masks: rows on 16-byte boundaries, KW a multiple of 4, a lane reads four words of its row at once.
__device__ __forceinline__ void build_class_table_direct(const StepArgs& a, const PartDev& P, const int* s_row, uint32_t* T, int warp,
                                                         int lane, int n_warps) {
    const uint32_t tail = (P.K & 31) ? (1u << (P.K & 31)) - 1u : 0xFFFFFFFFu;
    const int row = s_row[lane];
    const uint4* const cm = reinterpret_cast<const uint4*>(a.class_mask + int64_t(row < 0 ? 0 : row) * a.cm_stride);
    constexpr int U = 2;
    for (int q0 = warp; 4 * q0 < P.KW; q0 += U * n_warps) {
        uint4 x[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int q = q0 + u * n_warps;
            x[u] = row >= 0 && 4 * q < P.KW ? ld_after_wait(cm + q) : make_uint4(0, 0, 0, 0);
            if (4 * q + 4 == P.KW) x[u].w &= tail;
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int q = q0 + u * n_warps;
            if (4 * q >= P.KW) break;
            uint32_t* const dst = T + q * 128 + lane;
            dst[0] = warp_transpose32(x[u].x, lane);
            dst[32] = warp_transpose32(x[u].y, lane);
            dst[64] = warp_transpose32(x[u].z, lane);
            dst[96] = warp_transpose32(x[u].w, lane);
        }
    }
    if (warp == 0) T[P.KW * 32 + lane] = 0u;  // the padding class
}
__device__ __forceinline__ void make_class_table(const StepArgs& a, const PartDev& P, const int* s_row, uint32_t* T, uint32_t* stage,
                                                 int warp, int lane, int n_warps) {
    if (a.cm_bulk) build_class_table_direct(a, P, s_row, T, warp, lane, n_warps);
    else build_class_table_staged(a, P.K, P.KW, s_row, T, stage, warp, lane, n_warps);
}
// For groups of consecutive rows: kMasksBlock too, the group's masks copied as one piece of memory.
__device__ __forceinline__ void make_class_table_of_group(const StepArgs& a, const PartDev& P, int g, const int* s_row, uint32_t* T,
                                                          uint32_t* stage, int warp, int lane, int n_warps) {
    if (a.cm_bulk != kMasksBlock) {
        make_class_table(a, P, s_row, T, stage, warp, lane, n_warps);
        return;
    }
    const uint32_t* const src = a.class_mask + int64_t(g * kGroupRows) * a.cm_stride;
    const int quads = int(mask_block_bytes(a, g) / 16u), words = (min(kGroupRows, a.B - g * kGroupRows) - 1) * a.stage_stride + P.KW;
#pragma unroll 4
    for (int i = threadIdx.x; i < quads; i += 32 * n_warps)
        reinterpret_cast<uint4*>(stage)[i] = ld_after_wait(reinterpret_cast<const uint4*>(src) + i);
    for (int i = 4 * quads + threadIdx.x; i < words; i += 32 * n_warps) stage[i] = ld_after_wait(src + i);
    __syncthreads();
    build_class_table<false>(a, P.K, P.KW, s_row, T, stage, warp, lane, n_warps, 0, P.KW + 1, 0);
}

// From the class words of 8 tokens: byte i of (lo, hi) belongs to row 8*rb + i, bit j of it to token j.
__device__ __forceinline__ void row_batch_bytes(const uint32_t (&w)[8], int rb, uint32_t& lo, uint32_t& hi) {
    const uint32_t sel = uint32_t(rb) | (uint32_t(4 + rb) << 4);  // byte rb of both operands
    lo = __byte_perm(__byte_perm(w[0], w[1], sel), __byte_perm(w[2], w[3], sel), 0x5410);
    hi = __byte_perm(__byte_perm(w[4], w[5], sel), __byte_perm(w[6], w[7], sel), 0x5410);
    transpose8x8(lo, hi);
}

// Allow bits of rows 8*rb .. 8*rb+7 for the 8 tokens whose class ids are packed in cv:
// byte i of (lo, hi) belongs to row 8*rb + i, bit j of it to token j of the octet.
__device__ __forceinline__ void octet_allow_bits(const uint4& cv, const uint32_t* T, int rb, bool active, uint32_t& lo,
                                                 uint32_t& hi) {
    lo = hi = 0;
    if (!active) return;
    const uint32_t w[8] = {T[cv.x & 0xFFFFu], T[cv.x >> 16], T[cv.y & 0xFFFFu], T[cv.y >> 16],
                           T[cv.z & 0xFFFFu], T[cv.z >> 16], T[cv.w & 0xFFFFu], T[cv.w >> 16]};
    row_batch_bytes(w, rb, lo, hi);
}

// Lowest allowed token of a row, found from the class side: the first member of every allowed
// class (the member lists are ascending), minimum over the classes this caller looks at
// (words l, l+n, ... of the class mask). Returns (token << 32) | representative, ~0 if none.
// Only rows whose allowed logits are all -inf (or that allow nothing) come here.
__device__ __forceinline__ unsigned long long first_allowed_share(const StepArgs& a, const PartDev& P, int row, int l,
                                                                  int n) {
    unsigned long long best = ~0ull;
    const uint32_t* cm = a.class_mask + int64_t(row) * a.cm_stride;
    for (int kw = l; kw < P.KW; kw += n) {
        uint32_t w = cm[kw];
        if (kw == P.KW - 1 && (P.K & 31)) w &= (1u << (P.K & 31)) - 1u;
        while (w) {
            const int k = kw * 32 + __ffs(w) - 1;
            w &= w - 1u;
            const unsigned long long cand =
                (static_cast<unsigned long long>(P.tok[P.off[k]]) << 32) | static_cast<unsigned int>(P.r[k]);
            best = cand < best ? cand : best;
        }
    }
    return best;
}

__device__ __forceinline__ void write_row_outputs(const StepArgs& a, int row, float m, float s, unsigned long long pick) {
    int tok = -1, repv = -1;
    float lsev = -INFINITY, lpa = -INFINITY;
    if (pick != ~0ull) {
        tok = int(pick >> 32);
        repv = int(pick & 0xFFFFFFFFull);
        if (m > kRefFloor && s > 0.f) {
            const float l = logf(s);
            lsev = m + l;
            lpa = -l;
        }
    } else {
        atomicAdd(a.status + 0, 1);
    }
    a.argmax[row] = tok;
    if (a.rep) a.rep[row] = repv;
    if (a.lse) a.lse[row] = lsev;
    if (a.logp_argmax) a.logp_argmax[row] = lpa;
}

template <int DT>
__device__ __forceinline__ void warp_finalize_row(const StepArgs& a, const PartDev& P, int row, float m, float s,
                                                  int pos, int lane) {
    if (a.masks_per_row > 0 && s != s) {
        // the streaming kernel could not sum this mask beside the others (its logits lie too far below the row's largest)
        const char* rowp = reinterpret_cast<const char*>(a.logits) + logits_row(a, row) * a.row_stride * (DT == kBF16 ? 2 : 4);
        const uint32_t* cm = a.class_mask + int64_t(row) * a.cm_stride;
        s = 0.f;
        for (int t = lane; t < a.V; t += 32) {
            const int k = __ldg(P.c32 + t);
            if ((ld_after_wait(cm + (k >> 5)) >> (k & 31)) & 1u) s += ex2f((ldcg_elem<DT>(rowp, t) - m) * kLog2e);
        }
#pragma unroll
        for (int d = 16; d >= 1; d >>= 1) s += __shfl_xor_sync(0xFFFFFFFFu, s, d);
    }
    unsigned long long cand = ~0ull;
    if (pos == kNoPos) {
        cand = first_allowed_share(a, P, row, lane, 32);
    } else {
        // a position means that m is a finite allowed logit; the row is already masked in memory (disallowed
        // logits read -inf), so the first token of the octet that holds the value m is the choice. Its
        // representative is fetched side by side with the logit.
        // the position is the first octet of the 8 or 16 tokens its producer handled together: 16 lanes look
        const int t = 8 * pos + lane;
        if (lane < 16 && pos >= 0 && t < a.V) {
            const float z = ldcg_elem<DT>(reinterpret_cast<const char*>(a.logits) + logits_row(a, row) * a.row_stride * (DT == kBF16 ? 2 : 4), t);
            const int repv = __ldg(P.trep + t);
            bool ok = z == m;
            if (a.masks_per_row > 0) {  // the logits were left as they are: ask this row's class mask
                const int k = __ldg(P.c32 + t);
                ok = ok && ((ld_after_wait(a.class_mask + int64_t(row) * a.cm_stride + (k >> 5)) >> (k & 31)) & 1u);
            }
            if (ok) cand = (static_cast<unsigned long long>(t) << 32) | static_cast<unsigned int>(repv);
        }
    }
#pragma unroll
    for (int d = 16; d >= 1; d >>= 1) {
        const unsigned long long other = __shfl_xor_sync(0xFFFFFFFFu, cand, d);
        cand = other < cand ? other : cand;
    }
    if (lane == 0) write_row_outputs(a, row, m, s, cand);
}

// The octets past the last whole vector of a row (the ragged one when V is not a multiple of
// 8, and the padding octets up to the end of the last vocab-mask word): at most four per row.
// One warp takes them after the streaming loop, lane r = row slot r, token by token straight
// from the class-id vector and the row's class mask (compact code, run by one block per group).
template <int DT>
__device__ __forceinline__ Partial dense_tail_octets(const StepArgs& a, const PartDev& P, int row, int o_first, int o_end,
                                                     float scale) {
    constexpr int ES = DT == kBF16 ? 2 : 4;
    float m = -INFINITY, s = 0.f;
    int pos = kNoPos;
    if (row < 0) return Partial{m, s, pos, 0};
    const uint32_t* cm = a.class_mask + int64_t(row) * a.cm_stride;
    char* rowp = reinterpret_cast<char*>(a.logits) + logits_row(a, row) * a.row_stride * ES;
    uint8_t* vmp = a.vocab_mask ? reinterpret_cast<uint8_t*>(a.vocab_mask) + int64_t(row) * a.vm_stride * 4 : nullptr;
    for (int o = o_first; o < o_end; ++o) {
        uint32_t byte = 0;
        for (int j = 0; j < 8; ++j) {
            const int t = 8 * o + j;
            if (t >= a.V) break;
            const int k = P.c32[t];
            if ((cm[k >> 5] >> (k & 31)) & 1u) {
                byte |= 1u << j;
                const float z = load_elem<DT>(rowp, t);
                if (z > m) pos = o;
                const float ref_old = fmaxf(m, kRefFloor);
                m = fmaxf(m, z);
                const float ref = fmaxf(m, kRefFloor);
                s = fmaf(s, ex2f((ref_old - ref) * scale), ex2f((z - ref) * scale));
            } else if (a.masks_per_row == 0) {
                store_neg_inf<DT>(rowp, t);
            }
        }
        if (vmp) vmp[o] = uint8_t(byte);
    }
    return Partial{m, s, pos, 0};
}

// The blocks of a streaming launch that work on group g: a.S each, or, for a mixed batch with blocks enough, a.S_even each as
// long as the groups that turn up fit the launch at that number (two partitions of 24 rows: two groups, as 48 rows of one have),
// else in proportion to the groups' row batches, at least one (33 rows of one partition make a group of 32 and one of 1).
struct GroupShare {
    int first, S;
};
// (Functions of their own: a batch without a row plan, whose steps are the shortest, should not fetch past this code. Inlined in the
// per-row kernels it cost 256 rows that allow few tokens 1.8 of 27 us.)
__device__ __noinline__ GroupShare group_share(const StepArgs& a, int g) {
    const int n = ld_after_wait(a.n_groups), w0 = ld_after_wait(a.group_w + g), w1 = ld_after_wait(a.group_w + g + 1), W = ld_after_wait(a.group_w + a.max_groups);
    if (n * a.S_even <= a.blocks) return GroupShare{g * a.S_even, a.S_even};
    const int spare = a.blocks - n, first = g + spare * w0 / max(W, 1), next = g + 1 + spare * w1 / max(W, 1);
    return GroupShare{first, min(next - first, a.S)};
}
// The group of this block of such a launch (-1: none), its place among the group's blocks and their number. Called by one warp.
struct BlockPlace {
    int g, split, S;
};
__device__ __noinline__ BlockPlace block_place(const StepArgs& a) {
    const int b = blockIdx.x, n = ld_after_wait(a.n_groups), even = a.S_even;
    if (n * even <= a.blocks) {
        const int g = b / even;
        return BlockPlace{g < n ? g : -1, b - g * even, even};
    }
    const int lane = threadIdx.x & 31;
    for (int g0 = 0; g0 < n; g0 += 32) {
        const GroupShare s = g0 + lane < n ? group_share(a, g0 + lane) : GroupShare{0, 0};
        const uint32_t hit = __ballot_sync(0xFFFFFFFFu, b >= s.first && b < s.first + s.S);
        if (hit) {
            const int l = __ffs(int(hit)) - 1;
            return BlockPlace{g0 + l, b - __shfl_sync(0xFFFFFFFFu, s.first, l), __shfl_sync(0xFFFFFFFFu, s.S, l)};
        }
    }
    return BlockPlace{-1, 0, 0};
}
// Chunks in a run of a sampling step, as the warps of a group of such a batch dealt them.
__device__ __noinline__ int group_run_chunks(int n_octets, int chunk_octets, int warps) {
    return max(1, ((n_octets + chunk_octets - 1) / chunk_octets + warps - 1) / warps);
}
// States a row of group g has published.
__device__ __forceinline__ int group_states(const StepArgs& a, int g) {
    if (!a.group_w) return a.slots;
    const int S = group_share(a, g).S;
    return a.fold_off ? S : S * a.WT + 1 + a.head_state;
}

// Where the (max, sum-exp, position) states of a row go: every warp that streamed a row batch
// publishes one state per row in its own slot, slot = split * WT + wt, and the block that owns the
// end of the vocabulary adds the state of the octets past the last whole vector in the last
// slot. a.slots = S * WT + 1 states per row, rows of a group side by side.
__device__ __forceinline__ Partial* row_slots(const StepArgs& a, int g, int row_slot) {
    return a.partials + (int64_t(g) * kGroupRows + row_slot) * a.slots;
}

// After the streaming loop of a dense block: the warp that is told to (warp 0 of the block that
// owns the end of the vocabulary) handles the tail octets, lane r = row slot r.
template <int DT>
__device__ __forceinline__ void publish_tail_octets(const StepArgs& a, const PartDev& P, int g, const int* s_row, int lane,
                                                    int tail_first, int tail_end, float scale = kLog2e) {
    const Partial p = dense_tail_octets<DT>(a, P, s_row[lane], tail_first, tail_end, scale);
    if (s_row[lane] >= 0) row_slots(a, g, lane)[a.slots - 1] = p;
}
// Order-preserving map between floats and signed integers (for the integer warp reductions).
__device__ __forceinline__ int float_order_key(float x) {
    const int i = __float_as_int(x);
    return i >= 0 ? i : i ^ 0x7FFFFFFF;
}
__device__ __forceinline__ float float_from_order_key(int k) { return __int_as_float(k >= 0 ? k : k ^ 0x7FFFFFFF); }

// What the vectors of a row leave over: the tokens in front of the first vector (rows off the vector grid), those past
// the last one, and the vocab-mask octets from the last whole octet on (ragged end, padding of the last word). The
// rows of the group are dealt over its blocks and their warps, each warp takes its rows one at a time with a lane per
// token (lanes 0..7 the first octet, lanes 8..23 the 16 tokens from the last whole octet on), allow bits from the class
// table: two round trips to memory for a row, where one lane walking the tokens took two per token.
// to_head / to_tail(row slot): where the states go (the same place: one state for both). UNIT: tokens the vectors are taken in
// (8, or 16 for a kernel that takes them two at a time; rows on the vector grid only).
template <int DT, bool SHIFT, int UNIT = 8, typename H, typename T>
__device__ __forceinline__ void publish_edges(const StepArgs& a, const PartDev& P, const uint32_t* table, const int* s_row,
                                              int nrow, int split, int S, int warp, int lane, float scale, bool apart, H&& to_head,
                                              T&& to_tail) {
    constexpr int ES = DT == kBF16 ? 2 : 4;
    const int n_full = a.V >> 3, n_octets = 4 * a.VW;
    const bool in_head = lane < 8;
    const int t = in_head ? lane : 8 * (n_full - 1) + lane - 8;
    const bool have = lane < 24 && t >= 0 && t < a.V;
    const int n_warps = blockDim.x >> 5;
    if (!SHIFT && n_full == n_octets) {  // the vectors cover the vocabulary: nothing is left over
        for (int j = split + S * warp; j < nrow; j += S * n_warps)
            if (lane == 0) *to_tail(j) = partial_empty();
        return;
    }
    uint32_t word = 0u;
    bool asked = false;
    for (int j = split + S * warp; j < nrow; j += S * n_warps) {
        if (!asked && have) word = table[P.c16[t]];
        asked = true;
        const int row = s_row[j];
        char* rowp = reinterpret_cast<char*>(a.logits) + int64_t(row) * a.row_stride * ES;
        const int head = SHIFT ? row_head<DT>(rowp, a.V) : 0;
        const int tail = head + ((a.V - head) & ~(UNIT - 1));  // first token past the last whole vector
        const bool mine = have && (in_head ? t < head : t >= tail);
        const bool allowed = (word >> j) & 1u;
        const uint32_t allow = __ballot_sync(0xFFFFFFFFu, allowed && !in_head);
        const int first = UNIT == 8 ? n_full : n_full & ~1;  // first octet that is not all in whole vectors
        if (a.vocab_mask && lane < n_octets - first) {
            const int o = first + lane;
            reinterpret_cast<uint8_t*>(a.vocab_mask)[int64_t(row) * a.vm_stride * 4 + o] =
                o == n_full ? uint8_t(allow >> 16) : (o < n_full ? uint8_t(allow >> 8) : uint8_t(0));
        }
        float z = -INFINITY;
        if (mine) {
            if (allowed) z = load_elem<DT>(rowp, t);
            else store_neg_inf<DT>(rowp, t);
        }
        auto reduce = [&](bool part, int first) {  // the state of the lanes of one side; `first`: its octet position
            const float m = float_from_order_key(__reduce_max_sync(0xFFFFFFFFu, float_order_key(part ? z : -INFINITY)));
            float e = part && m > kRefFloor ? ex2f((z - m) * scale) : 0.f;
#pragma unroll
            for (int d = 16; d >= 1; d >>= 1) e += __shfl_xor_sync(0xFFFFFFFFu, e, d);
            return Partial{m, e, m > -INFINITY ? first : kNoPos, 0};
        };
        const Partial pt = reduce(mine && !in_head, UNIT == 8 ? (a.V - head) >> 3 : tail >> 3);
        if (!SHIFT) {
            if (lane == 0) *to_tail(j) = pt;
        } else {
            const Partial ph = reduce(mine && in_head, 0);
            if (lane == 0) {
                if (apart) {
                    *to_head(j) = ph;
                    *to_tail(j) = pt;
                } else {
                    float m = ph.m, sum = ph.s;
                    int pos = ph.pos;
                    partial_merge(m, sum, pos, pt.m, pt.s, pt.pos, scale);
                    *to_tail(j) = Partial{m, sum, pos, 0};
                }
            }
        }
    }
}

// ---------------------------------------------------------------------------------------
// Second kernel of a dense step: one block per (group, row slot). Folds the row's published
// states, finds the winning token among the 8 tokens of the winning octet (8 lanes side by side,
// each fetching its candidate's representative as well) and writes the row's results.
// ---------------------------------------------------------------------------------------
constexpr int kFinalizeThreads = 256;

template <int DT>
__global__ void __launch_bounds__(kFinalizeThreads) k_finalize_rows(const __grid_constant__ StepArgs a) {
    pdl_prologue();
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int g = blockIdx.x / kGroupRows, j = blockIdx.x - g * kGroupRows;
    // The states are asked for first, as many as a row can have: how many this one has, and whether there is a row, takes loads
    // in a chain where rows are grouped by a plan.
    const Partial* src = row_slots(a, g, j);
    int n_states = a.slots;
    auto fetch = [&](int base, int4 (&v)[4]) {
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int sp = base + u * kFinalizeThreads + tid;
            v[u] = make_int4(__float_as_int(-INFINITY), 0, kNoPos, 0);
            if (sp < n_states) v[u] = __ldcg(reinterpret_cast<const int4*>(src + sp));
        }
    };
    int4 v0[4];
    fetch(0, v0);
    if (a.group_w) {
        n_states = group_states(a, g);
#pragma unroll
        for (int u = 0; u < 4; ++u)
            if (u * kFinalizeThreads + tid >= n_states) v0[u] = make_int4(__float_as_int(-INFINITY), 0, kNoPos, 0);
    }
    if (a.n_groups && g >= ld_after_wait(a.n_groups)) return;
    int row;
    if (a.group_rows) {
        row = a.group_rows[g * kGroupRows + j];
    } else {
        row = g * kGroupRows + j;
        if (row >= a.B) row = -1;
    }
    if (row < 0) return;
    if (a.row_mode && a.row_mode[row]) return;  // automatic mode: the class-list kernel has finished this row
    const PartDev P = a.group_part ? a.parts[a.group_part[g]] : a.p0;
    // Two passes over the states, which stay in registers (up to four per thread, all loads in flight together):
    // first the row maximum (shuffles and max only), then every state's sum brought to that maximum with one
    // exponential per state, summed, and the lowest position among the states that hold the maximum. No
    // exponential sits inside a reduction chain, and the three reductions run side by side.
    constexpr int kWarps = kFinalizeThreads / 32;
    __shared__ float s_max[kWarps], s_sum[kWarps];
    __shared__ int s_pos[kWarps];
    float M = fmaxf(fmaxf(__int_as_float(v0[0].x), __int_as_float(v0[1].x)), fmaxf(__int_as_float(v0[2].x), __int_as_float(v0[3].x)));
    for (int base = 4 * kFinalizeThreads; base < n_states; base += 4 * kFinalizeThreads) {  // more than 1024 states: rare
        int4 w[4];
        fetch(base, w);
        M = fmaxf(M, fmaxf(fmaxf(__int_as_float(w[0].x), __int_as_float(w[1].x)), fmaxf(__int_as_float(w[2].x), __int_as_float(w[3].x))));
    }
#pragma unroll
    for (int d = 16; d >= 1; d >>= 1) M = fmaxf(M, __shfl_xor_sync(0xFFFFFFFFu, M, d));
    if (lane == 0) s_max[warp] = M;
    __syncthreads();
#pragma unroll
    for (int w = 0; w < kWarps; ++w) M = fmaxf(M, s_max[w]);
    const float Mf = fmaxf(M, kRefFloor);
    float sum = 0.f;
    int pos = kNoPos;
    auto gather = [&](const int4 (&v)[4]) {
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const float m = __int_as_float(v[u].x);
            sum = fmaf(__int_as_float(v[u].y), ex2f((fmaxf(m, kRefFloor) - Mf) * kLog2e), sum);
            pos = (m == M) ? min(pos, v[u].z) : pos;
        }
    };
    gather(v0);
    for (int base = 4 * kFinalizeThreads; base < n_states; base += 4 * kFinalizeThreads) {
        int4 w[4];
        fetch(base, w);
        gather(w);
    }
#pragma unroll
    for (int d = 16; d >= 1; d >>= 1) {
        sum += __shfl_xor_sync(0xFFFFFFFFu, sum, d);
        pos = min(pos, __shfl_xor_sync(0xFFFFFFFFu, pos, d));
    }
    if (lane == 0) {
        s_sum[warp] = sum;
        s_pos[warp] = pos;
    }
    __syncthreads();
    if (warp != 0) return;
    sum = 0.f;
    pos = kNoPos;
#pragma unroll
    for (int w = 0; w < kWarps; ++w) {  // every lane of warp 0 takes the same eight values in the same order
        sum += s_sum[w];
        pos = min(pos, s_pos[w]);
    }
    warp_finalize_row<DT>(a, P, row, M, sum, pos, lane);
}

// The same for rows with few published states (at most 4 per lane: large batches, where a group is
// shared by few blocks): one warp per row, 8 rows per block, no block-level step at all.
constexpr int kFinalizeWarpStates = 128;

template <int DT>
__global__ void __launch_bounds__(256) k_finalize_rows_warp(const __grid_constant__ StepArgs a) {
    pdl_prologue();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int idx = blockIdx.x * 8 + warp;  // (group, row slot)
    const int g = idx / kGroupRows, j = idx - g * kGroupRows;
    const Partial* src = row_slots(a, g, j);  // (the states first, as above)
    int4 v[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        const int sp = u * 32 + lane;
        v[u] = make_int4(__float_as_int(-INFINITY), 0, kNoPos, 0);
        if (sp < a.slots) v[u] = __ldcg(reinterpret_cast<const int4*>(src + sp));
    }
    if (a.group_w) {
        const int n_states = group_states(a, g);
#pragma unroll
        for (int u = 0; u < 4; ++u)
            if (u * 32 + lane >= n_states) v[u] = make_int4(__float_as_int(-INFINITY), 0, kNoPos, 0);
    }
    if (a.n_groups && g >= ld_after_wait(a.n_groups)) return;
    int row;
    if (a.group_rows) {
        row = a.group_rows[g * kGroupRows + j];
    } else {
        row = g * kGroupRows + j;
        if (row >= a.B) row = -1;
    }
    if (row < 0) return;
    if (a.row_mode && a.row_mode[row]) return;  // automatic mode: the class-list kernel has finished this row
    const PartDev P = a.group_part ? a.parts[a.group_part[g]] : a.p0;
    float m0 = __int_as_float(v[0].x), s0 = __int_as_float(v[0].y), m1 = __int_as_float(v[1].x), s1 = __int_as_float(v[1].y);
    int p0 = v[0].z, p1 = v[1].z;
    partial_merge(m0, s0, p0, __int_as_float(v[2].x), __int_as_float(v[2].y), v[2].z);
    partial_merge(m1, s1, p1, __int_as_float(v[3].x), __int_as_float(v[3].y), v[3].z);
    partial_merge(m0, s0, p0, m1, s1, p1);
    partial_warp_allreduce(m0, s0, p0);
    warp_finalize_row<DT>(a, P, row, m0, s0, p0, lane);
}

// One whole-vector octet of one row: mask, write back, note the vocab-mask byte, fold into the
// row state.
template <int DT>
__device__ __forceinline__ void dense_octet_row(Octet<DT>& oc, char* rowp, uint8_t* vmp, int o, uint32_t byte,
                                                RowAcc& acc, bool wide, bool write_back = true) {
    float f[8];
    oc.mask(byte, f);
    if (write_back) oc.store(rowp, o, wide);
    if (vmp) vmp[o] = uint8_t(byte);
    acc.add_octet(f, o);
}

// Reduce the 8 row states of a warp over its 32 lanes and publish them in the warp's slot of each row.
// The state of row slot r goes to base[r * stride + slot] (global scratch, or the block's shared array).
__device__ __forceinline__ void warp_rows_publish_to(RowAcc (&acc)[kBatchRows], int live, int rb, int lane, float scale,
                                                     Partial* base, int stride, int slot) {
    // Two passes, no exponential inside a reduction chain: the maximum of every row over the lanes (one integer
    // warp reduction each), every lane's sum brought to it with one exponential, the lowest position among the
    // lanes that hold the maximum (one more integer reduction), and the eight sums reduced by recursive halving
    // (lanes trade half of their rows with the lane 16 away, then 2 of 4 with the lane 8 away, then 1 of 2; two
    // butterfly steps finish the single row left).
    float M[kBatchRows], w[kBatchRows];
    int pos[kBatchRows];
#pragma unroll
    for (int i = 0; i < kBatchRows; ++i) M[i] = float_from_order_key(__reduce_max_sync(0xFFFFFFFFu, float_order_key(acc[i].m)));
#pragma unroll
    for (int i = 0; i < kBatchRows; ++i) {
        // (the comparison is not needed, the sum is empty there; without it the streaming kernel spills: 1024 bf16 rows 108.2 -> 112.5 us)
        w[i] = M[i] > kRefFloor ? acc[i].sum_below(M[i], scale) : 0.f;
        pos[i] = __reduce_min_sync(0xFFFFFFFFu, acc[i].m == M[i] ? acc[i].pos : kNoPos);
    }
#pragma unroll
    for (int half = 4; half >= 1; half >>= 1) {
        const int d = 4 * half;  // 16, 8, 4
        const bool up = lane & d;
#pragma unroll
        for (int k = 0; k < half; ++k) {
            const float keep = up ? w[k + half] : w[k];
            const float send = up ? w[k] : w[k + half];
            w[k] = keep + __shfl_xor_sync(0xFFFFFFFFu, send, d);
        }
    }
    w[0] += __shfl_xor_sync(0xFFFFFFFFu, w[0], 2);
    w[0] += __shfl_xor_sync(0xFFFFFFFFu, w[0], 1);
    const int i = ((lane >> 4) & 1) * 4 + ((lane >> 3) & 1) * 2 + ((lane >> 2) & 1);  // the row this lane ended with
    float Mi = M[0];
    int pi = pos[0];
#pragma unroll
    for (int k = 1; k < kBatchRows; ++k) {
        Mi = i == k ? M[k] : Mi;
        pi = i == k ? pos[k] : pi;
    }
    if ((lane & 3) == 0 && i < live) base[(rb * kBatchRows + i) * stride + slot] = Partial{Mi, w[0], pi, 0};
}
__device__ __forceinline__ void warp_rows_publish(const StepArgs& a, RowAcc (&acc)[kBatchRows], int live, int g, int slot,
                                                  int rb, int lane, float scale = kLog2e) {
    warp_rows_publish_to(acc, live, rb, lane, scale, row_slots(a, g, 0), a.slots, slot);
}

// Fold up to `n` states (16 bytes each, read through L2) with the lanes of a warp side by side; every lane returns
// the merged state. Four loads per lane are in flight together.
__device__ __forceinline__ void warp_fold_states(const Partial* src, int n, int lane, float& m, float& s, int& pos) {
    m = -INFINITY;
    s = 0.f;
    pos = kNoPos;
    for (int base = 0; base < n; base += 128) {
        int4 v[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int sp = base + u * 32 + lane;
            v[u] = make_int4(__float_as_int(-INFINITY), 0, kNoPos, 0);
            if (sp < n) v[u] = __ldcg(reinterpret_cast<const int4*>(src + sp));
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) partial_merge(m, s, pos, __int_as_float(v[u].x), __int_as_float(v[u].y), v[u].z);
    }
    partial_warp_allreduce(m, s, pos);
}

// ---------------------------------------------------------------------------------------
// Fused dense step, register version: expand + mask in place + (max, sum-exp, position) per
// row, logits fetched with 16-byte loads straight into registers (rows 16-byte aligned).
// Grid: n_groups * S thread blocks; block (g, split) owns octets [split*per_split, ...) of the
// 32 rows of group g. Warps are arranged WT (along tokens) x WR (row batches of 8).
// ---------------------------------------------------------------------------------------
template <int DT>
__global__ void __launch_bounds__(256) k_step_dense(const __grid_constant__ StepArgs a) {
    extern __shared__ __align__(128) uint32_t smem[];
    uint32_t* T = smem;
    int* s_row = reinterpret_cast<int*>(T + a.table_words);
    uint32_t* stage = reinterpret_cast<uint32_t*>(s_row + kGroupRows);

    pdl_prologue();
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, n_warps = blockDim.x >> 5;
    const int g = blockIdx.x / a.S, split = blockIdx.x - g * a.S;
    if (a.n_groups && g >= ld_after_wait(a.n_groups)) return;
    const int part = group_rows_setup(a, g, s_row, tid);
    __syncthreads();
    const PartDev P = a.group_part ? a.parts[part] : a.p0;
    const int nrow = __popc(__ballot_sync(0xFFFFFFFFu, s_row[lane] >= 0));
    if (a.cm_bulk || a.stage_stride >= min(P.KW, kMaskSlice)) make_class_table(a, P, s_row, T, stage, warp, lane, n_warps);
    else build_class_table_narrow_call(a, P.K, P.KW, smem_u32(s_row), smem_u32(T), smem_u32(stage));
    __syncthreads();

    const int wt = warp % a.WT, wr = warp / a.WT, WR = n_warps / a.WT;
    const int n_octets = 4 * a.VW, n_full = a.V >> 3;
    const int o_begin = split * a.per_split;
    const int o_end = min(o_begin + a.per_split, n_octets);
    const int o_vec_end = min(o_end, n_full);
    constexpr int ES = DT == kBF16 ? 2 : 4;
    uint8_t* vm8 = reinterpret_cast<uint8_t*>(a.vocab_mask);

    for (int rb = wr; rb * kBatchRows < nrow; rb += WR) {
        RowAcc acc[kBatchRows];
        char* rowp[kBatchRows];
        uint8_t* vmp[kBatchRows];
#pragma unroll
        for (int i = 0; i < kBatchRows; ++i) {
            acc[i].init();
            const int row = s_row[min(rb * kBatchRows + i, kGroupRows - 1)];
            rowp[i] = reinterpret_cast<char*>(a.logits) + logits_row(a, max(row, 0)) * a.row_stride * ES;
            vmp[i] = vm8 ? vm8 + int64_t(max(row, 0)) * a.vm_stride * 4 : nullptr;
        }
        const int live = min(kBatchRows, nrow - rb * kBatchRows);

        for (int o0 = o_begin + wt * 32; o0 < o_vec_end; o0 += a.WT * 32) {
            const int o = o0 + lane;
            const bool active = o < o_vec_end;
            Octet<DT> oc[kBatchRows];
#pragma unroll
            for (int i = 0; i < kBatchRows; ++i)
                if (i < live && active) oc[i].load(rowp[i], o);
            uint32_t lo, hi;
            uint4 cv = make_uint4(0, 0, 0, 0);
            if (active) cv = __ldg(reinterpret_cast<const uint4*>(P.c16) + o);
            octet_allow_bits(cv, T, rb, active, lo, hi);
#pragma unroll
            for (int i = 0; i < kBatchRows; ++i) {
                if (i < live && active) {
                    const uint32_t byte = ((i < 4 ? lo : hi) >> (8 * (i & 3))) & 0xFFu;
                    dense_octet_row<DT>(oc[i], rowp[i], vmp[i], o, byte, acc[i], a.wide != 0, a.masks_per_row == 0);
                }
            }
        }
        warp_rows_publish(a, acc, live, g, split * a.WT + wt, rb, lane);
    }
    // the block that reaches the end of the vocabulary takes the octets past the last whole vector
    if (warp == 0 && o_end == n_octets) publish_tail_octets<DT>(a, P, g, s_row, lane, max(o_begin, n_full), o_end);
}

// ---------------------------------------------------------------------------------------
// Fused dense step, pipelined version. Same decomposition as above, but the logits reach the
// SM through bulk asynchronous copies: every warp runs its own ring of `depth` stages in
// shared memory, each stage holding 32 octets of 8 rows plus the 32 octets of class ids,
// filled by copies that lane 0 issues `depth` work items ahead and that signal an mbarrier.
// The first copies are started before the class table is built. The lanes read their 16
// bytes per row from shared memory, so no registers wait on memory and the copies of later
// items overlap the arithmetic of this one. Masked logits go back with 16-byte stores.
// ---------------------------------------------------------------------------------------
// OPL: octets a lane handles per row of an item (1, or 2 for bf16: 32 bytes per lane and row either way for OPL = 2
// and for f32). A chunk is the 32 * OPL octets the lanes of a warp cover together.
template <int DT, int OPL>
struct PipeGeom {
    static constexpr int kOctetBytes = DT == kBF16 ? 16 : 32;
    static constexpr int kBoxBytes = kBatchRows * 32 * kOctetBytes;        // one tiled copy: 8 rows of 32 octets
    static constexpr int kRowBytes = 32 * OPL * kOctetBytes;               // one row of a stage
    static constexpr int kChunkOctets = 32 * OPL;
    static constexpr int kStageBytes = kBatchRows * kRowBytes + kChunkOctets * 16;  // + class ids of the chunk
};

// How the logits of a work item reach shared memory: one bulk copy per row, one tiled 2-D copy for 8 consecutive rows,
// or one bulk copy per row from that row's own first vector boundary on (rows that start anywhere).
enum : int { kSrcRows = 0, kSrcTiled = 1, kSrcShifted = 2 };
enum : int { kStepGreedy = 0, kStepSample = 1, kStepFiltered = 2 };

// Octets of a chunk. Where the rows start anywhere, vector o of a row holds the tokens 8 o + head .. 8 o + head + 7, so
// its allow bits come from the token octets o and o + 1: a chunk is then the 31 vectors whose bits the 32 octets of
// class ids in a stage give (lane l takes the second half of its bits from lane l + 1).
template <int OPL, int SRC>
struct PipeChunk {
    static constexpr int kOctets = SRC == kSrcShifted ? 31 : 32 * OPL;
};

// Where the rows of a batch live. With consecutive rows (CONSEC) the address of row i is one
// wide multiply-add from the batch's base; otherwise each row has its own base pointer.
struct BatchAddr {
    char* item_base;      // CONSEC: logits of row 0 of the batch at this lane's octet
    uint8_t* vm_item;     // CONSEC: vocab-mask byte of row 0 at this lane's octet (or null)
    uint32_t row_bytes;   // CONSEC: bytes between rows of the logits
    uint32_t vm_bytes;    // CONSEC: bytes between rows of the vocab mask
};

// One work item of a warp: the 32 * OPL octets of a chunk for the 8 rows of a batch, read from the stage `src`;
// this lane's OPL octets of row i lie at src + i * srow + lane_off. n_act: how many of the lane's octets are whole
// vectors of the row (OPL everywhere except at the end of the vocabulary).
// FULL: all 8 rows live and every lane's octets inside the whole-vector range (no per-row tests).
// kSrcShifted: n_ids octets of class ids are in the stage; heads: row_head of the 8 rows, four bits each; the vocab-mask
// byte of token octet o is written by the same lane as vector o of the rows. V: tokens.
// MAXIMA: chunk_m of lane i becomes the largest masked logit of the chunk in row i.
template <int DT, int OPL, bool FULL, int SRC, bool MAXIMA>
__device__ __forceinline__ void pipe_consume_item(const char* src, uint32_t lane_off, uint32_t srow, const uint32_t* T, int rb,
                                                  int live, int n_act, int o, int lane, const BatchAddr& ba,
                                                  char* const (&rowp)[kBatchRows], uint8_t* const (&vmp)[kBatchRows],
                                                  RowAcc (&acc)[kBatchRows], float scale, bool wide, int n_ids, uint32_t heads,
                                                  int V, float& chunk_m) {
    using G = PipeGeom<DT, OPL>;
    constexpr bool CONSEC = SRC == kSrcTiled;
    if constexpr (SRC == kSrcShifted) {
        uint32_t lo, hi;
        uint4 cv = make_uint4(0, 0, 0, 0);
        const bool have = FULL || lane < n_ids;
        if (have) cv = *reinterpret_cast<const uint4*>(src + kBatchRows * G::kRowBytes + lane * 16);
        octet_allow_bits(cv, T, rb, have, lo, hi);
        const uint32_t lo2 = __shfl_down_sync(0xFFFFFFFFu, lo, 1), hi2 = __shfl_down_sync(0xFFFFFFFFu, hi, 1);
        if (lane == 31) return;  // its bits served lane 30
#pragma unroll
        for (int i = 0; i < kBatchRows; ++i) {
            float top = -INFINITY;
            if (FULL || i < live) {
                const uint32_t byte = ((i < 4 ? lo : hi) >> (8 * (i & 3))) & 0xFFu;
                if (vmp[i] && (FULL || 8 * o + 8 <= V)) st_global_u8(vmp[i] + o, byte);
                const int head = int((heads >> (4 * i)) & 15u);
                if (FULL || 8 * o + head + 8 <= V) {
                    const uint32_t next = ((i < 4 ? lo2 : hi2) >> (8 * (i & 3))) & 0xFFu;
                    Octet<DT> oc;
                    float f[8];
                    oc.load_shared_at(src + i * G::kRowBytes + lane_off);
                    oc.mask(((byte | (next << 8)) >> head) & 0xFFu, f);
                    oc.store_at(rowp[i] + size_t(o) * G::kOctetBytes, true);  // f32 vectors sit on 32-byte boundaries here
                    top = acc[i].add_octet(f, o, scale);
                }
            }
            if constexpr (MAXIMA) {
                top = redux_max(top, 0x7FFFFFFFu);
                chunk_m = lane == i ? top : chunk_m;
            }
        }
    } else {
        uint32_t lo[OPL], hi[OPL];
#pragma unroll
        for (int q = 0; q < OPL; ++q) {
            const bool act = FULL || q < n_act;
            uint4 cv = make_uint4(0, 0, 0, 0);
            if (act) cv = *reinterpret_cast<const uint4*>(src + kBatchRows * G::kRowBytes + (lane * OPL + q) * 16);
            octet_allow_bits(cv, T, rb, act, lo[q], hi[q]);
        }
        const bool both = FULL || n_act == OPL;
#pragma unroll
        for (int i = 0; i < kBatchRows; ++i) {
            float top = -INFINITY;
            if (FULL || (i < live && n_act > 0)) {
                Octet<DT> oc[OPL];
                float f[8 * OPL];
                uint32_t bytes = 0;
#pragma unroll
                for (int q = 0; q < OPL; ++q) {
                    const uint32_t byte = ((i < 4 ? lo[q] : hi[q]) >> (8 * (i & 3))) & 0xFFu;  // 0 for an octet past the range
                    if (FULL || q < n_act)
                        oc[q].load_shared_at(src + i * srow + lane_off + q * G::kOctetBytes);
                    else
                        oc[q].fill_neg_inf();
                    oc[q].mask(byte, f + 8 * q);
                    bytes |= byte << (8 * q);
                }
                char* zp = CONSEC ? ptr_mad(ba.item_base, i, ba.row_bytes) : rowp[i] + size_t(o) * G::kOctetBytes;
                char* vp = CONSEC ? (ba.vm_item ? ptr_mad(reinterpret_cast<char*>(ba.vm_item), i, ba.vm_bytes) : nullptr)
                                  : (vmp[i] ? reinterpret_cast<char*>(vmp[i]) + o : nullptr);
                if (OPL == 1) {
                    oc[0].store_at(zp, wide);
                    if (vp) st_global_u8(vp, bytes);
                } else {
                    if (both && wide) {
                        st_stream32(zp, oc[0].raw(), oc[OPL - 1].raw());
                    } else {
                        oc[0].store_at(zp);
                        if (both) oc[OPL - 1].store_at(zp + G::kOctetBytes);
                    }
                    if (vp) {
                        if (both) st_global_u16(vp, bytes); else st_global_u8(vp, bytes & 0xFFu);
                    }
                }
                top = acc[i].template add_values<8 * OPL>(f, o, scale);
            }
            if constexpr (MAXIMA) {
                top = redux_max(top);
                chunk_m = lane == i ? top : chunk_m;
            }
        }
    }
}

// SRC: kSrcTiled: the 8 rows of a batch are consecutive rows of the logits matrix and arrive as tiled 2-D copies
// through `tmap` (box = 256 elements x 8 rows: one per chunk, two for a chunk of 512 bf16 tokens);
// otherwise one bulk copy per row. kSrcShifted: rows that start anywhere (an odd vocabulary packed end to end); their
// vectors start row_head tokens in, the tokens left over on both sides go through publish_edges. (One token per thread
// and one block per row took 223 us for 48 rows of 100003 bf16 logits.) OPL: octets per lane and row (see PipeGeom).
// LBT / MINB: launch bounds (threads per block, blocks per SM) the variant is compiled for; they set
// the register budget: (512, 1) 128 registers, (384, 1) 168, (320, 2) 96, (256, 3) 80.
// KIND: a greedy step (T = 1 is compiled in), or a sampling step, whose sums are of exp(z / T): kStepSample deals the chunks so that
// the states of a row follow the token order, kStepFiltered (top-k / top-p follow) deals them as a greedy step does and leaves the
// largest logit of every chunk of a row in chunk_max.
template <int DT, int OPL, int SRC, int LBT, int MINB, int KIND>
__global__ void __launch_bounds__(LBT, MINB) k_step_dense_pipe(const __grid_constant__ StepArgs a,
                                                         const __grid_constant__ CUtensorMap tmap) {
    using G = PipeGeom<DT, OPL>;
    constexpr bool TEMPERED = KIND != kStepGreedy, RUNS = KIND == kStepSample, MAXIMA = KIND == kStepFiltered;
    constexpr bool TMAP = SRC == kSrcTiled, SHIFT = SRC == kSrcShifted;
    constexpr int kChunkOctets = PipeChunk<OPL, SRC>::kOctets;
    __shared__ char* s_vec[SHIFT ? kGroupRows : 1];  // first vector of every row of the group
    __shared__ int s_nvec[SHIFT ? kGroupRows : 1];   // and the number of its whole vectors
    extern __shared__ __align__(128) uint32_t smem[];
    uint32_t* T = smem;
    int* s_row = reinterpret_cast<int*>(T + a.table_words);
    const int n_warps = blockDim.x >> 5;
    uint64_t* bars = reinterpret_cast<uint64_t*>(s_row + kGroupRows);  // n_warps * depth
    int* ring_info = reinterpret_cast<int*>(bars + n_warps * a.depth);         // n_warps * depth
    char* ring = reinterpret_cast<char*>(bars) + ((n_warps * a.depth * 12 + 127) & ~127);  // keeps 128-byte alignment
    // The staging area of the class masks is dead once the table is built. Where shared memory is short it
    // shares the space of the first warps' rings; those warps then start their copies after the table.
    uint32_t* stage = a.stage_alias ? reinterpret_cast<uint32_t*>(ring)
                                    : reinterpret_cast<uint32_t*>(ring + size_t(n_warps) * a.depth * G::kStageBytes);
    __shared__ uint64_t cm_bar;

    // Without a row plan nothing of the set-up reads memory (the rows of the group are g*32 .. g*32+31, its
    // partition is part0): it runs while the kernel in front is still finishing, and the wait for that kernel
    // comes just before the first copies. With a row plan the wait comes first, as the plan is read at once.
    pdl_launch_dependents();
    const bool implicit = !a.group_rows;
    if (!implicit) pdl_wait();
    const float scale = TEMPERED ? a.scale : kLog2e;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    int g, split, S;
    if (TMAP || !a.group_w) {  // (tiled copies: no row plan)
        g = blockIdx.x / a.S;
        split = blockIdx.x - g * a.S;
        S = a.S;
        if (!TMAP && a.n_groups && g >= ld_after_wait(a.n_groups)) return;
    } else {  // (one warp looks: sixteen of every block after the same few words wait for one another)
        __shared__ BlockPlace s_place;
        if (warp == 0) {
            const BlockPlace place = block_place(a);
            if (lane == 0) s_place = place;
        }
        __syncthreads();
        g = s_place.g;
        split = s_place.split;
        S = s_place.S;
        if (g < 0) return;
    }
    const bool early_cm = a.cm_bulk && implicit;
    if (early_cm && tid == 0) {
        mbar_init(&cm_bar, 1);
        mbar_init_fence();
        mbar_expect_tx(&cm_bar, a.cm_bulk == kMasksBlock ? mask_block_bytes(a, g) : uint32_t(min(kGroupRows, a.B - g * kGroupRows)) * uint32_t(a.p0.KW) * 4u);
        if (TMAP) asm volatile("prefetch.tensormap [%0];" ::"l"(&tmap) : "memory");
    }
    const int part = group_rows_setup(a, g, s_row, tid);
    if (SHIFT && tid < kGroupRows) {  // (the threads that have just set s_row)
        char* rowp = reinterpret_cast<char*>(a.logits) + int64_t(max(s_row[tid], 0)) * a.row_stride * (DT == kBF16 ? 2 : 4);
        const int head = row_head<DT>(rowp, a.V);
        s_vec[tid] = rowp + head * (DT == kBF16 ? 2 : 4);
        s_nvec[tid] = (a.V - head) >> 3;
    }
    __syncthreads();
    const PartDev P = a.group_part ? a.parts[part] : a.p0;
    const int nrow = __popc(__ballot_sync(0xFFFFFFFFu, s_row[lane] >= 0));

    const int depth = a.depth;
    const int wt = warp % a.WT, wr = warp / a.WT, WR = n_warps / a.WT;
    const int n_octets = 4 * a.VW, n_full = a.V >> 3;
    constexpr int ES = DT == kBF16 ? 2 : 4;
    uint8_t* vm8 = reinterpret_cast<uint8_t*>(a.vocab_mask);
    char* my_ring = ring + size_t(warp) * depth * G::kStageBytes;
    uint64_t* bar = bars + warp * depth;

    // Work items: (row batch, chunk of 32 whole-vector octets). A warp owns the row batches rb = wr,
    // wr+WR, ...; the chunks of a row batch are dealt round-robin to the warps of the group that own it
    // (warp index among them, then a stride of their number), so that at any moment the group's blocks
    // read neighbouring pieces of the same rows: measured 5 % faster on long steps than one contiguous
    // range per block, and as fast as handing chunks out through global counters.
    // In a sampling step without filters (RUNS) the states of a row must follow the token order: every warp slot then
    // takes one contiguous run of run_chunks chunks instead.
    // The number of chunks is rarely a multiple of the number of warp slots, so some slots get one chunk more than
    // the others; the deal starts at a different slot for every row batch (rot_chunks further on), which spreads the
    // extra chunks evenly over the warps and the blocks instead of giving the first ones one more in every row batch.
    const int n_chunks = (n_full + kChunkOctets - 1) / kChunkOctets;
    const int stride_chunks = RUNS ? 1 : S * a.WT;  // round-robin: warps that share a row batch of the group
    const int run_chunks = RUNS ? (!TMAP && a.group_w ? max(1, (n_chunks + S * a.WT - 1) / (S * a.WT)) : a.run_chunks) : 0;
    const int n_slots = !TMAP && a.group_w ? (a.fold_off ? S : S * a.WT + 1 + a.head_state) : a.slots;  // states of a row, the last one for its ends
    auto first_chunk_of = [&](int rb) {  // this warp's first chunk of row batch rb
        if (RUNS) return (split * a.WT + wt) * run_chunks;
        int c = split * a.WT + wt - rb * a.rot_chunks;
        c %= stride_chunks;
        return c < 0 ? c + stride_chunks : c;
    };
    const int chunk_end = RUNS ? min(first_chunk_of(0) + run_chunks, n_chunks) : n_chunks;
    int* const slot_info = ring_info + warp * depth; // (rb << 24) | chunk of the item in each slot, -1 = no more items

    // automatic mode: bit r = row slot r was finished by the class-list kernel (set after the wait below)
    uint32_t rows_done = 0u;
    auto batch_done = [&](int rb) {
        const int n = min(kBatchRows, nrow - rb * kBatchRows);
        const uint32_t all = n >= 8 ? 0xFFu : (1u << n) - 1u;
        return ((rows_done >> (rb * kBatchRows)) & 0xFFu) == all;
    };
    // Producer cursor: one lane issues the copies of an item when it is a tiled copy; a copy per row is issued side by side, a
    // lane each, and the whole warp keeps the cursor (256 rows over eight partitions, V = 256000: 65 -> 61 us; 48 rows off the vector grid 13.5 -> 12.8).
    constexpr bool COOP = !TMAP;
    int p_rb = wr, p_slot = 0, p_issued = 0, p_chunk = 0;
    bool p_first = true, p_done = wr * kBatchRows >= nrow, p_end = false;
    auto issue_next = [&]() {
        int chunk = -1;
        while (!p_done) {
            if (p_first && rows_done && batch_done(p_rb)) {  // nothing left to do for this row batch
                p_rb += WR;
                p_done = p_rb * kBatchRows >= nrow;
                continue;
            }
            if (p_first) {
                chunk = first_chunk_of(p_rb);
                p_first = false;
            } else {
                chunk = p_chunk + stride_chunks;
            }
            p_chunk = chunk;
            if (chunk < chunk_end) break;
            chunk = -1;  // this row batch is handed out completely: on to the warp's next one
            p_rb += WR;
            p_first = true;
            p_done = p_rb * kBatchRows >= nrow;
        }
        if (chunk < 0) {
            if (!COOP || lane == 0) slot_info[p_slot] = -1;
            p_end = true;
            return;
        }
        if (!COOP || lane == 0) slot_info[p_slot] = (p_rb << 24) | chunk;
        const int o0 = chunk * kChunkOctets;
        char* dst = my_ring + size_t(p_slot) * G::kStageBytes;
        const uint32_t nvec = uint32_t(min(n_full - o0, kChunkOctets));  // >= 1: chunk < n_chunks
        uint32_t n_ids = nvec;
        if (SHIFT) {
            n_ids = uint32_t(min(n_octets - o0, 32));  // one octet more than vectors (the class ids are padded to n_octets)
            const int live = min(kBatchRows, nrow - p_rb * kBatchRows);
            uint32_t bytes = 0u;
            if (lane < live) bytes = uint32_t(max(0, min(s_nvec[p_rb * kBatchRows + lane] - o0, kChunkOctets))) * G::kOctetBytes;
            const uint32_t total = __reduce_add_sync(0xFFFFFFFFu, bytes);
            if (lane == 0) mbar_expect_tx(bar + p_slot, total + n_ids * 16u);
            __syncwarp();
            if (bytes)
                bulk_g2s(dst + lane * G::kRowBytes, s_vec[p_rb * kBatchRows + lane] + size_t(o0) * G::kOctetBytes, bytes, bar + p_slot);
        } else if (TMAP) {
            // a box holds 32 octets of the 8 rows; the second box of a two-octet chunk is fetched only if the chunk
            // reaches into it (its lanes are idle otherwise); parts of a box past V or past the last row are filled in
            const int nbox = (OPL == 2 && nvec > 32u) ? 2 : 1;
            mbar_expect_tx(bar + p_slot, uint32_t(nbox * G::kBoxBytes) + nvec * 16u);
            tma_g2s_2d(dst, &tmap, o0 * 8, s_row[p_rb * kBatchRows], bar + p_slot);
            if (nbox == 2) tma_g2s_2d(dst + G::kBoxBytes, &tmap, o0 * 8 + 256, s_row[p_rb * kBatchRows], bar + p_slot);
        } else {
            const int live = min(kBatchRows, nrow - p_rb * kBatchRows);
            const uint32_t row_bytes = nvec * G::kOctetBytes;
            if (lane == 0) mbar_expect_tx(bar + p_slot, uint32_t(live) * row_bytes + nvec * 16u);
            __syncwarp();
            if (lane < live)
                bulk_g2s(dst + lane * G::kRowBytes,
                         reinterpret_cast<const char*>(a.logits) +
                             (int64_t(s_row[p_rb * kBatchRows + lane]) * a.row_stride * ES + int64_t(o0) * 8 * ES),
                         row_bytes, bar + p_slot);
        }
        if (!COOP || lane == kBatchRows)
            bulk_g2s(dst + kBatchRows * G::kRowBytes, reinterpret_cast<const char*>(P.c16) + size_t(o0) * 16, n_ids * 16u, bar + p_slot);
        ++p_issued;
        if (++p_slot == depth) p_slot = 0;
    };

    if (lane == 0) {
        for (int d = 0; d < depth; ++d) mbar_init(bar + d, 1);
        if (warp == 0 && !early_cm) mbar_init(&cm_bar, 1);
        mbar_init_fence();
    }
    if (implicit && a.prefetch_items > 0 && lane == 0 && !p_done) {
        // While the kernel in front is finishing, DRAM has little to do: ask this warp's first work items (and the
        // group's class masks) into the L2. These are hints only: they deliver nothing, and whatever the kernel in
        // front may still write reaches the same L2, so nothing stale can be read after the wait.
        const int row0 = g * kGroupRows + wr * kBatchRows;
        const int live0 = min(kBatchRows, nrow - wr * kBatchRows);
        int chunk = first_chunk_of(wr);
        for (int d = 0; d < a.prefetch_items && chunk < chunk_end; ++d, chunk += stride_chunks) {
            const int o0 = chunk * kChunkOctets;
            const uint32_t nvec = uint32_t(min(n_full - o0, kChunkOctets));
            if (SHIFT) {
                for (int i = 0; i < live0; ++i) {
                    const int n = min(s_nvec[wr * kBatchRows + i] - o0, kChunkOctets);
                    if (n > 0) bulk_prefetch(s_vec[wr * kBatchRows + i] + size_t(o0) * G::kOctetBytes, uint32_t(n) * G::kOctetBytes);
                }
            } else if (TMAP) {
                tma_prefetch_2d(&tmap, o0 * 8, row0);
                if (OPL == 2 && nvec > 32u) tma_prefetch_2d(&tmap, o0 * 8 + 256, row0);
            } else {
                for (int i = 0; i < live0; ++i)
                    bulk_prefetch(reinterpret_cast<const char*>(a.logits) + (int64_t(row0 + i) * a.row_stride * ES + int64_t(o0) * 8 * ES),
                                  nvec * G::kOctetBytes);
            }
        }
        if (warp == 0 && a.cm_bulk == kMasksBlock)
            bulk_prefetch(a.class_mask + int64_t(g * kGroupRows) * a.cm_stride, mask_block_bytes(a, g));
        else if (warp == 0 && a.cm_bulk)
            for (int r = 0; r < nrow; ++r)
                bulk_prefetch(a.class_mask + int64_t(g * kGroupRows + r) * a.cm_stride, uint32_t(a.p0.KW) * 4u);
    }
    if (implicit) pdl_wait();
    // automatic mode: row batches that allow few tokens were finished by the class-list kernel in front and get no
    // work items here (that kernel decides for the 8 row slots of a batch together).
    if (a.row_mode) {
        rows_done = __ballot_sync(0xFFFFFFFFu, s_row[lane] >= 0 && a.row_mode[s_row[lane]] != 0);
        if (rows_done == __ballot_sync(0xFFFFFFFFu, s_row[lane] >= 0)) return;  // the whole group is done
    }
    if (early_cm) {
        // the class masks first (everything waits for them): the rows dealt over the warps, so that no warp
        // issues more than a few copies; the barrier was set up by thread 0 before the block met above
        const int r = warp + n_warps * lane;
        if (a.cm_bulk == kMasksBlock) {
            const char* const src = reinterpret_cast<const char*>(a.class_mask + int64_t(g * kGroupRows) * a.cm_stride);
            const uint32_t bytes = mask_block_bytes(a, g);
            for (uint32_t at = uint32_t(r) * kMaskPiece; at < bytes; at += 32u * uint32_t(n_warps) * kMaskPiece)  // (once, but for blocks of one or two warps)
                bulk_g2s(reinterpret_cast<char*>(stage) + at, src + at, min(bytes - at, kMaskPiece), &cm_bar);
        } else if (r < kGroupRows && g * kGroupRows + r < a.B)
            bulk_g2s(stage + r * a.stage_stride, a.class_mask + int64_t(g * kGroupRows + r) * a.cm_stride, uint32_t(a.p0.KW) * 4u,
                     &cm_bar);
    }
    if (a.cm_bulk && !early_cm) {
        __syncthreads();  // the class-mask barrier is initialised for everybody
        if (warp == 0) {
            // one bulk copy per row of the group, issued side by side by the lanes of one warp
            if (lane == 0) mbar_expect_tx(&cm_bar, uint32_t(nrow) * uint32_t(P.KW) * 4u);
            __syncwarp();
            const int row = s_row[lane];
            if (row >= 0)
                bulk_g2s(stage + lane * a.stage_stride, a.class_mask + int64_t(row) * a.cm_stride, uint32_t(P.KW) * 4u, &cm_bar);
        }
    }
    if ((COOP || lane == 0) && warp >= a.hold_warps)  // hold_warps is 0 unless the staging area lies over the rings
        for (int d = 0; d < depth && !p_end; ++d) issue_next();  // in flight while the table is built
    bool failed = false;
    if (a.cm_bulk) {
        if (!mbar_wait(&cm_bar, 0)) failed = true;
        if (a.cm_bulk == kMasksBlock)
            build_class_table<true>(a, P.K, P.KW, s_row, T, stage, warp, lane, n_warps, 0, P.KW + 1, int(mask_block_bytes(a, g) / 4u));
        else
            build_class_table_quads(a, P, s_row, T, stage, warp, lane, n_warps);
    } else {
        build_class_table_staged_call(a, P.K, P.KW, smem_u32(s_row), smem_u32(T), smem_u32(stage));
    }
    __syncthreads();
    if (__any_sync(0xFFFFFFFFu, failed) && lane == 0) atomicAdd(a.status + 3, 1);  // class masks never arrived
    failed = false;
    if ((COOP || lane == 0) && warp < a.hold_warps) {
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // the staging area was read and written by plain accesses
        for (int d = 0; d < depth && !p_end; ++d) issue_next();
    }

    int slot = 0;
    uint32_t phase = 0;
    int consumed = 0;
    // Where this warp's row states go: its own slot of the global scratch, or (fold with block-level merge) the
    // block's shared array of (row slot, warp along tokens) states
    const bool fold = !TEMPERED && a.fold != 0;
    Partial* const s_state = (!TEMPERED && a.fold_off) ? reinterpret_cast<Partial*>(reinterpret_cast<char*>(smem) + a.fold_off) : nullptr;
    Partial* const pub_base = s_state ? s_state : row_slots(a, g, 0);
    const int pub_stride = s_state ? a.WT + 1 : a.slots;
    const int my_slot = s_state ? wt : split * a.WT + wt + (SHIFT ? a.head_state : 0);
    // What the vectors leave over, while the first copies are on their way
    publish_edges<DT, SHIFT>(
        a, P, T, s_row, nrow, split, S, warp, lane, scale, SHIFT && a.head_state != 0, [&](int j) { return row_slots(a, g, j); },
        [&](int j) { return pub_base + j * pub_stride + (s_state ? a.WT : n_slots - 1); });
    // where this lane's octets of a row sit inside a stage: two tiled copies leave two boxes of 8 rows x 32 octets
    // behind one another, anything else whole rows of the chunk
    const uint32_t lane_off = (TMAP && OPL == 2) ? uint32_t(lane >> 4) * G::kBoxBytes + uint32_t(lane & 15) * 2u * G::kOctetBytes
                                                 : uint32_t(lane) * OPL * G::kOctetBytes;
    const uint32_t srow = (TMAP && OPL == 2) ? 32u * G::kOctetBytes : uint32_t(G::kRowBytes);
    BatchAddr ba;
    ba.row_bytes = uint32_t(a.row_stride * ES);
    ba.vm_bytes = uint32_t(a.vm_stride * 4);
    RowAcc acc[kBatchRows];
    char* rowp[kBatchRows];
    uint8_t* vmp[kBatchRows];
    char* base0 = nullptr;
    uint8_t* vm0 = nullptr;
    int live = 0;
    uint32_t heads = 0u;  // SHIFT: tokens in front of the first vector of the batch's rows, four bits each
    auto open_batch = [&](int rb) {  // fresh row states and row addresses for row batch rb
        if (SHIFT) heads = 0u;
#pragma unroll
        for (int i = 0; i < kBatchRows; ++i) {
            acc[i].init();
            rowp[i] = nullptr;
            vmp[i] = nullptr;
            if (!TMAP) {
                const int row = s_row[min(rb * kBatchRows + i, kGroupRows - 1)];
                rowp[i] = reinterpret_cast<char*>(a.logits) + int64_t(max(row, 0)) * a.row_stride * ES;
                vmp[i] = vm8 ? vm8 + int64_t(max(row, 0)) * a.vm_stride * 4 : nullptr;
                if (SHIFT) {
                    const int head = row_head<DT>(rowp[i], a.V);
                    rowp[i] += head * ES;
                    heads |= uint32_t(head) << (4 * i);
                }
            }
        }
        live = min(kBatchRows, nrow - rb * kBatchRows);
        const int row0 = max(s_row[min(rb * kBatchRows, kGroupRows - 1)], 0);
        base0 = reinterpret_cast<char*>(a.logits) + int64_t(row0) * a.row_stride * ES;
        vm0 = vm8 ? vm8 + int64_t(row0) * a.vm_stride * 4 : nullptr;
    };
    int cur_rb = wr;
    if (cur_rb * kBatchRows < nrow) open_batch(cur_rb);
    __syncwarp();  // slot_info written by lane 0 above
    while (cur_rb * kBatchRows < nrow) {
        const int info = slot_info[slot];
        if (info < 0) break;
        const int rb = info >> 24, o0 = (info & 0xFFFFFF) * kChunkOctets;
        float chunk_m = -INFINITY;
        while (cur_rb < rb) {  // the previous row batch of this warp is complete (possibly without any chunk)
            warp_rows_publish_to(acc, live, cur_rb, lane, scale, pub_base, pub_stride, my_slot);
            cur_rb += WR;
            open_batch(cur_rb);
        }
        // (the test hook lets the wait complete and then reports it as run out, so that the error path below, drain
        // loop included, runs with every copy landed)
        const bool arrived = mbar_wait(bar + slot, phase) && !a.expire_test;
        if (!__all_sync(0xFFFFFFFFu, arrived)) {
            failed = true;
            break;
        }
        const char* src = my_ring + size_t(slot) * G::kStageBytes;
        const int o = o0 + lane * OPL;
        ba.item_base = base0 + size_t(o) * G::kOctetBytes;
        ba.vm_item = vm0 ? vm0 + o : nullptr;
        // (the vectors of a row that starts anywhere end at most one octet before the last whole octet)
        if (live == kBatchRows && o0 + kChunkOctets <= (SHIFT ? n_full - 1 : n_full))
            pipe_consume_item<DT, OPL, true, SRC, MAXIMA>(src, lane_off, srow, T, rb, live, OPL, o, lane, ba, rowp, vmp, acc, scale,
                                                  a.wide != 0, 32, heads, a.V, chunk_m);
        else
            pipe_consume_item<DT, OPL, false, SRC, MAXIMA>(src, lane_off, srow, T, rb, live, max(0, min(OPL, n_full - o)), o, lane, ba,
                                                   rowp, vmp, acc, scale, a.wide != 0, min(n_octets - o0, 32), heads, a.V, chunk_m);
        if (MAXIMA && a.chunk_max && lane < live) a.chunk_max[int64_t(s_row[rb * kBatchRows + lane]) * a.n_chunks + (info & 0xFFFFFF)] = chunk_m;
        ++consumed;
        if (++slot == depth) { slot = 0; phase ^= 1u; }
        __syncwarp();  // every lane has its data out of the slot before it is refilled
        if ((COOP || lane == 0) && !p_end) issue_next();
        __syncwarp();  // slot_info of the refilled slot is visible to the whole warp
    }
    if (!failed) {
        // whatever row batches of this warp are left (all of them if it never got a chunk) are published too
        for (; cur_rb * kBatchRows < nrow; cur_rb += WR) {
            warp_rows_publish_to(acc, live, cur_rb, lane, scale, pub_base, pub_stride, my_slot);
            if ((cur_rb + WR) * kBatchRows < nrow) open_batch(cur_rb + WR);
        }
    } else if (lane == 0) {
        // a copy never arrived: flag it, give the copies still in flight the same bounded time to land
        // (they target this block's shared memory), and let the block leave without results
        atomicAdd(a.status + 3, 1);
        for (int k = consumed; k < p_issued; ++k) {
            mbar_wait(bar + slot, phase);
            if (++slot == depth) { slot = 0; phase ^= 1u; }
        }
    }
    if (!fold && !s_state) return;
    __shared__ int s_last;
    if (s_state) {
        // first the block's own states: one per row and block goes out instead of one per row and warp
        __syncthreads();
        for (int j = warp; j < nrow; j += n_warps) {
            const int n_mine = a.WT + (j % S == split ? 1 : 0);  // the state of what the vectors left over
            float m = -INFINITY, s = 0.f;
            int pos = kNoPos;
            if (lane < n_mine) {
                const Partial p = s_state[j * (a.WT + 1) + lane];
                m = p.m; s = p.s; pos = p.pos;
            }
            partial_warp_allreduce(m, s, pos);
            if (lane == 0) row_slots(a, g, j)[split] = Partial{m, s, pos, 0};
        }
    }
    if (!fold) return;
    // ---- One launch per step: the group's blocks count themselves off, and the last one to finish folds the states
    // of the group's rows and writes their results (what k_finalize_rows does in a launch of its own otherwise).
    __threadfence();  // this block's states and masked logits are visible device-wide before its ticket is drawn
    __syncthreads();
    if (tid == 0) s_last = (atomicAdd(a.tickets + g, 1u) == unsigned(S - 1));
    __syncthreads();
    if (!s_last) return;
    __threadfence();  // the other blocks' states and masked logits, published before their tickets
    for (int j = warp; j < nrow; j += n_warps) {
        float m, s;
        int pos;
        warp_fold_states(row_slots(a, g, j), n_slots, lane, m, s, pos);
        warp_finalize_row<DT>(a, P, s_row[j], m, s, pos, lane);
    }
    if (tid == 0) a.tickets[g] = 0u;  // ready for the next launch
}

// ---------------------------------------------------------------------------------------
// Dense expansion only. Same row groups and class table as the fused kernel; a lane takes sixteen tokens next to its
// neighbours', looks up their class words once, turns them into two bytes per row (eight 8x8 bit transposes for the 32 rows)
// and stores these: 64 bytes side by side per row and warp. per_split counts units of 32 lanes. The class table straight from
// the masks, four words of a row to a lane, where their alignment allows, else by way of shared memory.
// Bound: the chain launch - class masks - table - lookups - stores for all but large batches, and for those instruction issue, some
// 350 instructions per 512 tokens and 32 rows. (Eight tokens a lane, a table for every quarter of an SM and an address from
// scratch for every row took 1070 with the tables: 512 rows of 128256 tokens 15.1 us, now 7.0; 40 rows of
// 200064 in 16384 classes with masking and mapping 56, now 21.)
// ---------------------------------------------------------------------------------------
constexpr int kExpandThreads = 512, kExpandWarps = kExpandThreads / 32;

// PLANNED: the row groups come from a row plan; else they are 32 consecutive rows each.
template <bool PLANNED>
__global__ void __launch_bounds__(kExpandThreads, 2) k_expand_dense(const __grid_constant__ StepArgs a) {
    extern __shared__ __align__(128) uint32_t smem[];
    uint32_t* T = smem;
    int* s_row = reinterpret_cast<int*>(T + a.table_words);
    uint32_t* stage = reinterpret_cast<uint32_t*>(s_row + kGroupRows);

    pdl_launch_dependents();
    if (PLANNED) pdl_wait();
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int g = blockIdx.x / a.S, split = blockIdx.x - g * a.S;
    if (PLANNED && g >= ld_after_wait(a.n_groups)) return;
    const int part = group_rows_setup(a, g, s_row, tid);
    __syncthreads();
    const PartDev P = PLANNED ? a.parts[part] : a.p0;
    const int nrow = PLANNED ? __popc(__ballot_sync(0xFFFFFFFFu, s_row[lane] >= 0)) : min(kGroupRows, a.B - g * kGroupRows);
    const int n_octets = 4 * a.VW, u_end = min((split + 1) * a.per_split, (n_octets + 63) >> 6);
    int unit = split * a.per_split + warp;
    const uint4* const ids = reinterpret_cast<const uint4*>(P.c16);  // padded to 32 * VW entries
    uint4 c0 = make_uint4(0, 0, 0, 0), c1 = c0;
    auto fetch = [&](int u) {
        const int o = u * 64 + lane * 2;
        if (u < u_end && o < n_octets) {
            c0 = __ldg(ids + o);
            c1 = __ldg(ids + o + 1);
        }
    };
    fetch(unit);
    if (!PLANNED) pdl_wait();
    make_class_table(a, P, s_row, T, stage, warp, lane, kExpandWarps);
    __syncthreads();

    uint8_t* const vm8 = reinterpret_cast<uint8_t*>(a.vocab_mask);
    const uint32_t vm_bytes = uint32_t(a.vm_stride * 4);
    for (; unit < u_end; unit += kExpandWarps) {
        const int o = unit * 64 + lane * 2;
        const bool active = o < n_octets;
        const uint4 i0 = c0, i1 = c1;
        fetch(unit + kExpandWarps);
        if (!active) continue;
        const uint32_t w0[8] = {T[i0.x & 0xFFFFu], T[i0.x >> 16], T[i0.y & 0xFFFFu], T[i0.y >> 16],
                                T[i0.z & 0xFFFFu], T[i0.z >> 16], T[i0.w & 0xFFFFu], T[i0.w >> 16]};
        const uint32_t w1[8] = {T[i1.x & 0xFFFFu], T[i1.x >> 16], T[i1.y & 0xFFFFu], T[i1.y >> 16],
                                T[i1.z & 0xFFFFu], T[i1.z >> 16], T[i1.w & 0xFFFFu], T[i1.w >> 16]};
        char* const first = reinterpret_cast<char*>(vm8 + int64_t(g * kGroupRows) * a.vm_stride * 4 + o);
#pragma unroll
        for (int rb = 0; rb < kGroupRows / kBatchRows; ++rb) {
            if (rb * kBatchRows >= nrow) break;
            uint32_t lo0, hi0, lo1, hi1;
            row_batch_bytes(w0, rb, lo0, hi0);
            row_batch_bytes(w1, rb, lo1, hi1);
#pragma unroll
            for (int i = 0; i < kBatchRows; ++i) {
                const int r = rb * kBatchRows + i;
                if (r >= nrow) break;
                const uint32_t two = prmt(i < 4 ? lo0 : hi0, i < 4 ? lo1 : hi1, uint32_t(i & 3) | (uint32_t(4 + (i & 3)) << 4));
                char* const dst = PLANNED ? reinterpret_cast<char*>(vm8 + int64_t(s_row[r]) * a.vm_stride * 4 + o) : ptr_mad(first, uint32_t(r), vm_bytes);
                st_global_u16(dst, two);
            }
        }
    }
}

// ---------------------------------------------------------------------------------------
// Step for rows that allow few tokens. Row groups and class table as in the gather kernels. A warp takes 32 vectors of 32
// bytes (8 f32 or 16 bf16 tokens) of 8 rows at a time; a vector without an allowed token is overwritten with -inf at once,
// without being read, the others go into a queue of the warp. Whenever 32 have come together they are asked for, a lane each,
// and the 32 asked for before are masked, written back and folded into the lane's states of the 8 rows (shared memory).
// Bound: HBM and the latency of the reads. The -inf stream waits for no load; alone it runs at 5.9 TB/s, and the reads, scattered
// sectors between the writes, cost a third on top (measured without them: 1024 rows of 128256 f32 logits 134 -> 100 us; more blocks
// per SM, longer runs per row, asking for the sectors ahead of the stream: no gain); with them DRAM is busy for 52 % of the time
// and the L1 for 61, and a warp waits mostly for loads. Building every row's mask from the class lists first, a block per row, as
// the kernel below does, streams nothing meanwhile: with few classes and long rows that takes 10 to 70 % longer (128 rows of 128256 in
// 512 classes, bf16 26.9 against 17.3 us, f32 30 against 23; 300 bf16 rows of 256000 in two partitions 80 against 46), at 1024 f32 rows
// the same (132). Where the table costs more than it saves the kernel below is taken (few_pays, where the launches are planned).
// Vectors of 32 bytes because a sector whose halves are written at different times costs a read of DRAM.
// ---------------------------------------------------------------------------------------
constexpr int kFewThreads = 256, kFewWarps = kFewThreads / 32;
constexpr int kFewQueue = 64;  // fewer than 32 entries are left when a row adds up to 32
struct FewWarp {
    float m[kBatchRows][32], s[kBatchRows][32];
    int pos[kBatchRows][32];
    uint2 queue[kFewQueue];  // vector << 3 | row of the batch, allow bits
};

template <int DT>
struct FewVec {  // 32 bytes of a row
    static constexpr int kTokens = DT == kBF16 ? 16 : 8;
    Octet<DT> o[DT == kBF16 ? 2 : 1];
    __device__ __forceinline__ void load(const char* p) {
        o[0].load(p, 0);
        if (DT == kBF16) o[DT == kBF16].load(p, 1);
    }
    __device__ __forceinline__ void store(char* p, bool wide) const {
        if constexpr (DT == kBF16) {
            if (wide) {
                st_stream32(p, o[0].v, o[1].v);
            } else {
                o[0].store(p, 0);
                o[1].store(p, 1);
            }
        } else {
            o[0].store_at(p, wide);
        }
    }
};

template <int DT>
__global__ void __launch_bounds__(kFewThreads, 3) k_step_few(const __grid_constant__ StepArgs a) {
    using Vec = FewVec<DT>;
    constexpr int kOct = Vec::kTokens / 8;  // octets per vector
    extern __shared__ __align__(128) uint32_t smem[];
    uint32_t* T = smem;
    int* s_row = reinterpret_cast<int*>(T + a.table_words);
    FewWarp* s_warp = reinterpret_cast<FewWarp*>(s_row + kGroupRows);
    uint32_t* stage = reinterpret_cast<uint32_t*>(s_warp + kFewWarps);

    pdl_prologue();
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int g = blockIdx.x / a.S, split = blockIdx.x - g * a.S;
    if (a.n_groups && g >= ld_after_wait(a.n_groups)) return;
    const int part = group_rows_setup(a, g, s_row, tid);
    __syncthreads();
    const PartDev P = a.group_part ? a.parts[part] : a.p0;
    const int nrow = __popc(__ballot_sync(0xFFFFFFFFu, s_row[lane] >= 0));
    make_class_table(a, P, s_row, T, stage, warp, lane, kFewWarps);
    __syncthreads();

    constexpr int ES = DT == kBF16 ? 2 : 4;
    const int wt = warp % a.WT, wr = warp / a.WT, WR = kFewWarps / a.WT;
    const int n_vec = a.V / Vec::kTokens, n_chunks = (n_vec + 31) >> 5, stride = a.S * a.WT;
    const bool wide = a.wide != 0;
    uint8_t* const vm8 = reinterpret_cast<uint8_t*>(a.vocab_mask);
    publish_edges<DT, false, Vec::kTokens>(
        a, P, T, s_row, nrow, split, a.S, warp, lane, kLog2e, false, [&](int j) { return row_slots(a, g, j); },
        [&](int j) { return row_slots(a, g, j) + a.slots - 1; });
    const uint4* const ids = reinterpret_cast<const uint4*>(P.c16);
    FewWarp& w = s_warp[warp];
    for (int rb = wr; rb * kBatchRows < nrow; rb += WR) {
        const int live = min(kBatchRows, nrow - rb * kBatchRows);
        const int* const rows = s_row + rb * kBatchRows;
        auto row_base = [&](int i) { return reinterpret_cast<char*>(a.logits) + int64_t(rows[i]) * a.row_stride * ES; };
#pragma unroll
        for (int i = 0; i < kBatchRows; ++i) {
            w.m[i][lane] = -INFINITY;
            w.s[i][lane] = 0.f;
            w.pos[i][lane] = kNoPos;
        }
        Vec held;         // what this lane has asked for
        uint2 entry = make_uint2(0u, 0u);  // and its queue entry (no allow bits: nothing)
        auto consume = [&]() {
            if (!entry.y) return;
            const int i = entry.x & 7, v = entry.x >> 3;
            float f[Vec::kTokens];
#pragma unroll
            for (int q = 0; q < kOct; ++q) held.o[q].mask((entry.y >> (8 * q)) & 0xFFu, f + 8 * q);
            held.store(row_base(i) + size_t(v) * 32, wide);
            float m = f[0];
#pragma unroll
            for (int q = 1; q < Vec::kTokens; ++q) m = fmaxf(m, f[q]);
            const float ref = fmaxf(m, kRefFloor);
            float sum = 0.f;
#pragma unroll
            for (int q = 0; q < Vec::kTokens; ++q) sum += ex2f((f[q] - ref) * kLog2e);
            float m0 = w.m[i][lane], s0 = w.s[i][lane];
            int p0 = w.pos[i][lane];
            partial_merge(m0, s0, p0, m, sum, m > -INFINITY ? v * kOct : kNoPos);
            w.m[i][lane] = m0;
            w.s[i][lane] = s0;
            w.pos[i][lane] = p0;
        };
        int head = 0, count = 0;  // of the queue
        auto ask = [&]() {        // consume what was asked for, ask for the next 32 (or what is left)
            consume();
            entry = make_uint2(0u, 0u);
            if (lane < count) {
                entry = w.queue[(head + lane) & (kFewQueue - 1)];
                held.load(row_base(entry.x & 7) + size_t(entry.x >> 3) * 32);
            }
            const int n = min(count, 32);
            head += n;
            count -= n;
            __syncwarp();
        };
        int c = (split * a.WT + wt - rb * a.rot_chunks) % stride;  // the deal starts at another warp for every row batch
        if (c < 0) c += stride;
        uint4 cv[kOct];
        auto fetch_ids = [&](int chunk) {
#pragma unroll
            for (int q = 0; q < kOct; ++q)
                if (chunk * 32 + lane < n_vec) cv[q] = __ldg(ids + (chunk * 32 + lane) * kOct + q);
        };
        fetch_ids(c);
        for (; c < n_chunks; c += stride) {
            const int v = c * 32 + lane;
            const bool active = v < n_vec;
            uint32_t lo[kOct], hi[kOct];
#pragma unroll
            for (int q = 0; q < kOct; ++q) octet_allow_bits(cv[q], T, rb, active, lo[q], hi[q]);
            fetch_ids(c + stride);
#pragma unroll
            for (int i = 0; i < kBatchRows; ++i) {
                if (i >= live) break;
                uint32_t bits = 0u;
#pragma unroll
                for (int q = 0; q < kOct; ++q) bits |= (((i < 4 ? lo[q] : hi[q]) >> (8 * (i & 3))) & 0xFFu) << (8 * q);
                const int row = rows[i];
                if (active && vm8) {
                    uint8_t* const vm = vm8 + int64_t(row) * a.vm_stride * 4 + v * kOct;
                    if (kOct == 1) st_global_u8(vm, bits); else st_global_u16(vm, bits);
                }
                const uint32_t some = __ballot_sync(0xFFFFFFFFu, bits != 0u);
                if (bits) {
                    w.queue[(head + count + __popc(some & ((1u << lane) - 1u))) & (kFewQueue - 1)] =
                        make_uint2((unsigned(v) << 3) | unsigned(i), bits);
                } else if (active) {
                    Vec none;
#pragma unroll
                    for (int q = 0; q < kOct; ++q) none.o[q].fill_neg_inf();
                    none.store(reinterpret_cast<char*>(a.logits) + int64_t(row) * a.row_stride * ES + size_t(v) * 32, wide);
                }
                count += __popc(some);
                __syncwarp();
                if (count >= 32) ask();
            }
        }
        ask();
        ask();
        consume();
        RowAcc acc[kBatchRows];
#pragma unroll
        for (int i = 0; i < kBatchRows; ++i) {
            acc[i].m = w.m[i][lane];
            acc[i].s = w.s[i][lane];
            acc[i].nrl = -(acc[i].m * kLog2e);
            if (!(acc[i].m * kLog2e > kRefLow)) {
                acc[i].s = 0.f;
                acc[i].nrl = -kRefLow;
            }
            acc[i].pos = w.pos[i][lane];
        }
        warp_rows_publish(a, acc, live, g, split * a.WT + wt, rb, lane);
    }
}

// ---------------------------------------------------------------------------------------
// The same for few or short rows, for many classes and for class ids beyond 16 bits: one row per block (S blocks per row).
// The row's vocab bitmask is built in shared memory by scattering the member lists of the allowed classes; then the row is
// streamed: octets with no allowed token are overwritten with -inf without being read.
// FUSED = false stops after writing the vocab mask.
// ---------------------------------------------------------------------------------------
constexpr int kBigClass = 256;   // classes at least this large are scattered by the whole block
constexpr int kBigListCap = 64;

__device__ __forceinline__ int lower_bound_tok(const int32_t* tok, int lo, int hi, int t) {
    while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if (__ldg(tok + mid) < t) lo = mid + 1; else hi = mid;
    }
    return lo;
}

template <int DT, bool FUSED>
__global__ void __launch_bounds__(256) k_step_sparse(const __grid_constant__ StepArgs a) {
    extern __shared__ __align__(128) uint32_t smem[];
    uint32_t* bits = smem;  // per_split words
    __shared__ int s_big[kBigListCap];
    __shared__ int s_nbig;
    __shared__ int s_last;
    __shared__ Partial s_red[8];

    pdl_prologue();
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, n_warps = blockDim.x >> 5;
    int row = blockIdx.x / a.S;
    const int split = blockIdx.x - row * a.S;
    __shared__ int s_batch[kBatchRows];
    if (a.row_mode) {
        // Automatic mode: the grid covers the (group, row slot) pairs of the gather kernel, and the choice is made
        // for the 8 row slots that kernel streams together (its row batch), so that no row is done twice.
        const int g = row / kGroupRows, j = row - g * kGroupRows;
        if (a.n_groups && g >= ld_after_wait(a.n_groups)) return;
        if (tid < kBatchRows) {
            const int slot = g * kGroupRows + (j & ~(kBatchRows - 1)) + tid;
            int r = a.group_rows ? a.group_rows[slot] : slot;
            if (r >= a.B) r = -1;
            s_batch[tid] = r;
        }
        __syncthreads();
        row = s_batch[j & (kBatchRows - 1)];
        if (row < 0) return;
    }
    const int part = a.row_part ? a.row_part[row] : a.part0;
    if (part < 0 || part >= a.n_parts || !a.parts[part].live || a.parts[part].V != a.V) {
        if (tid == 0 && split == 0) atomicAdd(a.status + 2, 1);  // (never in automatic mode: only grouped rows come here)
        return;
    }
    const PartDev P = a.parts[part];
    const int w_begin = split * a.per_split, w_end = min(w_begin + a.per_split, a.VW);
    const int t0 = w_begin * 32, t1 = min(w_end * 32, a.V);
    const uint32_t* cm = a.class_mask + int64_t(row) * a.cm_stride;
    if (a.row_mode) {
        // This kernel runs first and keeps the row batches that allow few tokens (it never reads a logit that is not
        // allowed); the others it leaves, marked, to the gather kernel launched behind it. The tokens a row allows
        // are the summed sizes of its allowed classes; the rows of a batch share their partition.
        __shared__ unsigned long long s_allowed;
        if (tid == 0) s_allowed = 0ull;
        __syncthreads();
        unsigned long long mine = 0ull;
        int n_live = 0;
#pragma unroll
        for (int q = 0; q < kBatchRows; ++q) n_live += s_batch[q] >= 0;
        // a thread per class: how many of the batch's rows allow it (their mask words are the same address for the 32
        // lanes of a warp), times its size; the cost does not depend on how many classes are allowed
        for (int k = tid; k < P.K; k += blockDim.x) {
            int cnt = 0;
#pragma unroll
            for (int q = 0; q < kBatchRows; ++q) {
                const int r = s_batch[q];
                if (r >= 0) cnt += (ld_after_wait(a.class_mask + int64_t(r) * a.cm_stride + (k >> 5)) >> (k & 31)) & 1u;
            }
            if (cnt) mine += static_cast<unsigned long long>(cnt) * static_cast<unsigned>(__ldg(P.off + k + 1) - __ldg(P.off + k));
        }
#pragma unroll
        for (int d = 16; d >= 1; d >>= 1) mine += __shfl_xor_sync(0xFFFFFFFFu, mine, d);
        if (lane == 0 && mine) atomicAdd(&s_allowed, mine);
        __syncthreads();
        const bool keep = s_allowed * 1000ull < static_cast<unsigned long long>(a.auto_permille) * unsigned(n_live) * unsigned(a.V);
        if (tid == 0 && split == 0) a.row_mode[row] = keep ? 1 : 0;
        if (!keep) return;
    }
    for (int i = tid; i < a.per_split; i += blockDim.x) bits[i] = 0u;
    if (tid == 0) s_nbig = 0;
    __syncthreads();

    for (int kw = warp; kw < P.KW; kw += n_warps) {
        uint32_t word = ld_after_wait(cm + kw);
        if (kw == P.KW - 1 && (P.K & 31)) word &= (1u << (P.K & 31)) - 1u;
        while (word) {
            const int k = kw * 32 + __ffs(word) - 1;
            word &= word - 1u;
            int lo = __ldg(P.off + k), hi = __ldg(P.off + k + 1);
            if (a.S > 1) {
                lo = lower_bound_tok(P.tok, lo, hi, t0);
                hi = lower_bound_tok(P.tok, lo, hi, t1);
            }
            if (hi - lo >= kBigClass) {
                int slot = 0;
                if (lane == 0) slot = atomicAdd(&s_nbig, 1);
                slot = __shfl_sync(0xFFFFFFFFu, slot, 0);
                if (slot < kBigListCap) {
                    if (lane == 0) s_big[slot] = k;
                    continue;
                }
            }
            for (int i = lo + lane; i < hi; i += 4 * 32) {  // four member ids in flight per lane
                int t[4];
#pragma unroll
                for (int q = 0; q < 4; ++q) t[q] = i + 32 * q < hi ? __ldg(P.tok + i + 32 * q) : -1;
#pragma unroll
                for (int q = 0; q < 4; ++q)
                    if (t[q] >= 0) atomicOr(bits + ((t[q] >> 5) - w_begin), 1u << (t[q] & 31));
            }
        }
    }
    __syncthreads();
    const int nbig = min(s_nbig, kBigListCap);
    for (int b = 0; b < nbig; ++b) {
        const int k = s_big[b];
        int lo = __ldg(P.off + k), hi = __ldg(P.off + k + 1);
        if (a.S > 1) {
            lo = lower_bound_tok(P.tok, lo, hi, t0);
            hi = lower_bound_tok(P.tok, lo, hi, t1);
        }
        for (int i = lo + tid; i < hi; i += 4 * blockDim.x) {
            int t[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) t[q] = i + int(blockDim.x) * q < hi ? __ldg(P.tok + i + blockDim.x * q) : -1;
#pragma unroll
            for (int q = 0; q < 4; ++q)
                if (t[q] >= 0) atomicOr(bits + ((t[q] >> 5) - w_begin), 1u << (t[q] & 31));
        }
    }
    __syncthreads();

    if (a.vocab_mask) {
        uint32_t* out = a.vocab_mask + int64_t(row) * a.vm_stride;
        for (int w = w_begin + tid; w < w_end; w += blockDim.x) out[w] = bits[w - w_begin];
    }
    if (!FUSED) return;

    constexpr int ES = DT == kBF16 ? 2 : 4;
    char* rowp = reinterpret_cast<char*>(a.logits) + int64_t(row) * a.row_stride * ES;
    const uint8_t* bytes = reinterpret_cast<const uint8_t*>(bits);
    const int o_begin = 4 * w_begin, o_end = 4 * w_end, n_full = a.V >> 3;
    const int o_vec_end = min(o_end, n_full);
    RowAcc acc;
    acc.init();
    constexpr int U = 4;
    for (int ob = o_begin + tid; ob < o_vec_end; ob += U * blockDim.x) {
        Octet<DT> oc[U];
        uint32_t byte[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int o = ob + u * blockDim.x;
            byte[u] = o < o_vec_end ? bytes[o - o_begin] : 0u;
            if (byte[u]) oc[u].load(rowp, o);  // octets without an allowed token are never read
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int o = ob + u * blockDim.x;
            if (o >= o_vec_end) continue;
            if (byte[u] == 0u) {
                oc[u].fill_neg_inf();
                oc[u].store(rowp, o, a.wide != 0);
            } else {
                float f[8];
                oc[u].mask(byte[u], f);
                if (byte[u] != 0xFFu) oc[u].store(rowp, o, a.wide != 0);
                acc.add_octet(f, o);
            }
        }
    }
    // octets past the last whole vector (ragged end of the row, padding of the last mask word)
    if (o_end > n_full) {
        const int o = max(o_begin, n_full) + tid;
        if (o < o_end) {
            float f[8];
            const uint32_t byte = bytes[o - o_begin];
            octet_scalar<DT>(rowp, o, a.V, byte, f);
            if (byte) acc.add_octet(f, o);
        }
    }
    const Partial mine = acc.to_partial();
    float m = mine.m, s = mine.s;
    int pos = mine.pos;
    partial_warp_allreduce(m, s, pos);
    if (lane == 0) s_red[warp] = Partial{m, s, pos, 0};
    __threadfence();  // the row's masked logits must be visible to whichever block finishes the row
    __syncthreads();
    if (warp == 0) {
        if (lane == 0)
            for (int w = 1; w < n_warps; ++w) partial_merge(m, s, pos, s_red[w].m, s_red[w].s, s_red[w].pos);
        if (a.S == 1) {
            m = __shfl_sync(0xFFFFFFFFu, m, 0);
            s = __shfl_sync(0xFFFFFFFFu, s, 0);
            pos = __shfl_sync(0xFFFFFFFFu, pos, 0);
            warp_finalize_row<DT>(a, P, row, m, s, pos, lane);
        } else if (lane == 0) {
            a.partials[int64_t(row) * a.S + split] = Partial{m, s, pos, 0};
            __threadfence();
            s_last = (atomicAdd(a.tickets + row, 1u) == unsigned(a.S - 1));
        }
    }
    if (a.S == 1) return;
    __syncthreads();
    if (!s_last || warp != 0) return;
    __threadfence();
    float m2 = -INFINITY, s2 = 0.f;
    int p2 = kNoPos;
    for (int sp = lane; sp < a.S; sp += 32) {
        const int4 raw = __ldcg(reinterpret_cast<const int4*>(a.partials + int64_t(row) * a.S + sp));
        partial_merge(m2, s2, p2, __int_as_float(raw.x), __int_as_float(raw.y), raw.z);
    }
    partial_warp_allreduce(m2, s2, p2);
    warp_finalize_row<DT>(a, P, row, m2, s2, p2, lane);
    if (lane == 0) a.tickets[row] = 0u;
}

// ---------------------------------------------------------------------------------------
// Generic step: one block per row, one token per thread per iteration, no alignment or
// size requirement (any K, int32 class ids, odd strides). FUSED = false: expansion only.
// ---------------------------------------------------------------------------------------
template <int DT, bool FUSED>
__global__ void __launch_bounds__(256) k_step_generic(const __grid_constant__ StepArgs a) {
    __shared__ Partial s_red[8];
    pdl_prologue();
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, n_warps = blockDim.x >> 5;
    const int row = blockIdx.x;
    const int part = a.row_part ? a.row_part[row] : a.part0;
    if (part < 0 || part >= a.n_parts || !a.parts[part].live || a.parts[part].V != a.V) {
        if (tid == 0) atomicAdd(a.status + 2, 1);
        return;
    }
    const PartDev P = a.parts[part];
    const uint32_t* cm = a.class_mask + int64_t(row) * a.cm_stride;
    constexpr int ES = DT == kBF16 ? 2 : 4;
    char* rowp = FUSED ? reinterpret_cast<char*>(a.logits) + int64_t(row) * a.row_stride * ES : nullptr;
    uint32_t* out = a.vocab_mask ? a.vocab_mask + int64_t(row) * a.vm_stride : nullptr;
    float m = -INFINITY, s = 0.f;
    int pos = kNoPos;
    for (int w = warp; w < a.VW; w += n_warps) {
        const int t = w * 32 + lane;
        bool allowed = false;
        if (t < a.V) {
            const int k = __ldg(P.c32 + t);
            allowed = (ld_after_wait(cm + (k >> 5)) >> (k & 31)) & 1u;
        }
        const uint32_t word = __ballot_sync(0xFFFFFFFFu, allowed);
        if (out && lane == 0) out[w] = word;
        if (FUSED && t < a.V) {
            if (allowed) {
                const float z = load_elem<DT>(rowp, t);
                const bool upd = (z > m) || pos == kNoPos;
                pos = upd ? t : pos;
                const float ref_old = fmaxf(m, kRefFloor);
                m = fmaxf(m, z);
                const float ref = fmaxf(m, kRefFloor);
                s = fmaf(s, ex2f((ref_old - ref) * a.scale), ex2f((z - ref) * a.scale));
            } else {
                store_neg_inf<DT>(rowp, t);
            }
        }
    }
    if (!FUSED) return;
    partial_warp_allreduce(m, s, pos, a.scale);
    if (lane == 0) s_red[warp] = Partial{m, s, pos, 0};
    __syncthreads();
    if (tid == 0) {
        for (int w = 1; w < n_warps; ++w) partial_merge(m, s, pos, s_red[w].m, s_red[w].s, s_red[w].pos, a.scale);
        if (a.u)
            a.partials[row] = Partial{m, s, pos, 0};  // a sampling step: the sampling kernel takes it from here
        else
            finalize_row<DT>(a, P, row, m, s, pos, true);
    }
}

// ---------------------------------------------------------------------------------------
// Second kernel of a sampling step: one block per row draws the row's token from the tempered
// distribution over its allowed tokens by inverse CDF in token order, with the row's uniform number
// u: the lowest token whose cumulative weight exceeds u times the total. The states the streaming
// kernel published stand for consecutive runs of tokens (state k: chunks [k * run_chunks,
// (k+1) * run_chunks) of chunk_tokens tokens; with tail_state the last one: the tokens past the last whole
// vector), so the block first scans the states for the run that holds the crossing, then re-reads
// the masked logits of that run only and scans them. All sums are taken in a fixed order.
// ---------------------------------------------------------------------------------------
constexpr int kSampleThreads = 256;

// Exclusive prefix sum of one value per thread over the block, in thread order; total to everybody.
__device__ __forceinline__ float block_exclusive_scan(float v, float* s_warp, float& total) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    float inc = v;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const float up = __shfl_up_sync(0xFFFFFFFFu, inc, d);
        if (lane >= d) inc += up;
    }
    if (lane == 31) s_warp[warp] = inc;  // the caller gives every call an array no thread may still be reading
    __syncthreads();
    float before = 0.f, all = 0.f;
#pragma unroll
    for (int w = 0; w < kSampleThreads / 32; ++w) {
        const float t = s_warp[w];
        if (w < warp) before += t;
        all += t;
    }
    total = all;
    return before + inc - v;
}

// SHARED_OUT: a.group_w is set (its code is kept out of the kernel for the short steps without a row plan).
template <int DT, bool SHARED_OUT>
__global__ void __launch_bounds__(kSampleThreads) k_sample_rows(const __grid_constant__ StepArgs a, int aligned) {
    __shared__ float s_warp[kSampleThreads / 32], s_scan_states[kSampleThreads / 32], s_scan_tokens[kSampleThreads / 32];
    __shared__ int s_pick, s_last;
    __shared__ int s_pick_state, s_last_state;
    __shared__ float s_base;
    pdl_prologue();
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int g = blockIdx.x / kGroupRows, j = blockIdx.x - g * kGroupRows;
    if (a.n_groups && g >= ld_after_wait(a.n_groups)) return;
    int row;
    if (a.group_rows) {
        row = a.group_rows[g * kGroupRows + j];
    } else {
        row = g * kGroupRows + j;
        if (row >= a.B) row = -1;
    }
    if (row < 0) return;
    PartDev P = a.p0;
    if (a.group_part) {
        P = a.parts[a.group_part[g]];
    } else if (a.row_part) {
        const int part = a.row_part[row];
        if (part < 0 || part >= a.n_parts || !a.parts[part].live || a.parts[part].V != a.V) return;  // counted by the step kernel
        P = a.parts[part];
    }
    const Partial* src = row_slots(a, g, j);
    const float u = ld_after_wait(a.u + row);  // needed late: in flight together with the states
    const int n_states = SHARED_OUT ? group_states(a, g) : a.slots;
    const int per = (n_states + kSampleThreads - 1) / kSampleThreads;  // consecutive states per thread
    const int k0 = tid * per, k1 = min(k0 + per, n_states);

    // the states of this thread: fetched once, all loads in flight together, kept in registers when there are
    // at most four of them (otherwise they are fetched again wherever they are needed)
    constexpr int kKeep = 4;
    const bool kept = per <= kKeep;
    float km[kKeep], ks[kKeep];
#pragma unroll
    for (int i = 0; i < kKeep; ++i) {
        km[i] = -INFINITY;
        ks[i] = 0.f;
        if (kept && k0 + i < k1) {
            const int4 raw = __ldcg(reinterpret_cast<const int4*>(src + k0 + i));
            km[i] = __int_as_float(raw.x);
            ks[i] = __int_as_float(raw.y);
        }
    }
    // the row maximum
    float M = -INFINITY;
    if (kept) {
#pragma unroll
        for (int i = 0; i < kKeep; ++i) M = fmaxf(M, km[i]);
    } else {
        for (int k = k0; k < k1; ++k) M = fmaxf(M, __ldcg(&src[k].m));
    }
#pragma unroll
    for (int d = 16; d >= 1; d >>= 1) M = fmaxf(M, __shfl_xor_sync(0xFFFFFFFFu, M, d));
    if (lane == 0) s_warp[warp] = M;
    if (tid == 0) {
        s_pick = kNoPos;
        s_last = -1;
        s_pick_state = kNoPos;
        s_last_state = -1;
    }
    __syncthreads();
#pragma unroll
    for (int w = 0; w < kSampleThreads / 32; ++w) M = fmaxf(M, s_warp[w]);
    if (!(M * a.scale > kRefLow)) {
        // nothing allowed, or nothing that weighs anything: the lowest allowed token (if any) and -inf logs
        if (warp == 0) {
            unsigned long long cand = first_allowed_share(a, P, row, lane, 32);
#pragma unroll
            for (int d = 16; d >= 1; d >>= 1) {
                const unsigned long long other = __shfl_xor_sync(0xFFFFFFFFu, cand, d);
                cand = other < cand ? other : cand;
            }
            if (lane == 0) write_row_outputs(a, row, -INFINITY, 0.f, cand);
        }
        return;
    }

    // weights of the states relative to M, their exclusive prefix sums in token order, the total
#pragma unroll
    for (int i = 0; i < kKeep; ++i) ks[i] *= ex2f((fmaxf(km[i], kRefFloor) - M) * a.scale);  // now the weight (0 if unused)
    auto weight = [&](int k) {
        if (kept) {
            float w = 0.f;
#pragma unroll
            for (int i = 0; i < kKeep; ++i) w = (k - k0 == i) ? ks[i] : w;
            return w;
        }
        const int4 raw = __ldcg(reinterpret_cast<const int4*>(src + k));
        return __int_as_float(raw.y) * ex2f((fmaxf(__int_as_float(raw.x), kRefFloor) - M) * a.scale);
    };
    float mine = 0.f;
    for (int k = k0; k < k1; ++k) mine += weight(k);
    float total;
    const float front = block_exclusive_scan(mine, s_scan_states, total);  // weight in front of this thread's states
    const float tau = u * total;
    float run = front;
    for (int k = k0; k < k1; ++k) {
        const float w = weight(k);
        if (w > 0.f) {
            atomicMax(&s_last_state, k);
            if (run + w > tau) {
                atomicMin(&s_pick_state, k);
                break;
            }
        }
        run += w;
    }
    __syncthreads();
    // rounding may leave tau at the very end: then the last run with weight
    const int pick = s_pick_state != kNoPos ? s_pick_state : s_last_state;
    if (pick >= k0 && pick < k1) {  // the thread that owns the chosen state: the weight in front of it
        float r2 = front;
        for (int k = k0; k < pick; ++k) r2 += weight(k);
        s_base = r2;
    }
    __syncthreads();
    float base = s_base;

    // the tokens the chosen state stands for
    constexpr int ES = DT == kBF16 ? 2 : 4;
    const char* rowp = reinterpret_cast<const char*>(a.logits) + int64_t(row) * a.row_stride * ES;
    const int head = a.shifted ? row_head<DT>(rowp, a.V) : 0;
    const int vec_end = head + ((a.V - head) & ~7);  // first token past the last whole vector
    int run_chunks = a.run_chunks;
    if (SHARED_OUT) run_chunks = group_run_chunks(a.V >> 3, a.chunk_tokens >> 3, group_share(a, g).S * a.WT);
    int t_lo, t_hi;
    if (a.tail_state && pick == n_states - 1) {
        t_lo = vec_end;
        t_hi = a.V;
    } else if (a.head_state && pick == 0) {
        t_lo = 0;
        t_hi = head;
    } else {
        const long long lim = a.tail_state ? vec_end : a.V, run_tokens = static_cast<long long>(run_chunks) * a.chunk_tokens;
        const long long first = head + (pick - a.head_state) * run_tokens;
        t_lo = int(min(first, lim));
        t_hi = int(min(first + run_tokens, lim));
    }
    auto load8 = [&](int t0, float (&e)[8]) {
        if (aligned && t0 + 8 <= t_hi) {  // t_lo is on a vector boundary: 16-byte (bf16) / 32-byte (f32) vectors
            if (DT == kBF16) {
                const uint4 v = __ldcg(reinterpret_cast<const uint4*>(rowp + size_t(t0) * 2));
                e[0] = __uint_as_float(v.x << 16); e[1] = __uint_as_float(v.x & 0xFFFF0000u);
                e[2] = __uint_as_float(v.y << 16); e[3] = __uint_as_float(v.y & 0xFFFF0000u);
                e[4] = __uint_as_float(v.z << 16); e[5] = __uint_as_float(v.z & 0xFFFF0000u);
                e[6] = __uint_as_float(v.w << 16); e[7] = __uint_as_float(v.w & 0xFFFF0000u);
            } else {
                const float4 v0 = __ldcg(reinterpret_cast<const float4*>(rowp + size_t(t0) * 4));
                const float4 v1 = __ldcg(reinterpret_cast<const float4*>(rowp + size_t(t0) * 4 + 16));
                e[0] = v0.x; e[1] = v0.y; e[2] = v0.z; e[3] = v0.w;
                e[4] = v1.x; e[5] = v1.y; e[6] = v1.z; e[7] = v1.w;
            }
        } else {
#pragma unroll
            for (int q = 0; q < 8; ++q) e[q] = t0 + q < t_hi ? ldcg_elem<DT>(rowp, t0 + q) : -INFINITY;
        }
    };
    auto write_token = [&](int token, float zt, int repv) {
        const float l = logf(total);
        a.argmax[row] = token;
        if (a.rep) a.rep[row] = repv;
        if (a.lse) a.lse[row] = fmaf(M, a.inv_t, l);
        if (a.logp_argmax) a.logp_argmax[row] = (zt - M) * a.inv_t - l;
    };
    auto write_empty = [&]() {  // no token of the run carried weight: report the row as empty
        a.argmax[row] = -1;
        if (a.rep) a.rep[row] = -1;
        if (a.lse) a.lse[row] = -INFINITY;
        if (a.logp_argmax) a.logp_argmax[row] = -INFINITY;
    };
    if (pick < 0) {  // no state carried weight
        if (tid == 0) write_empty();
        return;
    }
    int token = -1;
    for (int p0 = t_lo; p0 < t_hi; p0 += kSampleThreads * 8) {
        const int t0 = p0 + tid * 8;
        float e[8];
        load8(t0, e);
        float z8[8], sum8 = 0.f;
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            z8[q] = e[q];
            e[q] = ex2f((e[q] - M) * a.scale);  // a masked logit is -inf: weight 0
            sum8 += e[q];
        }
        float piece;
        float r3 = base + block_exclusive_scan(sum8, s_scan_tokens, piece);
        int mine_tok = -1, mine_last = -1;
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            if (e[q] > 0.f && mine_tok < 0) {
                mine_last = t0 + q;
                r3 += e[q];
                if (r3 > tau) mine_tok = t0 + q;
            }
        }
        if (mine_last >= 0) atomicMax(&s_last, mine_last);
        if (mine_tok >= 0) atomicMin(&s_pick, mine_tok);
        int my_rep = mine_tok >= 0 ? __ldg(P.trep + mine_tok) : -1;  // in flight across the barrier
        __syncthreads();
        token = s_pick != kNoPos ? s_pick : -1;
        const bool last_piece = p0 + kSampleThreads * 8 >= t_hi;
        if (token < 0 && last_piece) token = s_last;  // rounding: the last token with weight in the run
        if (token >= t0 && token < t0 + 8) {          // the thread that holds the token writes the row's results
            float zt = 0.f;
#pragma unroll
            for (int q = 0; q < 8; ++q) zt = (token - t0 == q) ? z8[q] : zt;
            if (token != mine_tok) my_rep = __ldg(P.trep + token);
            write_token(token, zt, my_rep);
        }
        if (token >= 0) break;
        base += piece;
    }
    if (token < 0 && tid == 0) write_empty();
}

// ---------------------------------------------------------------------------------------
// Row-split step on caller-provided tables: the per-row kernel above, with each row shared by
// S blocks that meet through a scratch area of (max, sum-exp, token) states and one ticket
// per row, exactly as the sparse kernel's blocks do. It touches no context: token->class and
// class->representative vectors, masks, logits and outputs all come from the caller, the
// scratch area from whoever launches it.
// ---------------------------------------------------------------------------------------
struct RowSplitArgs {
    const int32_t* c;   // dev [V]
    const int32_t* r;   // dev [K]
    int32_t V, K, VW;
    const uint32_t* class_mask;
    int64_t cm_stride;
    void* logits;
    int64_t row_stride;
    uint32_t* vocab_mask;  // nullable
    int64_t vm_stride;
    int32_t* argmax;
    int32_t* rep;          // nullable
    float* logp_argmax;    // nullable
    float* lse;            // nullable
    int32_t B, S, words_per_split;
    Partial* partials;     // [B * S]
    unsigned int* tickets; // [B], zero on entry, left zero
};

template <int DT>
__global__ void __launch_bounds__(256) k_step_rowsplit(const __grid_constant__ RowSplitArgs a) {
    __shared__ Partial s_red[8];
    __shared__ int s_last;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, n_warps = blockDim.x >> 5;
    const int row = blockIdx.x / a.S, split = blockIdx.x - row * a.S;
    const uint32_t* cm = a.class_mask + int64_t(row) * a.cm_stride;
    constexpr int ES = DT == kBF16 ? 2 : 4;
    char* rowp = reinterpret_cast<char*>(a.logits) + int64_t(row) * a.row_stride * ES;
    uint32_t* out = a.vocab_mask ? a.vocab_mask + int64_t(row) * a.vm_stride : nullptr;
    const int w_begin = split * a.words_per_split, w_end = min(w_begin + a.words_per_split, a.VW);
    float m = -INFINITY, s = 0.f;
    int pos = kNoPos;
    for (int w = w_begin + warp; w < w_end; w += n_warps) {
        const int t = w * 32 + lane;
        bool allowed = false;
        if (t < a.V) {
            const int k = __ldg(a.c + t);
            if (k >= 0 && k < a.K) allowed = (__ldg(cm + (k >> 5)) >> (k & 31)) & 1u;  // ids out of range: not allowed
        }
        const uint32_t word = __ballot_sync(0xFFFFFFFFu, allowed);
        if (out && lane == 0) out[w] = word;
        if (t < a.V) {
            if (allowed) {
                const float z = load_elem<DT>(rowp, t);
                const bool upd = (z > m) || pos == kNoPos;
                pos = upd ? t : pos;
                const float ref_old = fmaxf(m, kRefFloor);
                m = fmaxf(m, z);
                const float ref = fmaxf(m, kRefFloor);
                s = fmaf(s, ex2f((ref_old - ref) * kLog2e), ex2f((z - ref) * kLog2e));
            } else {
                store_neg_inf<DT>(rowp, t);
            }
        }
    }
    partial_warp_allreduce(m, s, pos);
    if (lane == 0) s_red[warp] = Partial{m, s, pos, 0};
    __syncthreads();
    if (warp != 0) return;
    if (lane == 0)
        for (int w = 1; w < n_warps; ++w) partial_merge(m, s, pos, s_red[w].m, s_red[w].s, s_red[w].pos);
    if (a.S > 1) {
        if (lane == 0) {
            a.partials[int64_t(row) * a.S + split] = Partial{m, s, pos, 0};
            __threadfence();
            s_last = (atomicAdd(a.tickets + row, 1u) == unsigned(a.S - 1));
        }
        __syncwarp();
        if (!s_last) return;
        __threadfence();
        m = -INFINITY; s = 0.f; pos = kNoPos;
        for (int sp = lane; sp < a.S; sp += 32) {
            const int4 raw = __ldcg(reinterpret_cast<const int4*>(a.partials + int64_t(row) * a.S + sp));
            partial_merge(m, s, pos, __int_as_float(raw.x), __int_as_float(raw.y), raw.z);
        }
        partial_warp_allreduce(m, s, pos);
        if (lane == 0) a.tickets[row] = 0u;
    }
    if (lane != 0) return;
    int tok = -1, repv = -1;
    float lsev = -INFINITY, lpa = -INFINITY;
    if (pos != kNoPos) {
        tok = pos;
        const int k = a.c[tok];
        repv = a.r[k];
        if (m > kRefFloor && s > 0.f) {
            const float l = logf(s);
            lsev = m + l;
            lpa = -l;
        }
    }
    a.argmax[row] = tok;
    if (a.rep) a.rep[row] = repv;
    if (a.lse) a.lse[row] = lsev;
    if (a.logp_argmax) a.logp_argmax[row] = lpa;
}

// ---------------------------------------------------------------------------------------
// Row plan for batches that mix partitions: bucket the rows by partition into groups of
// up to 32 rows (valid slots first). One block.
// ---------------------------------------------------------------------------------------
constexpr int kMaxParts = 256;

__global__ void __launch_bounds__(1024) k_plan_rows(const PartDev* parts, int n_parts, const int32_t* row_part, int B,
                                                    int V, int max_groups, int32_t* group_part, int32_t* group_rows,
                                                    int32_t* n_groups, int32_t* group_w, int32_t* status) {
    __shared__ int cnt[kMaxParts], gbase[kMaxParts + 1], cur[kMaxParts];
    pdl_prologue();
    const int tid = threadIdx.x;
    for (int p = tid; p < kMaxParts; p += blockDim.x) { cnt[p] = 0; cur[p] = 0; }
    __syncthreads();
    for (int b = tid; b < B; b += blockDim.x) {
        const int p = row_part[b];
        if (p >= 0 && p < n_parts && parts[p].live && parts[p].V == V) atomicAdd(&cnt[p], 1);
        else atomicAdd(status + 2, 1);
    }
    __syncthreads();
    if (tid == 0) {
        int acc = 0;
        for (int p = 0; p < n_parts; ++p) { gbase[p] = acc; acc += (cnt[p] + kGroupRows - 1) / kGroupRows; }
        gbase[n_parts] = acc;
        *n_groups = acc;
        int w = 0, gq = 0;  // row batches in front of every group
        for (int p = 0; p < n_parts; ++p)
            for (int left = cnt[p]; left > 0; left -= kGroupRows) {
                group_w[gq++] = w;
                w += (min(left, kGroupRows) + kBatchRows - 1) / kBatchRows;
            }
        for (; gq <= max_groups; ++gq) group_w[gq] = w;
    }
    __syncthreads();
    const int total = gbase[n_parts];
    for (int i = tid; i < max_groups * kGroupRows; i += blockDim.x) group_rows[i] = -1;
    for (int p = 0; p < n_parts; ++p)
        for (int gq = gbase[p] + tid; gq < gbase[p + 1]; gq += blockDim.x) group_part[gq] = p;
    for (int gq = total + tid; gq < max_groups; gq += blockDim.x) group_part[gq] = 0;
    __syncthreads();
    for (int b = tid; b < B; b += blockDim.x) {
        const int p = row_part[b];
        if (p >= 0 && p < n_parts && parts[p].live && parts[p].V == V) {
            const int slot = atomicAdd(&cur[p], 1);
            group_rows[(gbase[p] + slot / kGroupRows) * kGroupRows + (slot % kGroupRows)] = b;
        }
    }
}

// ---------------------------------------------------------------------------------------
// mask_logits: apply an existing vocab bitmask in place. A row's vectors begin at its own first vector boundary, `head` tokens
// in (0 for rows on the vector grid), so vector o takes its 8 bits from the bytes o and o + 1 of the mask. Vectors whose 8
// tokens are all allowed are neither read nor written; those with none allowed are written without a read. The tokens left
// over at both ends go one by one.
// Bound: HBM (read and write once). The mask bytes of the next piece of work are fetched while the logits of this one are
// on their way.
// ---------------------------------------------------------------------------------------
constexpr int kMaskUnroll = 2, kMaskChunk = 256 * kMaskUnroll;  // vectors per block and piece

template <int DT>
__global__ void __launch_bounds__(256) k_mask_logits(void* logits, int64_t row_stride, int B, int V, const uint32_t* vocab_mask,
                                                     int64_t vm_stride, int chunks, int row_step, int ch_step) {
    pdl_prologue();
    constexpr int ES = DT == kBF16 ? 2 : 4;
    const int tid = threadIdx.x;
    struct Piece {
        char* vec;  // first vector of the row
        int o;      // this thread's first vector
        uint32_t byte[kMaskUnroll];
    };
    auto fetch = [&](const PieceWalk& at) {
        Piece p;
        char* rowp = reinterpret_cast<char*>(logits) + at.row * row_stride * ES;
        const uint8_t* bits = reinterpret_cast<const uint8_t*>(vocab_mask) + at.row * vm_stride * 4;
        const int head = row_head<DT>(rowp, V), n_vec = (V - head) >> 3;
        p.vec = rowp + head * ES;
        p.o = at.ch * kMaskChunk + tid;
#pragma unroll
        for (int u = 0; u < kMaskUnroll; ++u) {
            const int o = p.o + u * 256;
            p.byte[u] = 0xFFu;
            if (o < n_vec) {
                p.byte[u] = ld_after_wait(bits + o);
                if (head) p.byte[u] = ((p.byte[u] | (ld_after_wait(bits + o + 1) << 8)) >> head) & 0xFFu;
            }
        }
        if (at.ch == 0 && tid < 16) {  // the ends of the row
            const int t = tid < 8 ? tid : head + 8 * n_vec + tid - 8;
            if ((tid < 8 ? t < head : t < V) && !((ld_after_wait(bits + (t >> 3)) >> (t & 7)) & 1u)) store_neg_inf<DT>(rowp, t);
        }
        return p;
    };
    PieceWalk at(blockIdx.x, chunks, row_step, ch_step);
    if (at.row >= B) return;
    Piece p = fetch(at);
    for (;;) {
        Octet<DT> oc[kMaskUnroll];
#pragma unroll
        for (int u = 0; u < kMaskUnroll; ++u)
            if (p.byte[u] != 0xFFu && p.byte[u] != 0u) oc[u].load(p.vec, p.o + u * 256);
        const Piece now = p;
        at.next();
        const bool more = at.row < B;
        if (more) p = fetch(at);
#pragma unroll
        for (int u = 0; u < kMaskUnroll; ++u) {
            if (now.byte[u] == 0xFFu) continue;
            float f[8];
            if (now.byte[u] == 0u) oc[u].fill_neg_inf(); else oc[u].mask(now.byte[u], f);
            oc[u].store(now.vec, now.o + u * 256, true);  // (f32 vectors sit on 32-byte boundaries)
        }
        if (!more) return;
    }
}

// Measurement aid: the cheapest in-place read-modify-write over a logits matrix (every whole 16-byte vector of
// every row is read, the sign bits of its elements are flipped, and it is written back). It moves the bytes a
// step must at least move and does nothing else, so its time under the same launch protocol is what the
// step's time is compared with.
template <int DT>
__global__ void __launch_bounds__(256) k_rmw_floor(void* logits, int64_t row_stride, int B, int V) {
    pdl_prologue();
    constexpr int ES = DT == kBF16 ? 2 : 4;
    constexpr int U = 4;
    constexpr uint32_t kSign = DT == kBF16 ? 0x80008000u : 0x80000000u;
    const int nvec = int((int64_t(V) * ES) >> 4);
    const int chunks = (nvec + 256 * U - 1) / (256 * U);
    const int64_t total = int64_t(B) * chunks;
    for (int64_t item = blockIdx.x; item < total; item += gridDim.x) {
        const int row = int(item / chunks), ch = int(item - int64_t(row) * chunks);
        char* rowp = reinterpret_cast<char*>(logits) + int64_t(row) * row_stride * ES;
        uint4 v[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int i = ch * 256 * U + u * 256 + threadIdx.x;
            if (i < nvec) v[u] = ld_stream16(rowp + size_t(i) * 16);
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int i = ch * 256 * U + u * 256 + threadIdx.x;
            if (i < nvec) {
                v[u].x ^= kSign; v[u].y ^= kSign; v[u].z ^= kSign; v[u].w ^= kSign;
                st_stream16(rowp + size_t(i) * 16, v[u]);
            }
        }
    }
}

// logp_full[b, i] = z'[b, i] - lse[b] from the masked logits (fp32 out, row stride V). Bound: HBM. QUADS: rows of both sides
// allow four tokens at a time (16-byte stores, 16- or 8-byte loads); otherwise a token per thread. Four loads per thread
// are in flight either way (one at a time, token by token, took 42 us for 128 rows of 151936 f32 logits; now 20).
template <int DT, bool QUADS>
__global__ void __launch_bounds__(256) k_logp_full(const void* logits, int64_t row_stride, int B, int V, const float* lse,
                                                   float* out) {
    pdl_prologue();
    constexpr int kPer = QUADS ? 4 : 1, kInFlight = 4;
    const int units = V / kPer, tid = threadIdx.x;  // (V is a multiple of 4 with QUADS)
    auto value = [](float z, float l) { return (l == -INFINITY || z == -INFINITY) ? -INFINITY : z - l; };
    // grid: x strides over the pieces of a row, y over the rows
    for (int row = blockIdx.y; row < B; row += gridDim.y) {
        const float l = ld_after_wait(lse + row);
        const char* zrow = reinterpret_cast<const char*>(logits) + int64_t(row) * row_stride * (DT == kBF16 ? 2 : 4);
        float* orow = out + int64_t(row) * V;
        for (int u0 = blockIdx.x * 256 * kInFlight + tid; u0 < units; u0 += gridDim.x * 256 * kInFlight) {
            if (QUADS) {
                uint4 v[kInFlight];
#pragma unroll
                for (int k = 0; k < kInFlight; ++k) {
                    const int u = u0 + k * 256;
                    if (u >= units) break;
                    if (DT == kF32) {
                        v[k] = __ldcs(reinterpret_cast<const uint4*>(zrow) + u);
                    } else {
                        const uint2 h = __ldcs(reinterpret_cast<const uint2*>(zrow) + u);
                        v[k] = make_uint4(h.x << 16, h.x & 0xFFFF0000u, h.y << 16, h.y & 0xFFFF0000u);
                    }
                }
#pragma unroll
                for (int k = 0; k < kInFlight; ++k) {
                    const int u = u0 + k * 256;
                    if (u >= units) break;
                    __stcs(reinterpret_cast<float4*>(orow) + u,
                           make_float4(value(__uint_as_float(v[k].x), l), value(__uint_as_float(v[k].y), l),
                                       value(__uint_as_float(v[k].z), l), value(__uint_as_float(v[k].w), l)));
                }
            } else {
                float z[kInFlight];
#pragma unroll
                for (int k = 0; k < kInFlight; ++k)
                    if (u0 + k * 256 < units) z[k] = load_elem<DT>(zrow, u0 + k * 256);
#pragma unroll
                for (int k = 0; k < kInFlight; ++k)
                    if (u0 + k * 256 < units) orow[u0 + k * 256] = value(z[k], l);
            }
        }
    }
}

// reps[b] = r[c[tokens[b]]]
// one: the partition of all rows, as an argument (a look less in the chain: token, representative); else parts[row_part[b]].
__global__ void __launch_bounds__(256) k_map_tokens(const PartDev* parts, int n_parts, const __grid_constant__ PartDev one,
                                                    const int32_t* row_part, const int32_t* tokens, int32_t* reps, int B,
                                                    int V_expected, int32_t* status) {
    pdl_prologue();
    const int b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b >= B) return;
    const int32_t* trep = one.trep;
    const int t = tokens[b];
    if (row_part) {
        const int p = row_part[b];
        if (p < 0 || p >= n_parts || !parts[p].live || parts[p].V != V_expected) {
            atomicAdd(status + 2, 1);
            return;
        }
        trep = parts[p].trep;
    }
    int rv = -1;
    if (t >= 0 && t < V_expected) rv = trep[t];
    else atomicAdd(status + 1, 1);
    reps[b] = rv;
}

}  // namespace cfgzip
