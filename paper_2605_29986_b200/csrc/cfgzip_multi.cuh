// Several class masks per logits row: the streaming half of the call (k_finalize_rows is the other).
#pragma once

#include "cfgzip_kernels.cuh"

namespace cfgzip {

// ---------------------------------------------------------------------------------------
// Row groups and class table as in the gather kernels, over "virtual rows" (logits row, mask): virtual row r belongs to logits
// row r / masks_per_row. A warp takes 32 octets of 8 virtual rows at a time. What depends on the logits alone is done once per
// logits row: the octet is loaded and its eight exponentials are taken, and the lane writes down (largest logit, sum of
// exponentials) of all 16 subsets of either half of the octet. A mask then costs two lookups with the two halves of its byte.
// Bound: instruction latency and issue (the schedulers issue in 56 % of the cycles with some four warps each, the shared-memory
// pipe is busy for 42 %, DRAM for 2; a warp waits mostly for its own last instruction and for shared memory): some 20 instructions
// per octet and mask, 8 KB of subsets written per octet and warp, 0.5 KB read per mask. (Masking and exponentials anew for every mask, a class table per short block:
// 8 rows x 16 masks of 128256 bf16 logits 24.3 us, now 14.5; 32 x 32 masks of 151936 f32 logits 134 us, now 65.)
//
// The exponentials of a lane share one reference per logits row, whatever a mask allows. It is set 64 powers of two below the
// largest logit seen and moves when one overtakes it by more than 84, so that sums stay below 2^102 and a mask whose largest
// logit lies up to 164 powers of two (113 nats) below the row's loses nothing. Beyond that the state's sum is marked (NaN)
// and the second kernel sums the row anew for that mask.
// ---------------------------------------------------------------------------------------
constexpr int kMultiWarps = 8;
constexpr float kMultiLift = 64.f, kMultiMove = 84.f, kMultiFloor = -100.f;  // powers of two
constexpr size_t kMultiTable = 32 * 32 * sizeof(float2);                     // per warp: 2 x 16 subsets, a column per lane

template <int DT>
__device__ __forceinline__ void octet_floats(const Octet<DT>& o, float (&f)[8]) {
    if constexpr (DT == kBF16) {
        const uint32_t r[4] = {o.v.x, o.v.y, o.v.z, o.v.w};
#pragma unroll
        for (int q = 0; q < 8; ++q) f[q] = __uint_as_float((q & 1) ? r[q / 2] & 0xFFFF0000u : r[q / 2] << 16);
    } else {
        const uint32_t r[8] = {o.a.x, o.a.y, o.a.z, o.a.w, o.b.x, o.b.y, o.b.z, o.b.w};
#pragma unroll
        for (int q = 0; q < 8; ++q) f[q] = __uint_as_float(r[q]);
    }
}

template <int DT>
__global__ void __launch_bounds__(kMultiWarps * 32, 2) k_step_multi(const __grid_constant__ StepArgs a) {
    extern __shared__ __align__(128) uint32_t smem[];
    uint32_t* T = smem;
    int* s_row = reinterpret_cast<int*>(T + a.table_words);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, n_warps = blockDim.x >> 5;
    float2* const subsets = reinterpret_cast<float2*>(s_row + kGroupRows) + warp * (kMultiTable / sizeof(float2)) + lane;
    uint32_t* stage = reinterpret_cast<uint32_t*>(reinterpret_cast<char*>(s_row + kGroupRows) + n_warps * kMultiTable);

    pdl_launch_dependents();
    const int g = blockIdx.x / a.S, split = blockIdx.x - g * a.S;
    group_rows_setup(a, g, s_row, tid);  // (no row plan here: nothing is read)
    const PartDev P = a.p0;
    const int nrow = min(kGroupRows, a.B - g * kGroupRows);
    __syncthreads();

    constexpr int ES = DT == kBF16 ? 2 : 4;
    const int M = a.masks_per_row;
    const int wt = warp % a.WT, wr = warp / a.WT, WR = n_warps / a.WT;
    const int n_full = a.V >> 3, n_chunks = (n_full + 31) >> 5, stride = a.S * a.WT;
    const uint4* const ids = reinterpret_cast<const uint4*>(P.c16);
    const int64_t row_bytes = a.row_stride * ES;
    // the warp's first chunk of a row batch: its logits and class ids are asked for at once (before the class table is built,
    // for the first row batch)
    Octet<DT> next;
    uint4 cv = make_uint4(0, 0, 0, 0);
    int c = 0;
    auto first_row = [&](int rb) {
        return reinterpret_cast<const char*>(a.logits) + ((g * kGroupRows + rb * kBatchRows) / M) * row_bytes;
    };
    auto open = [&](int rb) {
        c = (split * a.WT + wt - rb * a.rot_chunks) % stride;  // the deal starts at another warp for every row batch
        if (c < 0) c += stride;
        next.fill_neg_inf();
        if (c * 32 + lane < n_full) {
            next.load(first_row(rb), c * 32 + lane);
            cv = __ldg(ids + c * 32 + lane);
        }
    };
    pdl_wait();
    if (wr * kBatchRows < nrow) open(wr);
    make_class_table_of_group(a, P, g, s_row, T, stage, warp, lane, n_warps);
    __syncthreads();

    for (int rb = wr; rb * kBatchRows < nrow; rb += WR) {
        const int r0 = g * kGroupRows + rb * kBatchRows, live = min(kBatchRows, nrow - rb * kBatchRows);
        const char* const row0 = first_row(rb);
        uint32_t starts = 1u;  // bit i: virtual row i of the batch is the first of its logits row
#pragma unroll
        for (int i = 1; i < kBatchRows; ++i)
            if (i < live && (r0 + i) % M == 0) starts |= 1u << i;
        uint8_t* vm = a.vocab_mask ? reinterpret_cast<uint8_t*>(a.vocab_mask) + int64_t(r0) * a.vm_stride * 4 : nullptr;
        RowAcc acc[kBatchRows];
#pragma unroll
        for (int i = 0; i < kBatchRows; ++i) acc[i].init();

        if (rb != wr) open(rb);
        for (; c < n_chunks; c += stride) {
            const int o = c * 32 + lane, o_next = o + stride * 32;
            const bool active = o < n_full;
            uint32_t lo, hi;
            octet_allow_bits(cv, T, rb, active, lo, hi);
            if (o_next < n_full) cv = __ldg(ids + o_next);
            const char* row = row0;
            // one logits row of the batch after the other: virtual rows i0 .. i1 - 1 (rolled: the code is long)
#pragma unroll 1
            for (int i0 = 0, i1; i0 < live; i0 = i1) {
                const uint32_t later = starts >> (i0 + 1);
                i1 = later ? i0 + __ffs(int(later)) : live;
                float f[8];
                octet_floats<DT>(next, f);
                // one load ahead: the batch's next logits row, or the first one of the next chunk
                if (i1 < live) {
                    row += row_bytes;
                    if (active) next.load(row, o);
                } else if (o_next < n_full) {
                    next.load(row0, o_next);
                } else {
                    next.fill_neg_inf();
                }
                float nrl = acc[0].nrl;
#pragma unroll
                for (int k = 1; k < kBatchRows; ++k) nrl = i0 == k ? acc[k].nrl : nrl;
                const float top = fmax3(fmax3(f[0], f[1], f[2]), fmax3(f[3], f[4], f[5]), fmaxf(f[6], f[7]));
                if (fmaf(top, kLog2e, nrl) > kMultiMove) {  // rare: the reference moves, for all masks of this row
                    const float n2 = kMultiLift - top * kLog2e, scale = ex2f(n2 - nrl);
#pragma unroll
                    for (int k = 0; k < kBatchRows; ++k)
                        if (k >= i0 && k < i1) {
                            acc[k].s *= scale;
                            acc[k].nrl = n2;
                        }
                    nrl = n2;
                }
                float e[8];
#pragma unroll
                for (int q = 0; q < 8; ++q) e[q] = ex2f(fmaf(f[q], kLog2e, nrl));
#pragma unroll
                for (int half = 0; half < 2; ++half) {
                    float m[16], s[16];
                    m[0] = -INFINITY;
                    s[0] = 0.f;
#pragma unroll
                    for (int k = 1; k < 16; ++k) {
                        const int bit = k & 8 ? 3 : (k & 4 ? 2 : (k & 2 ? 1 : 0)), rest = k ^ (1 << bit);
                        m[k] = rest ? fmaxf(m[rest], f[half * 4 + bit]) : f[half * 4 + bit];
                        s[k] = rest ? s[rest] + e[half * 4 + bit] : e[half * 4 + bit];
                    }
#pragma unroll
                    for (int k = 0; k < 16; ++k) subsets[(half * 16 + k) * 32] = make_float2(m[k], s[k]);
                }
#pragma unroll
                for (int i = 0; i < kBatchRows; ++i) {
                    if (i < i0 || i >= i1) continue;
                    const uint32_t byte = ((i < 4 ? lo : hi) >> (8 * (i & 3))) & 0xFFu;
                    if (vm && active) st_global_u8(vm + int64_t(i) * a.vm_stride * 4 + o, byte);
                    const float2 x = subsets[(byte & 15u) * 32], y = subsets[(16 + (byte >> 4)) * 32];
                    const float best = fmaxf(x.x, y.x);
                    acc[i].pos = best > acc[i].m ? o : acc[i].pos;
                    acc[i].m = fmaxf(acc[i].m, best);
                    acc[i].s += x.y + y.y;
                }
            }
        }
        // sums relative to each mask's own largest logit (in two steps: the way may be longer than a float's exponent)
#pragma unroll
        for (int i = 0; i < kBatchRows; ++i) {
            if (!(acc[i].m > kRefFloor)) continue;
            const float above = fmaf(acc[i].m, kLog2e, acc[i].nrl), half = ex2f(-0.5f * above);
            acc[i].s = above < kMultiFloor ? __int_as_float(0x7FC00000) : acc[i].s * half * half;
            acc[i].nrl = -(acc[i].m * kLog2e);
        }
        warp_rows_publish(a, acc, live, g, split * a.WT + wt, rb, lane);
    }
    if (warp == 0 && split == 0) publish_tail_octets<DT>(a, P, g, s_row, lane, n_full, 4 * a.VW);
}

}  // namespace cfgzip
