// The whole step of a short batch in one launch: a thread-block cluster holds a row, or a few, in its shared memory.
#pragma once

#include "cfgzip_kernels.cuh"

namespace cfgzip {

// ---------------------------------------------------------------------------------------
// One launch per step. R consecutive rows belong to one cluster; its blocks take consecutive pieces of the vocabulary and their
// warps consecutive runs of octets, all of which is asked for at once (bulk copies, one barrier per 32 octets) and stays in shared
// memory. Allow bits come from a table with one byte per class (bit 7 - r: row r of the cluster allows it). A warp masks its run, writes
// it back and folds it into a state per row; the block folds its warps' states, finds the winning token in shared memory and asks
// for its representative; and the blocks send what they have to the first one, or to all of them where every block needs the row's
// total: in a sampling step the block that holds the crossing draws the token from its shared memory, and full log-probabilities
// are written from there as well. Nothing is read twice and nothing goes through global scratch.
// Against the streaming kernel and a second launch (us, greedy, bf16): one row of 32000 f32 5.7 -> 3.3 on the GPU and 6.6 -> 3.8 as a
// program calls it, 8 rows of 128256 6.7 -> 4.7, 32 rows 8.5 -> 7.6, 48 rows of 100003 off the vector grid 12.8 -> 10.6; 32 rows of
// four partitions, which need no row plan here, 23.3 -> 8.6; 32 rows with full log-probabilities 13.0 -> 10.6; sampling 10.6 -> 8.4.
// Bound: some 2.8 us are launch, class masks, the way of the first bytes and the exchange between the blocks; after that instruction
// issue, 0.34 us per row and chunk of a block's 16 warps and 0.19 for the lookups that the rows of a chunk share (least squares over
// rows x blocks of 4 to 80 rows), which is why rows share a cluster as soon as there are more than a few.
// ---------------------------------------------------------------------------------------
constexpr int kClusterThreads = 512, kClusterWarps = kClusterThreads / 32;
constexpr int kClusterRows = 4;    // rows of a cluster
constexpr int kClusterMost = 16;   // blocks of a cluster
constexpr int kClusterChunks = 8;  // chunks of a warp's run
constexpr int kClusterSlots = kClusterWarps + 2;  // states of a block: tokens in front of the first vector, the warps, tokens past the last one
constexpr size_t kClusterStatic = 5 * 1024;       // most shared memory the kernel has beside the dynamic one

struct ClusterGeom {
    int rows;       // of a cluster
    int blocks;     // of a cluster
    int per_block;  // octets of a block
    int run;        // octets of a warp
    float* full;    // greedy step: full log-probabilities, or null
    int quads;      // ... whose rows take 16-byte stores
};

// Where things lie in dynamic shared memory: the class table, then for every warp its rows' runs and the run's class ids.
__host__ __device__ inline int cluster_table_bytes(int KW) { return ((KW + 1) * 32 + 127) & ~127; }
__host__ __device__ inline int cluster_warp_bytes(int run, int rows, int octet_bytes) { return run * rows * octet_bytes + (run + 1) * 16; }

// Where the draw of a row goes on inside a block.
struct ClusterDraw {
    int warp;     // whose run holds the crossing; -1: another block's, or done
    float M;      // the row's largest logit
    float total;  // and weight
    float tau;    // the weight the drawn token's prefix passes first
    float front;  // in front of the run
};

template <int R>
struct ClusterShared {
    uint64_t bar[kClusterWarps][kClusterChunks];  // a chunk's logits
    uint64_t ids_bar[kClusterWarps];
    uint64_t peer_bar;
    Partial state[R][kClusterSlots];
    uint4 peer[R][kClusterMost];  // largest logit, sum, token, representative (or state of the block)
    float edge[R][32];            // masked logits of the tokens in front of the first vector (0..7) and past the last one (8..23)
    float lse[R];
    ClusterDraw draw[R];          // sampling step
    float scan[R][kClusterWarps];
};

// The top bits of the bytes of two words as the bits of a byte. ALONE: the other bits are zero.
template <bool ALONE>
__device__ __forceinline__ uint32_t gather_msbs(uint32_t lo, uint32_t hi) {
    const uint32_t l = (ALONE ? lo : lo & 0x80808080u) * 0x00204081u, h = (ALONE ? hi : hi & 0x80808080u) * 0x00204081u;
    return (l >> 28) | ((h >> 24) & 0xF0u);
}
// Inclusive prefix sums over the lanes of a warp.
__device__ __forceinline__ float warp_inclusive_scan(float v, int lane) {
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const float up = __shfl_up_sync(0xFFFFFFFFu, v, d);
        if (lane >= d) v += up;
    }
    return v;
}
// The first lane with weight whose inclusive prefix passes tau; where rounding leaves tau at the very end the last one with weight,
// -1 where none has any.
__device__ __forceinline__ int crossing_lane(float weight, float inclusive, float tau) {
    const uint32_t some = __ballot_sync(0xFFFFFFFFu, weight > 0.f), past = __ballot_sync(0xFFFFFFFFu, weight > 0.f && inclusive > tau);
    return past ? __ffs(int(past)) - 1 : 31 - __clz(int(some));
}

__device__ __forceinline__ unsigned long long first_allowed_warp(const StepArgs& a, const PartDev& P, int row, int lane) {
    unsigned long long pick = first_allowed_share(a, P, row, lane, 32);
#pragma unroll
    for (int d = 16; d >= 1; d >>= 1) {
        const unsigned long long other = __shfl_xor_sync(0xFFFFFFFFu, pick, d);
        pick = other < pick ? other : pick;
    }
    return pick;
}

__device__ __forceinline__ float front_of(float inclusive, int l) {  // what lies in front of lane l
    const float f = __shfl_sync(0xFFFFFFFFu, inclusive, max(l - 1, 0));
    return l > 0 ? f : 0.f;
}
__device__ __forceinline__ void write_draw(const StepArgs& a, const PartDev& P, int row, float M, float total, int token, float z) {
    const float l = logf(total);
    a.argmax[row] = token;
    if (a.rep) a.rep[row] = __ldg(P.trep + token);
    if (a.lse) a.lse[row] = fmaf(M, a.inv_t, l);
    if (a.logp_argmax) a.logp_argmax[row] = (z - M) * a.inv_t - l;
}
__device__ __forceinline__ void write_no_draw(const StepArgs& a, int row) {  // no token carries weight: the row counts as empty
    a.argmax[row] = -1;
    if (a.rep) a.rep[row] = -1;
    if (a.lse) a.lse[row] = -INFINITY;
    if (a.logp_argmax) a.logp_argmax[row] = -INFINITY;
}

// The draw of a sampling step, first half: a warp of every block of the row's cluster. M: the row's largest logit; weight (lane b):
// what block b weighs. All blocks come to the same block, and that one to the run that holds the crossing; the few tokens outside the
// vectors are done with here. All sums of a draw are taken in a fixed order.
template <int R>
__device__ __forceinline__ void cluster_draw(const StepArgs& a, const PartDev& P, ClusterShared<R>& sh, int row, int r, int lane, int rank,
                                             float M, float weight) {
    if (lane == 0) sh.draw[r].warp = -1;
    if (!(M * a.scale > kRefLow)) {  // nothing allowed, or nothing that weighs anything: the lowest allowed token (if any) and -inf logs
        if (rank == 0) {
            const unsigned long long pick = first_allowed_warp(a, P, row, lane);
            if (lane == 0) write_row_outputs(a, row, -INFINITY, 0.f, pick);
        }
        return;
    }
    float inc = warp_inclusive_scan(weight, lane);
    const float total = __shfl_sync(0xFFFFFFFFu, inc, 31), tau = ld_after_wait(a.u + row) * total;
    const int block = crossing_lane(weight, inc, tau);
    if (block < 0 && rank == 0 && lane == 0) write_no_draw(a, row);  // (an allowed +inf makes every weight NaN or zero)
    if (block != rank) return;
    float base = front_of(inc, block);
    const Partial p = lane < kClusterSlots ? sh.state[r][lane] : partial_empty();
    float w = p.m > kRefFloor ? p.s * ex2f((p.m - M) * a.scale) : 0.f;
    inc = warp_inclusive_scan(w, lane);
    const int slot = crossing_lane(w, base + inc, tau);
    if (slot < 0) {
        if (lane == 0) write_no_draw(a, row);
        return;
    }
    base += front_of(inc, slot);
    if (slot > 0 && slot < kClusterSlots - 1) {
        if (lane == 0) sh.draw[r] = ClusterDraw{slot - 1, M, total, tau, base};
        return;
    }
    const int token = slot == 0 ? lane : 8 * ((a.V >> 3) - 1) + lane - 8;
    const float z = (slot == 0) == (lane < 8) ? sh.edge[r][lane] : -INFINITY;
    w = ex2f((z - M) * a.scale);
    inc = warp_inclusive_scan(w, lane);
    const int winner = crossing_lane(w, base + inc, tau);
    if (winner >= 0 ? lane == winner : lane == 0) {
        if (winner >= 0) write_draw(a, P, row, M, total, token, z); else write_no_draw(a, row);
    }
}

template <int DT, int R, bool SHIFT, bool TEMPERED>
__global__ void __launch_bounds__(kClusterThreads, 1) k_step_cluster(const __grid_constant__ StepArgs a, const __grid_constant__ ClusterGeom g) {
    constexpr int ES = DT == kBF16 ? 2 : 4, OB = 8 * ES;
    constexpr int U = SHIFT ? 31 : 32;  // vectors of a chunk: a shifted vector's bits come from two octets, the last lane's serve its neighbour
    __shared__ ClusterShared<R> sh;
    extern __shared__ __align__(128) uint32_t smem[];
    uint8_t* const T = reinterpret_cast<uint8_t*>(smem);

    pdl_launch_dependents();
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int rank = int(cluster_rank()), cid = blockIdx.x / g.blocks;
    const int row0 = cid * g.rows, live = min(g.rows, a.B - row0);
    const bool to_all = TEMPERED || g.full != nullptr;  // every block needs the totals of the rows
    const float scale = TEMPERED ? a.scale : kLog2e;
    const int n_octets = 4 * a.VW, n_full = a.V >> 3;
    const int b_begin = min(rank * g.per_block, n_full), b_end = min(b_begin + g.per_block, n_full);
    const int o_begin = min(b_begin + warp * g.run, b_end), n_run = min(g.run, b_end - o_begin);
    const int n_chunks = (n_run + U - 1) / U;
    const int warp_bytes = cluster_warp_bytes(g.run, g.rows, OB);
    auto row_addr = [&](int r) { return reinterpret_cast<char*>(a.logits) + int64_t(row0 + r) * a.row_stride * ES; };
    auto head_of = [&](int r) { return SHIFT ? row_head<DT>(row_addr(r), a.V) : 0; };

    // Set-up: nothing of it reads what the kernel in front writes.
    if (tid == 0) {
        mbar_init(&sh.peer_bar, 1);
        mbar_init_fence();
        if (to_all || rank == 0) mbar_expect_tx(&sh.peer_bar, uint32_t(g.blocks * live) * 16u);
    }
    if (lane == 0) {
        for (int c = 0; c < n_chunks; ++c) mbar_init(&sh.bar[warp][c], 1);
        mbar_init(&sh.ids_bar[warp], 1);
        mbar_init_fence();
    }
    __syncwarp();
    cluster_arrive();  // (every thread waits for its peers before the first of them is written to)
    PartDev P = a.p0;
    const bool mixed = R == 1 && a.row_part != nullptr;
    if (mixed) {
        pdl_wait();
        const int part = a.row_part[row0];
        if (part < 0 || part >= a.n_parts || !a.parts[part].live || a.parts[part].V != a.V) {
            if (rank == 0 && tid == 0) atomicAdd(a.status + 2, 1);
            return;  // (all blocks of the cluster)
        }
        P = a.parts[part];
    }
    const int table_bytes = cluster_table_bytes(P.KW);
    char* const ring = reinterpret_cast<char*>(smem) + table_bytes + size_t(warp) * warp_bytes;
    char* const ids = ring + g.run * g.rows * OB;
    if (lane == 0 && n_run > 0) {
        const uint32_t bytes = uint32_t(min(n_run + (SHIFT ? 1 : 0), n_octets - o_begin)) * 16u;
        mbar_expect_tx(&sh.ids_bar[warp], bytes);
        bulk_g2s(ids, reinterpret_cast<const char*>(P.c16) + size_t(o_begin) * 16, bytes, &sh.ids_bar[warp]);
    }
    if (!mixed) pdl_wait();

    // The class masks first (everything waits for them), then all logits.
    uint32_t w[R];
#pragma unroll
    for (int r = 0; r < R; ++r) w[r] = r < live && tid < P.KW ? ld_after_wait(a.class_mask + int64_t(row0 + r) * a.cm_stride + tid) : 0u;
    {
        auto vectors = [&](int r, int c) {  // of row r in chunk c
            const int nvec = (a.V - head_of(r)) >> 3;
            return max(0, min(min(U, n_run - c * U), nvec - (o_begin + c * U)));
        };
        if (lane < n_chunks) {
            uint32_t bytes = 0u;
            for (int r = 0; r < live; ++r) bytes += uint32_t(vectors(r, lane)) * OB;
            mbar_expect_tx(&sh.bar[warp][lane], bytes);
        }
        __syncwarp();
        static_assert(R * kClusterChunks <= 32 && sizeof(sh) <= kClusterStatic, "a lane per copy; the launch leaves room for sh");
        const int r = lane % R, c = lane / R;
        if (c < n_chunks && r < live) {
            const int n = vectors(r, c);
            if (n > 0)
                bulk_g2s(ring + (r * g.run + c * U) * OB, row_addr(r) + head_of(r) * ES + size_t(o_begin + c * U) * OB, uint32_t(n) * OB,
                         &sh.bar[warp][c]);
        }
    }
    // The tokens that the vectors leave over: lanes 0..7 of one warp of the first block those in front, lanes 8..23 of the last
    // block's those from the last whole octet on.
    const bool first = SHIFT && rank == 0, last = rank == g.blocks - 1, in_head = lane < 8;
    const int et = in_head ? lane : 8 * (n_full - 1) + lane - 8;
    const bool edges = warp == kClusterWarps - 1 && (first || last) && (SHIFT || n_full != n_octets);
    const bool have_edge = edges && lane < 24 && (in_head ? first : last) && et >= 0 && et < a.V;
    uint32_t edge_id = 0u;
    float edge_z[R];
    auto edge_mine = [&](int r) {
        const int head = head_of(r), tail = head + ((a.V - head) & ~7);
        return have_edge && r < live && (in_head ? et < head : et >= tail);
    };
    if (edges) {
        if (have_edge) edge_id = P.c16[et];
#pragma unroll
        for (int r = 0; r < R; ++r) edge_z[r] = edge_mine(r) ? load_elem<DT>(row_addr(r), et) : -INFINITY;
    }
    // Class table: byte k, bit 7 - r. Entries from K on are zero, so that the padding class K looks up "nobody".
    for (int kw = tid; kw <= P.KW; kw += kClusterThreads) {
        const uint32_t keep = kw == P.KW ? 0u : (kw == P.KW - 1 && (P.K & 31)) ? (1u << (P.K & 31)) - 1u : 0xFFFFFFFFu;
        if (kw != tid) {
#pragma unroll
            for (int r = 0; r < R; ++r) w[r] = r < live && kw < P.KW ? ld_after_wait(a.class_mask + int64_t(row0 + r) * a.cm_stride + kw) : 0u;
        }
        uint32_t x[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            x[j] = 0u;
#pragma unroll
            for (int r = 0; r < R; ++r) x[j] |= (nibble_to_byte_msbs(((w[r] & keep) >> (4 * j)) & 0xFu) & 0x80808080u) >> r;
        }
        uint4* const dst = reinterpret_cast<uint4*>(T + kw * 32);
        dst[0] = make_uint4(x[0], x[1], x[2], x[3]);
        dst[1] = make_uint4(x[4], x[5], x[6], x[7]);
    }
    __syncthreads();

    if (warp == kClusterWarps - 1) {
        if (edges) {
            const uint32_t allow8 = have_edge ? T[edge_id] : 0u;
#pragma unroll
            for (int r = 0; r < R; ++r) {
                if (r >= live) break;
                const bool allowed = (allow8 << r) & 0x80u, mine = edge_mine(r);
                const uint32_t allow = __ballot_sync(0xFFFFFFFFu, allowed && !in_head);
                if (last && a.vocab_mask && lane < n_octets - n_full)
                    reinterpret_cast<uint8_t*>(a.vocab_mask + int64_t(row0 + r) * a.vm_stride)[n_full + lane] =
                        lane == 0 ? uint8_t(allow >> 16) : uint8_t(0);
                if (mine && !allowed) store_neg_inf<DT>(row_addr(r), et);
                const float z = mine && allowed ? edge_z[r] : -INFINITY;
                sh.edge[r][lane] = z;
#pragma unroll
                for (int side = 0; side < 2; ++side) {
                    const float zs = in_head == (side == 0) ? z : -INFINITY;
                    const float m = float_from_order_key(__reduce_max_sync(0xFFFFFFFFu, float_order_key(zs)));
                    float e = m > kRefFloor ? ex2f((zs - m) * scale) : 0.f;
#pragma unroll
                    for (int d = 16; d >= 1; d >>= 1) e += __shfl_xor_sync(0xFFFFFFFFu, e, d);
                    const int pos = __reduce_min_sync(0xFFFFFFFFu, m > -INFINITY && zs == m ? et : kNoPos);
                    if (lane == 0) sh.state[r][side ? kClusterSlots - 1 : 0] = Partial{m, e, pos, 0};
                }
            }
        } else if (lane < 2 * R) {  // (the draw never looks at the tokens of an empty state)
            sh.state[lane >> 1][lane & 1 ? kClusterSlots - 1 : 0] = partial_empty();
        }
    }

    // The run: mask, write back, fold.
    RowAcc acc[R];
#pragma unroll
    for (int r = 0; r < R; ++r) acc[r].init();
    bool failed = false;
    if (n_run > 0) failed = !mbar_wait(&sh.ids_bar[warp], 0);
    uint8_t* const vm8 = reinterpret_cast<uint8_t*>(a.vocab_mask);
    const bool wide = SHIFT || a.wide != 0;  // (f32 vectors of rows that start anywhere sit on 32-byte boundaries)
#pragma unroll 1
    for (int c = 0; c < n_chunks; ++c) {
        const bool arrived = mbar_wait(&sh.bar[warp][c], 0) && !a.expire_test;
        if (!__all_sync(0xFFFFFFFFu, arrived)) {
            failed = true;
            continue;  // (the copies of the other chunks are waited for all the same)
        }
        const int i = c * U + lane, o = o_begin + i;  // octet of the run, of the vocabulary
        uint32_t lo = 0u, hi = 0u;
        if (SHIFT ? i <= n_run && o < n_octets : i < n_run) {
            const uint4 cv = *reinterpret_cast<const uint4*>(ids + i * 16);
            lo = __byte_perm(__byte_perm(T[cv.x & 0xFFFFu], T[cv.x >> 16], 0x0040), __byte_perm(T[cv.y & 0xFFFFu], T[cv.y >> 16], 0x0040), 0x5410);
            hi = __byte_perm(__byte_perm(T[cv.z & 0xFFFFu], T[cv.z >> 16], 0x0040), __byte_perm(T[cv.w & 0xFFFFu], T[cv.w >> 16], 0x0040), 0x5410);
        }
        uint32_t lo2 = 0u, hi2 = 0u;
        if (SHIFT) {
            lo2 = __shfl_down_sync(0xFFFFFFFFu, lo, 1);
            hi2 = __shfl_down_sync(0xFFFFFFFFu, hi, 1);
        }
        if (lane >= U || i >= n_run) continue;
#pragma unroll
        for (int r = 0; r < R; ++r) {
            if (r >= live) break;
            if (vm8) st_global_u8(vm8 + int64_t(row0 + r) * a.vm_stride * 4 + o, gather_msbs<R == 1>(lo << r, hi << r));
            uint32_t xl = lo, xh = hi;
            int head = 0;
            if (SHIFT) {
                head = head_of(r);
                if (8 * o + head + 8 > a.V) continue;
                const uint32_t sel = 0x3210u + 0x1111u * uint32_t(head & 3);
                const uint32_t w0 = head & 4 ? hi : lo, w1 = head & 4 ? lo2 : hi, w2 = head & 4 ? hi2 : lo2;
                xl = __byte_perm(w0, w1, sel);
                xh = __byte_perm(w1, w2, sel);
            }
            char* const src = ring + (r * g.run + i) * OB;
            Octet<DT> oc;
            float f[8];
            oc.load_shared_at(src);
            oc.mask_tokens(xl << r, xh << r, f);
            oc.store_at(row_addr(r) + (8 * size_t(o) + head) * ES, wide);
            if (to_all) oc.store_shared_at(src);
            acc[r].add_octet(f, 8 * o + head, scale);
        }
    }
    if (__any_sync(0xFFFFFFFFu, failed) && lane == 0) atomicAdd(a.status + 3, 1);
#pragma unroll
    for (int r = 0; r < R; ++r) {
        if (r >= live) break;
        const float M = float_from_order_key(__reduce_max_sync(0xFFFFFFFFu, float_order_key(acc[r].m)));
        float s = acc[r].sum_below(M, scale);
#pragma unroll
        for (int d = 16; d >= 1; d >>= 1) s += __shfl_xor_sync(0xFFFFFFFFu, s, d);
        const int pos = __reduce_min_sync(0xFFFFFFFFu, acc[r].m == M ? acc[r].pos : kNoPos);
        if (lane == 0) sh.state[r][1 + warp] = Partial{M, s, pos, 0};
    }
    cluster_wait();
    __syncthreads();

    // A warp per row: the block's state goes to the first block of the cluster, or to all of them.
    if (warp < live) {
        const int r = warp, head = head_of(r);
        const Partial p = lane < kClusterSlots ? sh.state[r][lane] : partial_empty();
        const float M = float_from_order_key(__reduce_max_sync(0xFFFFFFFFu, float_order_key(p.m)));
        float s = p.m > kRefFloor ? p.s * ex2f((p.m - M) * scale) : 0.f;
#pragma unroll
        for (int d = 16; d >= 1; d >>= 1) s += __shfl_xor_sync(0xFFFFFFFFu, s, d);
        int token = kNoPos, repv = -1;
        if (!TEMPERED) {
            token = __reduce_min_sync(0xFFFFFFFFu, p.m == M ? p.pos : kNoPos);
            if (token != kNoPos) {
                const int slot = __ffs(int(__ballot_sync(0xFFFFFFFFu, p.m == M && p.pos == token))) - 1;
                if (slot > 0 && slot < kClusterSlots - 1) {  // the first token of a vector of warp slot - 1: which of the eight is it?
                    const char* const wring = reinterpret_cast<const char*>(smem) + table_bytes + size_t(slot - 1) * warp_bytes;
                    const int i = ((token - head) >> 3) - (b_begin + (slot - 1) * g.run);
                    bool ok = false;
                    if (lane < 8) {
                        const uint32_t k = reinterpret_cast<const uint16_t*>(wring + g.run * g.rows * OB)[i * 8 + head + lane];
                        ok = ((T[k] << r) & 0x80u) && load_elem<DT>(wring + (r * g.run + i) * OB, lane) == M;
                    }
                    token += __ffs(int(__ballot_sync(0xFFFFFFFFu, ok))) - 1;
                }
                repv = __ldg(P.trep + token);
            }
        }
        if (lane < (to_all ? g.blocks : 1))
            st_async_peer_v4(peer_shared(&sh.peer[r][rank], uint32_t(lane)),
                             make_uint4(__float_as_uint(M), __float_as_uint(s), uint32_t(token), uint32_t(repv)),
                             peer_shared(&sh.peer_bar, uint32_t(lane)));
        if (to_all || rank == 0) {
            if (!mbar_wait_cluster(&sh.peer_bar, 0) && lane == 0) atomicAdd(a.status + 3, 1);
            uint4 q = make_uint4(__float_as_uint(-INFINITY), 0u, uint32_t(kNoPos), 0u);
            if (lane < g.blocks) q = sh.peer[r][lane];
            const float qm = __uint_as_float(q.x);
            const float MM = float_from_order_key(__reduce_max_sync(0xFFFFFFFFu, float_order_key(qm)));
            const float weight = qm > kRefFloor ? __uint_as_float(q.y) * ex2f((qm - MM) * scale) : 0.f;
            if (TEMPERED) {
                cluster_draw<R>(a, P, sh, row0 + r, r, lane, rank, MM, weight);
            } else {
                float total = weight;
#pragma unroll
                for (int d = 16; d >= 1; d >>= 1) total += __shfl_xor_sync(0xFFFFFFFFu, total, d);
                if (rank == 0) {
                    const int best = __reduce_min_sync(0xFFFFFFFFu, qm == MM ? int(q.z) : kNoPos);
                    unsigned long long pick = ~0ull;
                    if (best != kNoPos) {
                        const int from = __ffs(int(__ballot_sync(0xFFFFFFFFu, qm == MM && int(q.z) == best))) - 1;
                        const uint32_t best_rep = __shfl_sync(0xFFFFFFFFu, q.w, from);
                        pick = (static_cast<unsigned long long>(best) << 32) | best_rep;
                    } else {
                        pick = first_allowed_warp(a, P, row0 + r, lane);
                    }
                    if (lane == 0) write_row_outputs(a, row0 + r, MM, total, pick);
                }
                if (lane == 0) sh.lse[r] = MM > kRefFloor && total > 0.f ? MM + logf(total) : -INFINITY;
            }
        }
    }
    if constexpr (TEMPERED) {
        // The draw's second half: all threads of a block that holds a row's crossing, four tokens of the run each; then the warp
        // that holds the crossing, and its lane.
        __syncthreads();
        for (int r = 0; r < live; ++r) {
            const ClusterDraw d = sh.draw[r];
            if (d.warp < 0) continue;
            const int head = head_of(r), first_octet = min(b_begin + d.warp * g.run, b_end);
            const int n_tok = 8 * max(0, min(min(g.run, b_end - first_octet), ((a.V - head) >> 3) - first_octet));
            const char* const run = reinterpret_cast<const char*>(smem) + table_bytes + size_t(d.warp) * warp_bytes + r * g.run * OB;
            float z[4], w[4], mine = 0.f;
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                z[q] = 4 * tid < n_tok ? load_elem<DT>(run, 4 * tid + q) : -INFINITY;
                w[q] = ex2f((z[q] - d.M) * scale);
                mine += w[q];
            }
            const float inc = warp_inclusive_scan(mine, lane);
            if (lane == 31) sh.scan[r][warp] = inc;
            __syncthreads();
            const float per_warp = lane < kClusterWarps ? sh.scan[r][lane] : 0.f, inc_warps = warp_inclusive_scan(per_warp, lane);
            const int owner = crossing_lane(per_warp, d.front + inc_warps, d.tau);
            if (warp != max(owner, 0)) continue;
            float base = d.front + front_of(inc_warps, warp);
            const int l = crossing_lane(mine, base + inc, d.tau);
            base += front_of(inc, max(l, 0));
            if (l >= 0 ? lane != l : lane != 0) continue;
            int at = -1;
            float zt = 0.f;
            bool past = false;
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                base += w[q];
                if (w[q] > 0.f && !past) {  // (where rounding leaves tau at the very end: the last token with weight)
                    at = q;
                    zt = z[q];
                    past = base > d.tau;
                }
            }
            if (at >= 0) write_draw(a, P, row0 + r, d.M, d.total, 8 * first_octet + head + 4 * tid + at, zt); else write_no_draw(a, row0 + r);
        }
        return;
    }
    if (!g.full) return;

    // Full log-probabilities from the masked logits in shared memory, every warp its own run.
    __syncthreads();
    auto logp = [](float z, float l) { return l == -INFINITY || z == -INFINITY ? -INFINITY : z - l; };
    for (int r = 0; r < live; ++r) {
        const int head = head_of(r), nvec = max(0, min(n_run, ((a.V - head) >> 3) - o_begin));
        const float l = sh.lse[r];
        float* const orow = g.full + int64_t(row0 + r) * a.V;
        float* const out = orow + 8 * o_begin + head;
        const char* const src = ring + r * g.run * OB;
        if (!SHIFT && g.quads) {
#pragma unroll 4
            for (int q = lane; q < 2 * nvec; q += 32) {
                uint4 v;
                if (DT == kF32) {
                    v = reinterpret_cast<const uint4*>(src)[q];
                } else {
                    const uint2 h = reinterpret_cast<const uint2*>(src)[q];
                    v = make_uint4(h.x << 16, h.x & 0xFFFF0000u, h.y << 16, h.y & 0xFFFF0000u);
                }
                __stcs(reinterpret_cast<float4*>(out) + q, make_float4(logp(__uint_as_float(v.x), l), logp(__uint_as_float(v.y), l),
                                                                       logp(__uint_as_float(v.z), l), logp(__uint_as_float(v.w), l)));
            }
        } else {
#pragma unroll 4
            for (int t = lane; t < 8 * nvec; t += 32) __stcs(out + t, logp(load_elem<DT>(src, t), l));
        }
        if (edges && edge_mine(r)) orow[et] = logp(sh.edge[r][lane], l);
    }
}

}  // namespace cfgzip
